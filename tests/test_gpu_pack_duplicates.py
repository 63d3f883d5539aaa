"""Matrices with repeated coordinates: their values are summed in input order by the packer for matrices itself, at
repeats inside a bucket, at its edges, in many buckets, in long rows and in inputs of every size class."""
import numpy as np
import pytest

from gpu_util import MATRIX_ENCODINGS, assert_storage_equal, sp, to_dev
from paper_2202_04305_b200 import inputs as I

pytestmark = pytest.mark.gpu


def _coo(rows, cols, dims, seed):
    """The entries in random order; values of very different sizes, so that the order of a sum shows."""
    rng = np.random.default_rng(seed)
    o = rng.permutation(rows.size)
    vals = I.uniform_pm1(seed, 5, rows.size) * 10.0 ** rng.integers(-8, 9, rows.size)
    return I.Coo(dims, [rows[o].astype(np.int64), cols[o].astype(np.int64)], vals)


def _random(m, n, nnz, distinct, seed):
    rng = np.random.default_rng(seed)
    key = rng.choice(m * n, distinct, replace=False)
    key = np.concatenate([key, rng.choice(key, nnz - distinct)])
    return _coo(key // n, key % n, (m, n), seed)


def _case(name):
    rng = np.random.default_rng(11)
    if name == "one_pair":
        return _random(300, 64, 6001, 6000, 1)
    if name == "one_coordinate":                                   # a bucket of nothing else
        return _coo(np.full(300, 2), np.full(300, 5), (4, 9), 2)
    if name == "full_bucket_of_one":
        return _coo(np.full(5120, 2), np.full(5120, 5), (4, 9), 2)
    if name == "first_and_last":                                   # of the matrix, and so of the first and the last bucket
        c = _random(900, 70, 9000, 9000, 3)
        rows = np.r_[c.coords[0], np.repeat([0, 899], 40)]
        cols = np.r_[c.coords[1], np.repeat([0, 69], 40)]
        return _coo(rows, cols, c.dims, 3)
    if name == "every_bucket":
        return _random(5000, 5000, 40000, 10000, 4)
    if name == "long_rows":                                        # cut into bins
        rows, cols = np.repeat(np.arange(30), 600), rng.integers(0, 400, 18000)
        return _coo(rows, cols, (30, 400), 5)
    if name == "wide":
        rows, cols = rng.integers(0, 50, 3000), (1 << 32) - 2 - rng.integers(0, 40, 3000)
        return _coo(rows, cols, (50, (1 << 32) - 1), 6)
    if name == "empty_buckets":
        rows = np.r_[np.repeat(np.arange(100), 6), 70000 + np.repeat(np.arange(100), 6)]
        return _coo(rows, rng.integers(0, 4, rows.size), (80000, 4), 7)
    if name == "tiles":
        return _random(4000, 3000, 120000, 60000, 8)
    if name == "many_tiles":
        return _random(30000, 3000, 400001, 100000, 9)
    if name == "counted":
        return _random(200000, 3000, 2000003, 1000000, 10)
    if name == "counted_few_entries":
        return _random(3000000, 50, 3001, 2000, 11)
    raise KeyError(name)


CASES = ["one_pair", "one_coordinate", "full_bucket_of_one", "first_and_last", "every_bucket", "long_rows", "wide", "empty_buckets", "tiles",
         "many_tiles", "counted", "counted_few_entries"]


@pytest.mark.parametrize("enc", list(MATRIX_ENCODINGS))
@pytest.mark.parametrize("name", CASES)
def test_duplicates_are_summed_in_input_order(oracle, name, enc):
    lt, od = MATRIX_ENCODINGS[enc]
    coo = _case(name)
    if od == (1, 0):
        coo = I.Coo(coo.dims[::-1], coo.coords[::-1], coo.vals)
    ref = oracle.pack(coo.dims, coo.coords, coo.vals, lt, od)
    for bits, pb, cb in ((32, 32, 32), (64, 64, 64)):
        if bits == 32 and max(coo.dims) > 1 << 31:
            continue
        coords, vals = to_dev(coo, bits)
        before = sp().sp_launch_count()
        A = sp().sp_pack(coo.dims, coords, vals, lt, od, pb, cb)
        assert sp().sp_launch_count() - before <= 6, "packed twice"
        assert A.nval == ref.val.size < coo.vals.size
        assert_storage_equal(A, ref)
        if od == (1, 0):                                           # the columns kept for SpMM, by the product with ones
            out = sp().sp_spmm(A, vals.new_ones((coo.dims[1], 1))).cpu().numpy() if max(coo.dims) < 1 << 24 else None
            if out is not None:
                want, bound = oracle.spmm(coo.dims[0], coo.coords[0], coo.coords[1], coo.vals, np.ones((coo.dims[1], 1)))
                assert np.all(np.abs(out - want) <= 1e-12 * bound)
        with pytest.raises(sp().SpError) as e:
            sp().sp_pack(coo.dims, coords, vals, lt, od, pb, cb, sp().DUP_ERROR)
        assert e.value.code == 5


def test_out_of_range_comes_before_duplicates():
    b = sp()
    coo = _case("every_bucket")
    coords, vals = to_dev(coo)
    coords[1][17] = coo.dims[1]
    for flags in (b.DUP_SUM, b.DUP_ERROR):
        with pytest.raises(b.SpError) as e:
            b.sp_pack(coo.dims, coords, vals, (0, 1), None, 32, 32, flags)
        assert e.value.code == 3


def test_a_failed_allocation_while_duplicates_are_closed_up():
    from test_gpu_alloc_failure import FailingAllocator, sweep
    coo = _case("every_bucket")
    coords, vals = to_dev(coo)
    for enc in ("CSR", "DCSC"):
        lt, od = MATRIX_ENCODINGS[enc]
        with FailingAllocator() as a:
            assert sweep(a, lambda: sp().sp_pack(coo.dims, coords, vals, lt, od)) >= 3
        assert not a.live
