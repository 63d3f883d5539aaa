"""Packing matrices without a sort by key: segment lengths at the edges of buckets and tiles, and the inputs
that have to take the radix path (a bucket that overflows, duplicates)."""
import numpy as np
import pytest

from gpu_util import MATRIX_ENCODINGS, assert_storage_equal, sp, to_dev
from paper_2202_04305_b200 import inputs as I

pytestmark = pytest.mark.gpu


def _matrix(lens, n, seed, repeat=0):
    """Rows of the given lengths, distinct columns within a row (then `repeat` entries once more), random order."""
    rng = np.random.default_rng(seed)
    rows = np.repeat(np.arange(len(lens)), lens)
    cols = np.concatenate([rng.choice(n, k, replace=False) for k in lens])
    order = rng.permutation(rows.size)
    rows, cols = rows[order], cols[order]
    rows, cols = np.concatenate([rows, rows[:repeat]]), np.concatenate([cols, cols[:repeat]])
    return I.Coo((len(lens), n), [rows.astype(np.int64), cols.astype(np.int64)], I.uniform_pm1(seed, 5, rows.size))


CASES = {
    "one_entry": ([1], 1, 0),
    "one_row": ([70], 90, 0),
    "full_bucket": ([4096], 5000, 0),
    "overfull_bucket": ([4097], 5000, 0),
    "full_among_others": ([5, 4000, 7] + [0] * 1990, 5000, 0),
    "far_too_long": ([3, 20000, 3], 30000, 0),
    "many_empty": ([0] * 5000 + [3] + [0] * 60000 + [1], 10, 0),
    "empty_buckets": ([1] * 2048 + [0] * 4096 + [1] * 2049, 50, 0),
    "bucket_edges": ([1, 2047, 2049, 0, 0, 1, 2047, 2, 2048] * 3, 2100, 0),
    "long_rows": ([500] * 40 + [0, 1, 2] * 20 + [1500] * 20, 1600, 0),       # cut into bins
    "many_tiles": ([30] * 20000, 60, 0),                                    # the larger tiles of entries
    "full_at_capacity": ([5120], 6000, 0),
    "over_capacity": ([5, 5121, 3], 6000, 0),
    "whole_tiles": ([32] * 12288, 40, 0),                                   # 128 tiles of 3072
    "one_entry_over": ([32] * 12288 + [1], 40, 0),
    "many_tiles_overfull": ([30] * 11000 + [5500] + [30] * 100, 6000, 0),
    "duplicates": ([20] * 300, 64, 17),
    "duplicates_in_bins": ([300] * 30, 400, 2),
}


@pytest.mark.parametrize("enc", list(MATRIX_ENCODINGS))
@pytest.mark.parametrize("name", list(CASES))
def test_pack_rows(oracle, name, enc):
    lens, n, repeat = CASES[name]
    lt, od = MATRIX_ENCODINGS[enc]
    coo = _matrix(lens, n, 3, repeat)
    if od == (1, 0):                                                # the lengths are those of the outer dimension
        coo = I.Coo(coo.dims[::-1], coo.coords[::-1], coo.vals)
    ref = oracle.pack(coo.dims, coo.coords, coo.vals, lt, od)
    for bits, pb, cb in ((32, 32, 32), (64, 64, 64), (32, 64, 32), (64, 32, 64)):
        coords, vals = to_dev(coo, bits)
        A = sp().sp_pack(coo.dims, coords, vals, lt, od, pb, cb)
        assert_storage_equal(A, ref)
        if repeat:
            with pytest.raises(sp().SpError) as e:
                sp().sp_pack(coo.dims, coords, vals, lt, od, pb, cb, sp().DUP_ERROR)
            assert e.value.code == 5
    coords[0][coords[0].numel() // 2] = coo.dims[0]                 # one coordinate past the end
    with pytest.raises(sp().SpError) as e:
        sp().sp_pack(coo.dims, coords, vals, lt, od)
    assert e.value.code == 3


def test_pack_rows_clustered_columns(oracle):
    """Long rows whose columns lie close together, at both ends of a wide matrix."""
    rng = np.random.default_rng(8)
    n = (1 << 32) - 1                                                # the widest that 32-bit coordinates hold
    rows = np.repeat(np.arange(12), 300)
    near = np.where(rows % 2 == 0, 0, n - 400)
    cols = np.concatenate([rng.choice(400, 300, replace=False) for _ in range(12)]) + near
    cols[5] = n - 1                                                  # one far away: all others of its row in one bin
    order = rng.permutation(rows.size)
    coo = I.Coo((12, n), [rows[order].astype(np.int64), cols[order].astype(np.int64)], I.uniform_pm1(8, 5, rows.size))
    coords, vals = to_dev(coo, 64)
    for lt in ((0, 1), (1, 1)):
        assert_storage_equal(sp().sp_pack(coo.dims, coords, vals, lt), oracle.pack(coo.dims, coo.coords, coo.vals, lt, (0, 1)))
