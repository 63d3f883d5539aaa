"""The routes of sp_spmspm: rows of A around the length from which a block takes them instead of a warp, results that fit
shared memory and that do not, and operands on both sides of the lines between the bitmaps and a block per row."""
import numpy as np
import pytest

from gpu_util import assert_close, sp, to_dev, unsigned
from paper_2202_04305_b200 import inputs as I

pytestmark = pytest.mark.gpu

BLOCKS, BITMAPS, BITMAPS_LONG = 3, 5, 6                     # launches


def _matrix(lens, n, seed):
    rng = np.random.default_rng(seed)
    rows = np.repeat(np.arange(len(lens)), lens)
    cols = np.concatenate([rng.choice(n, k, replace=False) for k in lens])
    return I.Coo((len(lens), n), [rows.astype(np.int64), cols.astype(np.int64)], I.uniform_pm1(seed, 5, rows.size))


def _check(oracle, A, B, launches, bits=32):
    hA = sp().sp_pack(A.dims, *to_dev(A, bits), (0, 1), None, bits, bits)
    hB = sp().sp_pack(B.dims, *to_dev(B, bits), (0, 1), None, bits, bits)
    before = sp().sp_launch_count()
    hC = sp().sp_spmspm(hA, hB, bits, bits)
    assert sp().sp_launch_count() - before == launches
    pos, crd, val, bd = oracle.spmspm(A.dims[0], A.dims[1], B.dims[1], A.coords[0], A.coords[1], A.vals, B.coords[0], B.coords[1], B.vals)
    assert np.array_equal(unsigned(hC.positions(1)), pos)
    assert np.array_equal(unsigned(hC.coordinates(1)), crd)
    assert_close(hC.values().cpu().numpy(), val, bd, "spmspm")


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("n,per", [(3000, 50), (25600, 60), (30000, 70)])
def test_rows_much_longer_than_the_others(oracle, n, per, bits):
    lens = [45] * 600 + [0, 512, 513, 1300, 1, 700]
    B = _matrix([per] * 1299 + [0], n, 2)
    _check(oracle, _matrix(lens, 1300, 1), B, BITMAPS_LONG, bits)
    _check(oracle, _matrix([45] * 600 + [512], 1300, 3), B, BITMAPS, bits)


def test_rows_long_against_their_mean(oracle):
    """Rows of 200 on average: longer than 800 entries counts, 512 does not."""
    B = _matrix([60] * 2000, 2000, 4)
    _check(oracle, _matrix([200] * 1700 + [801, 800], 2000, 5), B, BITMAPS_LONG)
    _check(oracle, _matrix([200] * 1700 + [799, 700], 2000, 5), B, BITMAPS)


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("n", [9000, 25000])
def test_few_entries_a_row_in_shared_memory(oracle, n, bits):
    rng = np.random.default_rng(n)
    A, B = _matrix(rng.integers(0, 30, 500), 400, 6), _matrix(rng.integers(1, 6, 400), n, 7)
    _check(oracle, A, B, BLOCKS, bits)


@pytest.mark.parametrize("na,nb,n,launches", [(60, 24, 1000, BITMAPS), (60, 23, 1000, BLOCKS), (5, 24, 1000, BITMAPS), (4, 24, 1000, BLOCKS),
                                              (2, 50, 1000, BITMAPS), (1, 90, 1000, BLOCKS), (60, 38, 9000, BITMAPS), (60, 37, 9000, BLOCKS)])
def test_lines_between_the_routes(oracle, na, nb, n, launches):
    """100 products a row and block of columns; rows of B of 24 entries for 1,000 columns, of 38 for 9,000."""
    _check(oracle, _matrix([na] * 700, 800, 8), _matrix([nb] * 800, n, 9), launches)
