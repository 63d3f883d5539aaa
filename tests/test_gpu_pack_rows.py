"""Packing matrices with short segments: lengths at the edges of the tiles and of the range that is packed
without a sort by key, and the inputs that have to fall back to it."""
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
    "tile_edge": ([2047, 1, 2048, 0, 0, 1, 2047, 2], 2100, 0),      # segments that end on, before and after a tile's edge
    "longest_taken": ([5, 2048, 7], 2100, 0),
    "too_long": ([5, 2049, 7], 2100, 0),
    "far_too_long": ([3, 20000, 3], 30000, 0),                      # counting gives up
    "many_empty": ([0] * 5000 + [3] + [0] * 60000 + [1], 10, 0),
    "empty_tiles": ([1] * 2048 + [0] * 4096 + [1] * 2049, 50, 0),
    "words": ([31, 33, 32, 64, 1, 0, 65] * 40, 300, 0),
    "duplicates": ([20] * 300, 64, 17),
    "squares_too_many": ([1500] * 100, 1600, 0),                    # within the longest segment, but too much counting
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
