"""Unpacking matrices by tiles where segments are few, many or mostly empty: spans on both sides of the longest that a
block goes over (4096 segments for 1024 entries), gaps at the ends and in the middle, tiles just full and one over."""
import numpy as np
import pytest

from gpu_util import MATRIX_ENCODINGS, sp, to_dev, unsigned
from paper_2202_04305_b200 import inputs as I

pytestmark = pytest.mark.gpu


def _rows(kind):
    """Row numbers of the entries, in order, and the number of rows."""
    if kind.startswith("span"):                                   # one tile whose first and last rows are that far apart
        span = int(kind[4:])
        return np.r_[np.zeros(500, np.int64), np.full(300, span // 2), np.full(224, span)], span + 1
    return {
        "single": (np.array([70000]), 100000),
        "ends": (np.r_[np.zeros(1000, np.int64), np.full(1, 65000), np.full(1500, 69999)], 70000),
        "every_hundredth": (np.arange(0, 300000, 100), 300001),
        "gap_between_tiles": (np.r_[np.repeat(np.arange(512), 2), 50000 + np.repeat(np.arange(512), 2)], 60000),
        "gap_inside_a_tile": (np.r_[np.repeat(np.arange(500), 2), 50000 + np.repeat(np.arange(525), 2)], 60000),
    }[kind]


@pytest.mark.parametrize("enc", list(MATRIX_ENCODINGS))
@pytest.mark.parametrize("kind", ["single", "ends", "every_hundredth", "gap_between_tiles", "gap_inside_a_tile", "span4095", "span4096", "span4097"])
def test_unpack_returns_the_entries(kind, enc):
    rows, m = _rows(kind)
    n = 1600
    cols = (np.arange(rows.size) * 7) % n
    key = np.unique(rows * n + cols)                              # distinct, in row order
    rows, cols = key // n, key % n
    lt, od = MATRIX_ENCODINGS[enc]
    dims, coords = ((m, n), [rows, cols]) if od == (0, 1) else ((n, m), [cols, rows])
    coo = I.Coo(dims, coords, I.uniform_pm1(3, 5, rows.size))
    for bits in (32, 64):
        A = sp().sp_pack(dims, *to_dev(coo, bits), lt, od, bits, bits)
        out, vals = sp().sp_unpack(A)
        for d in range(2):
            assert np.array_equal(unsigned(out[d]), coords[d])
        assert np.array_equal(vals.cpu().numpy(), coo.vals)


def test_few_entries_in_many_rows_cost_no_walk_over_the_rows():
    """1,000 entries in 10,000,000 rows: tens of microseconds; going over the rows between them takes 7.7 ms."""
    import torch
    b = sp()
    m = 10_000_000
    rows = torch.arange(1000, device="cuda", dtype=torch.int32) * 10000
    A = b.sp_pack((m, 1000), [rows, rows % 1000], rows.double(), (0, 1))
    b.sp_unpack(A)
    ts = []
    for _ in range(5):
        s, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        s.record()
        b.sp_unpack(A)
        e.record()
        torch.cuda.synchronize()
        ts.append(s.elapsed_time(e))
    assert min(ts) < 1.0
