"""Row-major SpMM at the edges of its pieces: rows that span many pieces and blocks, runs of rows without
entries, gaps between stored rows, and output widths on both sides of every tile width."""
import numpy as np
import pytest

from gpu_util import assert_close, dev, sp, to_dev
from paper_2202_04305_b200 import inputs as I

pytestmark = pytest.mark.gpu


def _rows(lens, n, seed):
    """One matrix with the given row lengths, distinct random columns per row, entries in random order."""
    rng = np.random.default_rng(seed)
    rows = np.repeat(np.arange(len(lens)), lens)
    cols = np.concatenate([rng.choice(n, k, replace=False) for k in lens if k] or [np.empty(0, np.int64)])
    order = rng.permutation(rows.size)
    return I.Coo((len(lens), n), [rows[order].astype(np.int64), cols[order].astype(np.int64)], I.uniform_pm1(seed, 5, rows.size))


PATTERNS = {
    "one_entry": [0, 1, 0],
    "long_rows": [1, 3000, 0, 0, 2500, 1],                        # a row over many pieces and blocks
    "piece_edges": [31, 1, 32, 33, 63, 64, 65, 0, 0, 127, 128, 129],
    "empty_runs": [0] * 700 + [5, 0, 0, 7] + [0] * 900 + [40] + [0] * 300,
    "single_entries": [1] * 2000,
    "ends_full": [0] * 129 + [2, 2] + [0] * 130 + [64] * 20,
    "many_pieces": [16, 0, 48, 3] * 4800 + [0] * 50,              # more than 300,000 items: the longer pieces
}


@pytest.mark.parametrize("lt", [(0, 1), (1, 1)], ids=["csr", "dcsr"])
@pytest.mark.parametrize("name", list(PATTERNS))
def test_spmm_pieces(oracle, name, lt):
    import torch
    lens = PATTERNS[name]
    coo = _rows(lens, 3100, 11)
    coords, vals = to_dev(coo)
    A = sp().sp_pack(coo.dims, coords, vals, lt)
    for N in (1, 8, 9, 16, 17, 18, 32, 33, 48, 49, 64, 66, 128, 130):
        B = I.dense_operand(3, N, coo.dims[1], N)
        ref, bd = oracle.spmm(coo.dims[0], coo.coords[0], coo.coords[1], coo.vals, B)
        out = torch.full((coo.dims[0], N + 3), 7.0, dtype=torch.float64, device="cuda")
        for C in (out[:, :N], torch.full((coo.dims[0], N), 7.0, dtype=torch.float64, device="cuda")):
            assert_close(sp().sp_spmm(A, dev(B), C).cpu().numpy(), ref, bd, f"{name} N={N}")
        assert torch.all(out[:, N:] == 7.0)


def test_spmm_infinite_operand_rows_stay_where_they_belong():
    """A row of B with an infinity reaches exactly the rows of C that use it."""
    lens = [3, 0, 70, 1, 2]
    coo = _rows(lens, 200, 4)
    coords, vals = to_dev(coo)
    A = sp().sp_pack(coo.dims, coords, vals, (0, 1))
    B = I.dense_operand(3, 1, 200, 32)
    hit = int(coo.coords[1][0])
    B[hit, 5] = np.inf
    C = sp().sp_spmm(A, dev(B)).cpu().numpy()
    uses = np.zeros(5, bool)
    uses[coo.coords[0][coo.coords[1] == hit]] = True
    assert np.array_equal(np.isinf(C[:, 5]), uses) and np.all(np.isfinite(np.delete(C, 5, axis=1)))
