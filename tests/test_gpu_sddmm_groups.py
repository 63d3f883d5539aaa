"""SDDMM at the edges of its lane groups and pieces: every K around a group's width, rows that span pieces,
runs of rows without samples, operands off the 16-byte grid, and row- and column-major storage."""
import numpy as np
import pytest

from gpu_util import MATRIX_ENCODINGS, assert_close, dev, sp, to_dev
from paper_2202_04305_b200 import inputs as I

pytestmark = pytest.mark.gpu

KS = (1, 2, 3, 4, 15, 16, 17, 31, 32, 33, 50, 63, 64, 65, 95, 96, 97, 100, 127, 128, 129, 255, 256, 257, 511, 512, 513, 514)


@pytest.mark.parametrize("enc", list(MATRIX_ENCODINGS))
@pytest.mark.parametrize("shift", [0, 1], ids=["aligned", "odd_rows"])
def test_sddmm_widths(oracle, enc, shift):
    import torch
    rng = np.random.default_rng(5)
    lens = [1, 90, 0, 0, 3, 4, 5, 15, 16, 17, 1, 1, 1] + [0] * 40 + [33, 2, 0]
    m, n = len(lens), 120
    rows = np.repeat(np.arange(m), lens)
    cols = np.concatenate([rng.choice(n, k, replace=False) for k in lens])
    order = rng.permutation(rows.size)
    coo = I.Coo((m, n), [rows[order].astype(np.int64), cols[order].astype(np.int64)], I.uniform_pm1(5, 5, rows.size))
    lt, od = MATRIX_ENCODINGS[enc]
    coords, vals = to_dev(coo)
    S = sp().sp_pack(coo.dims, coords, vals, lt, od)
    (si, sj), sv = oracle.unpack(oracle.pack(coo.dims, coo.coords, coo.vals, lt, od))
    for K in KS:
        A, B = I.dense_operand(5, 8, m, K), I.dense_operand(5, 9, K, n)
        ref, bound = oracle.sddmm(si, sj, sv, A, B)
        wide = torch.full((m, K + K % 2 + shift), 1e300, dtype=torch.float64, device="cuda")
        wide[:, :K] = dev(A)
        out = torch.full((S.nval + 2,), 7.0, dtype=torch.float64, device="cuda")
        sp().sp_sddmm(S, wide[:, :K], dev(B), out[1:-1])
        assert_close(out[1:-1].cpu().numpy(), ref, bound, f"K={K}")
        assert out[0] == 7.0 and out[-1] == 7.0


def test_sddmm_many_pieces(oracle):
    """More than 200,000 row ends and samples: the longer pieces."""
    coo = I.uniform_matrix(9000, 7000, 220000, seed=3)
    coords, vals = to_dev(coo)
    S = sp().sp_pack(coo.dims, coords, vals, (0, 1))
    ref = oracle.pack(coo.dims, coo.coords, coo.vals, (0, 1))
    (si, sj), sv = oracle.unpack(ref)
    for K in (20, 96, 128):
        A, B = I.dense_operand(6, 8, 9000, K), I.dense_operand(6, 9, K, 7000)
        xr, xb = oracle.sddmm(si, sj, sv, A, B)
        assert_close(sp().sp_sddmm(S, dev(A), dev(B)).cpu().numpy(), xr, xb, f"K={K}")
