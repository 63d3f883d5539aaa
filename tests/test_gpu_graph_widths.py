"""Graph capture after a warm-up with another operand width: what a handle's first product lays out serves every width."""
import numpy as np
import pytest
import torch

from gpu_util import MATRIX_ENCODINGS, assert_close, dev, sp, to_dev
from paper_2202_04305_b200 import inputs as I

pytestmark = pytest.mark.gpu


def _captured(call):
    g, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side), torch.cuda.graph(g, stream=side):
        call()
    return g


@pytest.mark.parametrize("enc", ["CSR", "DCSR"])
@pytest.mark.parametrize("warm,then", [(32, 64), (32, 50), (16, 33), (64, 32), (33, 16)])
def test_spmm(oracle, enc, warm, then):
    """B beyond 100 MB and even rows of more than 16 entries: widths 16 and 32 go another way than the others."""
    rng = np.random.default_rng(3)
    m, n = 400, 1 << 20
    rows = np.repeat(np.arange(m), 20)
    cols = np.concatenate([rng.choice(n, 20, replace=False) for _ in range(m)])
    o = rng.permutation(rows.size)
    coo = I.Coo((m, n), [rows[o].astype(np.int64), cols[o].astype(np.int64)], I.uniform_pm1(3, 5, rows.size))
    A = sp().sp_pack(coo.dims, *to_dev(coo), *MATRIX_ENCODINGS[enc])
    used = np.unique(cols)
    compact = np.searchsorted(used, coo.coords[1])

    def operand(N):
        B = torch.zeros(n, N, dtype=torch.float64, device="cuda")
        host = I.dense_operand(4, N, used.size, N)
        B[torch.as_tensor(used, device="cuda")] = dev(host)
        return B, host, torch.full((m, N), float("nan"), dtype=torch.float64, device="cuda")
    B, _, C = operand(warm)
    sp().sp_spmm(A, B, C)
    B, host, C = operand(then)
    g = _captured(lambda: sp().sp_spmm(A, B, C))
    C.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    ref, bound = oracle.spmm(m, coo.coords[0], compact, coo.vals, host)
    assert_close(C.cpu().numpy(), ref, bound, f"{enc} N={then} after N={warm}")


@pytest.mark.parametrize("warm,then", [(64, 600), (600, 64), (17, 513)])
@pytest.mark.parametrize("enc", list(MATRIX_ENCODINGS))
def test_sddmm(oracle, enc, warm, then):
    coo = I.uniform_matrix(150, 140, 2500, seed=5)
    S = sp().sp_pack(coo.dims, *to_dev(coo), *MATRIX_ENCODINGS[enc])
    x = torch.empty(S.nval, dtype=torch.float64, device="cuda")
    ops = {K: (I.dense_operand(3, K, 150, K), I.dense_operand(4, K, K, 140)) for K in (warm, then)}
    d = {K: (dev(a), dev(b)) for K, (a, b) in ops.items()}
    sp().sp_sddmm(S, *d[warm], x)
    g = _captured(lambda: sp().sp_sddmm(S, *d[then], x))
    x.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    e, b = oracle.sddmm(coo.coords[0], coo.coords[1], coo.vals, *ops[then])
    at = oracle.pack(coo.dims, coo.coords, coo.vals, *MATRIX_ENCODINGS[enc]).entry_pos
    ref, bound = np.empty_like(e), np.empty_like(b)
    ref[at], bound[at] = e, b
    assert_close(x.cpu().numpy(), ref, bound, f"{enc} K={then} after K={warm}")
