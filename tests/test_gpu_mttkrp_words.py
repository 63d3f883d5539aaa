"""The words that MTTKRP lays out per entry are a handle's, not a number of columns': one table serves every R, and a
call captured with one R may have been warmed up with another."""
import numpy as np
import pytest

from gpu_util import assert_close, dev, sp, to_dev
from paper_2202_04305_b200 import inputs as I
from test_gpu_pack_scratch import Meter

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nnz", [30_000, 1_000_100])
def test_one_table_for_every_number_of_columns(oracle, nnz):
    import torch
    dims = (300, 250, 200)
    t = I.uniform_tensor(dims, nnz, seed=4)
    coords, vals = to_dev(t)
    F = {R: (I.dense_operand(4, R, dims[1], R), I.dense_operand(5, R, dims[2], R)) for R in (32, 48, 17, 8)}
    D = {R: (dev(a), dev(b)) for R, (a, b) in F.items()}
    M = {R: torch.empty(dims[0], R, dtype=torch.float64, device="cuda") for R in F}
    with Meter() as m:
        T = sp().sp_pack(dims, coords, vals, (1, 1, 1))
        sp().sp_mttkrp(T, *D[32], M[32])
        held = m.held
        for R in F:
            sp().sp_mttkrp(T, *D[R], M[R])
            assert m.held == held, f"R = {R} added {m.held - held} bytes to the handle"
        T.free()
    T = sp().sp_pack(dims, coords, vals, (1, 1, 1))
    sp().sp_mttkrp(T, *D[32], M[32])                       # the only call outside the graph
    torch.cuda.synchronize()
    g, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(side), torch.cuda.graph(g, stream=side):
        for R in (48, 17, 8):
            sp().sp_mttkrp(T, *D[R], M[R])
    for R in (48, 17, 8):
        M[R].fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    for R in F:
        ref, bound = oracle.mttkrp(dims[0], *t.coords, t.vals, *F[R])
        assert_close(M[R].cpu().numpy(), ref, bound, f"R={R}")
