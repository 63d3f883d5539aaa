"""Column-major SpMM at the edges of its lane groups: every width around a group's columns, entries that do not fill a
warp, and operands whose rows lie apart or off the 16-byte grid."""
import numpy as np
import pytest

from gpu_util import assert_close, dev, sp, to_dev
from paper_2202_04305_b200 import inputs as I

pytestmark = pytest.mark.gpu

NS = (1, 7, 8, 9, 16, 17, 20, 24, 25, 32, 33, 48, 63, 64, 65, 96, 100, 127, 128, 129, 200)


@pytest.mark.parametrize("lt", [(0, 1), (1, 1)], ids=["csc", "dcsc"])
@pytest.mark.parametrize("nnz", [1, 31, 32, 33, 127, 129, 5003])
def test_spmm_scatter_widths(oracle, lt, nnz):
    import torch
    coo = I.uniform_matrix(90, 140, nnz, seed=nnz)
    coords, vals = to_dev(coo, 32 if nnz % 2 else 64)
    A = sp().sp_pack(coo.dims, coords, vals, lt, (1, 0))
    for N in NS:
        B = I.dense_operand(3, N, coo.dims[1], N)
        ref, bound = oracle.spmm(coo.dims[0], coo.coords[0], coo.coords[1], coo.vals, B)
        wide = torch.full((coo.dims[1], N + 3), 1e300, dtype=torch.float64, device="cuda")
        wide[:, 1:N + 1] = dev(B)
        out = torch.full((coo.dims[0], N + 3), 7.0, dtype=torch.float64, device="cuda")
        assert_close(sp().sp_spmm(A, wide[:, 1:N + 1], out[:, 1:N + 1]).cpu().numpy(), ref, bound, f"N={N}")
        assert torch.all(out[:, :1] == 7.0) and torch.all(out[:, N + 1:] == 7.0)
