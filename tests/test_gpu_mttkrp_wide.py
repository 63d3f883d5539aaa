"""MTTKRP with more columns than one launch has tiles for (65,535 of 64 columns), odd and even counts."""
import numpy as np
import pytest
import torch

from gpu_util import sp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [65535 * 64, 65535 * 64 + 1, 65535 * 64 + 66])
def test_columns_beyond_one_launch(R):
    i, j, k = np.array([0, 1, 1]), np.array([1, 0, 1]), np.array([0, 1, 1])
    v = np.array([2.0, 3.0, -5.0])                                  # small integers: every product is exact
    T = sp().sp_pack((2, 2, 2), [torch.tensor(c, dtype=torch.int32, device="cuda") for c in (i, j, k)], torch.tensor(v, device="cuda"), (1, 1, 1))
    r = torch.arange(R, device="cuda", dtype=torch.float64)
    B = torch.stack([r % 13, r % 7 - 3])
    C = torch.stack([r % 11, 5 - r % 9])
    want = torch.stack([2 * B[1] * C[0], 3 * B[0] * C[1] - 5 * B[1] * C[1]])
    M = torch.full((2 * R + 1,), 7.0, dtype=torch.float64, device="cuda")
    assert torch.equal(sp().sp_mttkrp(T, B, C, M[:2 * R].view(2, R)), want)
    assert M[2 * R] == 7.0
