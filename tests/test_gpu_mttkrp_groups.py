"""MTTKRP by lane groups at its edges: every R around a group's width, fibres and slices that end on, before and
after the end of a group's range, one slice over many blocks, slices without entries, factors off the 16-byte grid."""
import numpy as np
import pytest

from gpu_util import assert_close, dev, sp, to_dev
from paper_2202_04305_b200 import inputs as I

pytestmark = pytest.mark.gpu

RS = (1, 2, 7, 8, 9, 15, 16, 17, 18, 23, 24, 25, 26, 31, 32, 33, 34, 47, 48, 49, 50, 63, 64, 65, 66, 128, 130)


def _tensor(fibres, dims, seed):
    """fibres: (i, j, entries) in any order; distinct random k in a fibre, entries in random order."""
    rng = np.random.default_rng(seed)
    i = np.repeat([f[0] for f in fibres], [f[2] for f in fibres])
    j = np.repeat([f[1] for f in fibres], [f[2] for f in fibres])
    k = np.concatenate([rng.choice(dims[2], f[2], replace=False) for f in fibres])
    o = rng.permutation(i.size)
    return I.Coo(dims, [i[o].astype(np.int64), j[o].astype(np.int64), k[o].astype(np.int64)], I.uniform_pm1(seed, 5, i.size))


TENSORS = {
    "one": ([(2, 1, 1)], (4, 3, 5)),
    "range_edges": ([(0, 0, 15), (0, 1, 1), (1, 0, 16), (1, 1, 17), (3, 2, 31), (3, 3, 1), (5, 0, 32), (9, 4, 33), (9, 5, 64)], (12, 7, 90)),
    "single_entries": ([(i, (i * 7) % 50, 1) for i in range(300)], (301, 50, 60)),
    "one_slice": ([(3, j, 1 + (j * 5) % 40) for j in range(200)], (5, 200, 64)),
    "gaps": ([(i, j, 3) for i in (0, 1, 40, 41, 199) for j in range(0, 30, 7)], (260, 30, 20)),
}


@pytest.mark.parametrize("lt", [(1, 1, 1), (0, 1, 1)], ids=["csf", "dss"])
@pytest.mark.parametrize("name", list(TENSORS))
def test_mttkrp_groups(oracle, name, lt):
    import torch
    fibres, dims = TENSORS[name]
    t = _tensor(fibres, dims, 3)
    coords, vals = to_dev(t)
    T = sp().sp_pack(dims, coords, vals, lt)
    for R in RS:
        B, C = I.dense_operand(4, R, dims[1], R), I.dense_operand(5, R, dims[2], R)
        ref, bound = oracle.mttkrp(dims[0], *t.coords, t.vals, B, C)
        out = torch.full((dims[0] * R + 3,), 7.0, dtype=torch.float64, device="cuda")
        for shift in (0, 1):
            flat = torch.empty(C.size + 1, dtype=torch.float64, device="cuda")
            Cd = flat[shift:shift + C.size].view(C.shape)
            Cd.copy_(dev(C))
            M = out[2 - shift:2 - shift + dims[0] * R].view(dims[0], R)
            assert_close(sp().sp_mttkrp(T, dev(B), Cd, M).cpu().numpy(), ref, bound, f"{name} R={R} shift={shift}")
        assert out[0] == 7.0 and out[-1] == 7.0


def test_mttkrp_longer_ranges(oracle):
    """Enough entries for ranges beyond the shortest, and for a slice over many blocks."""
    t = I.zipf_tensor3(300, 700000, 1.2, 9)
    coords, vals = to_dev(t)
    T = sp().sp_pack(t.dims, coords, vals, (1, 1, 1))
    for R in (17, 32, 50):
        B, C = I.dense_operand(4, R, 300, R), I.dense_operand(5, R, 300, R)
        ref, bound = oracle.mttkrp(300, *t.coords, t.vals, B, C)
        assert_close(sp().sp_mttkrp(T, dev(B), dev(C)).cpu().numpy(), ref, bound, f"R={R}")
