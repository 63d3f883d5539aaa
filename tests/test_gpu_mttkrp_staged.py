"""MTTKRP of tensors of a million entries and more: every width of the staged warps, with factors on and off the 32-byte
grid, fibres and slices that end on, before and after the ranges' 128 entries, slices without entries, 32- and 64-bit
storage; and the kernel for level-1 sizes that the entries' words cannot hold."""
import numpy as np
import pytest
import torch

from gpu_util import assert_close, dev, sp, to_dev
from paper_2202_04305_b200 import inputs as I

pytestmark = pytest.mark.gpu

DIMS = (900, 400, 700)


@pytest.fixture(scope="module")
def tensor():
    """Slices whose lengths add up to multiples of 128 at first, then arbitrary; some slices empty; 1,000,059 entries."""
    rng = np.random.default_rng(5)
    fibres, total = [], 0
    for i in range(40):                                            # fibres of 128, 64 and 1 + 127: ends on the ranges' ends
        for j in range(6):
            for length in ((128,), (64, 64), (1, 127), (127, 1), (32, 96))[(i + j) % 5]:
                fibres.append((i, len(fibres) % 400, length))
                total += length
    i = 41
    while total < 1_000_059:
        for j in range(int(rng.integers(1, 30))):
            length = int(min(rng.integers(1, 500), 1_000_059 - total))
            if length:
                fibres.append((i, j * 13, length))
                total += length
        i += 1 if i < 860 and rng.random() < 0.9 else 2
        i = min(i, 897)
    seen, rows = set(), []
    for a, b, length in fibres:                                    # a fibre's coordinates once
        while (a, b) in seen:
            b = (b + 1) % 400
        seen.add((a, b))
        rows.append((a, b, length))
    ii = np.repeat([f[0] for f in rows], [f[2] for f in rows])
    jj = np.repeat([f[1] for f in rows], [f[2] for f in rows])
    kk = np.concatenate([(rng.permutation(700)[:f[2]]) for f in rows])
    o = rng.permutation(ii.size)
    return I.Coo(DIMS, [ii[o].astype(np.int64), jj[o].astype(np.int64), kk[o].astype(np.int64)], I.uniform_pm1(5, 5, ii.size))


def _at(a, shift):
    """A copy of a on the device that starts `shift` doubles after a 256-byte boundary."""
    flat = torch.empty(a.size + 8, dtype=torch.float64, device="cuda")
    out = flat[shift:shift + a.size].view(a.shape)
    out.copy_(dev(a))
    return out


@pytest.mark.parametrize("R", [10, 12, 14, 16, 18, 22, 24, 26, 28, 30, 32])
def test_staged(oracle, tensor, R):
    t = tensor
    assert t.vals.size == 1_000_059
    B, C = I.dense_operand(4, R, DIMS[1], R), I.dense_operand(5, R, DIMS[2], R)
    ref, bound = oracle.mttkrp(DIMS[0], *t.coords, t.vals, B, C)
    for lt, bits in (((1, 1, 1), 32), ((0, 1, 1), 32), ((1, 1, 1), 64), ((0, 1, 1), 64)):
        T = sp().sp_pack(DIMS, *to_dev(t, bits), lt, None, bits, bits)
        for sb, sc in ((0, 0), (2, 0), (0, 2)):
            out = torch.full((DIMS[0] * R + 8,), 7.0, dtype=torch.float64, device="cuda")
            M = out[2:2 + DIMS[0] * R].view(DIMS[0], R)
            assert_close(sp().sp_mttkrp(T, _at(B, sb), _at(C, sc), M).cpu().numpy(), ref, bound, f"{lt} {bits} R={R} {sb} {sc}")
            assert bool((out[:2] == 7.0).all()) and bool((out[2 + DIMS[0] * R:] == 7.0).all())


@pytest.mark.parametrize("R", [1, 2])
@pytest.mark.parametrize("lt", [(1, 1, 1), (0, 1, 1)], ids=["csf", "dss"])
def test_level_1_beyond_the_words(oracle, lt, R):
    rng = np.random.default_rng(7)
    far = (1 << 29) + 8
    used = np.sort(rng.choice(far, 60, replace=False))
    used[-1] = far - 1
    key = np.unique(rng.integers(0, 5 * 60 * 300, 9000))           # slice 2 stays empty
    i, j, k = key // (60 * 300), key // 300 % 60, key % 300
    i = i + (i >= 2)
    o = rng.permutation(key.size)
    i, j, k = i[o], j[o], k[o]
    vals = I.uniform_pm1(7, 5, key.size)
    dims = (6, far, 300)
    coords = [torch.as_tensor(c, device="cuda").int() for c in (i, used[j], k)]
    T = sp().sp_pack(dims, coords, dev(vals), lt)
    B, C = I.dense_operand(4, R, 60, R), I.dense_operand(5, R, 300, R)
    F = torch.empty((far, R), dtype=torch.float64, device="cuda")  # only the rows that are used hold anything
    F[torch.as_tensor(used, device="cuda")] = dev(B)
    ref, bound = oracle.mttkrp(6, i, j, k, vals, B, C)
    assert_close(sp().sp_mttkrp(T, F, dev(C)).cpu().numpy(), ref, bound, f"{lt} R={R}")
