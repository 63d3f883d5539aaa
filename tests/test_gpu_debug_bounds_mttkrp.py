"""The bounds-checking build and the coordinates that MTTKRP lays out in words before its first product: a slice or fibre
coordinate out of range, also one that a word could not hold, makes that call report status 3 instead of going unnoticed."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import torch
import oracle as O
import paper_2202_04305_b200.binding as sp
from paper_2202_04305_b200 import inputs as I
from gpu_util import assert_close, dev, to_dev

assert sp.DEBUG_BOUNDS
t = I.config5(seed=3, dim=96, nnz=20000)
tc, tv = to_dev(t)
for R in (8, 17):
    Bf, Cf = I.dense_operand(3, 37, 96, R), I.dense_operand(3, 38, 96, R)
    ref, bound = O.mttkrp(96, *t.coords, t.vals, Bf, Cf)
    for level in (0, 1):
        for bad in (96, 96 + 5, (1 << 30) + 5):
            T = sp.sp_pack(t.dims, tc, tv, (1, 1, 1))
            c = T.coordinates(level)
            at = 0 if level == 0 else 11
            keep = int(c[at])
            c[at] = bad
            try:
                sp.sp_mttkrp(T, dev(Bf), dev(Cf))
            except sp.SpError as e:
                assert e.code == 3, e.code
            else:
                raise AssertionError(f"level {level}: {bad} went unnoticed")
            c[at] = keep
            assert_close(sp.sp_mttkrp(T, dev(Bf), dev(Cf)).cpu().numpy(), ref, bound, "after repair")
torch.cuda.synchronize()
print("words checked")
"""


def test_coordinates_are_checked_where_the_words_are_made():
    from paper_2202_04305_b200 import build
    build.build(debug_bounds=True)
    env = dict(os.environ, SP_DEBUG_BOUNDS="1", PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")]))
    r = subprocess.run([sys.executable, "-c", CHILD], env=env, cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "words checked" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
