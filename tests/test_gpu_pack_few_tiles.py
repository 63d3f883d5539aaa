"""Packing of rank-3 tensors by the radix sort where a scatter adds up the tile counts itself: entry counts at the
edges of its tiles, at the change of the tile's size and at the last count that goes without scan kernels."""
import numpy as np
import pytest

from gpu_util import assert_storage_equal, sp, to_dev
from paper_2202_04305_b200 import inputs as I

pytestmark = pytest.mark.gpu

SMALL = (96, 80, 72)                     # the entry index fits beside the key
WIDE = (1 << 21, 1 << 20, 1 << 21)       # it does not: values travel beside their keys, in tiles of 2048


@pytest.mark.parametrize("dims,n", [(SMALL, n) for n in (1, 1023, 1024, 1025, 65535, 65536, 65537, 262144, 262145)]
                         + [(WIDE, n) for n in (2, 2048, 2049, 131072, 131073)])
def test_pack_few_tiles(oracle, dims, n):
    rng = np.random.default_rng(n)
    cells = rng.choice(int(np.prod(SMALL)), n, replace=False)
    coords = [c.astype(np.int64) for c in np.unravel_index(cells, SMALL)]
    coords = [c * (d // s) for c, d, s in zip(coords, dims, SMALL)]
    coo = I.Coo(dims, coords, I.uniform_pm1(n, 5, n))
    c, v = to_dev(coo)
    T = sp().sp_pack(coo.dims, c, v, (1, 1, 1), (2, 0, 1))
    assert_storage_equal(T, oracle.pack(coo.dims, coo.coords, coo.vals, (1, 1, 1), (2, 0, 1)))
