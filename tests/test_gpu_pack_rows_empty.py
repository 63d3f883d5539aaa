"""DCSR and DCSC of matrices whose rows or columns far outnumber the entries: both sides of the line from which they are
sorted instead of sent to buckets."""
import numpy as np
import pytest

from gpu_util import MATRIX_ENCODINGS, assert_storage_equal, sp, to_dev
from paper_2202_04305_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("enc", ["DCSR", "DCSC"])
@pytest.mark.parametrize("nnz,outer,sorted_", [(1000, 3_002_000, False), (1000, 3_002_001, True), (1, 3_000_002, False), (1, 8_000_000, True),
                                               (300_000, 3_600_000, False), (300_000, 3_600_001, True)])
def test_more_rows_than_entries(oracle, enc, nnz, outer, sorted_):
    rng = np.random.default_rng(nnz)
    lt, od = MATRIX_ENCODINGS[enc]
    key = np.unique(rng.integers(0, outer * 700, nnz - 1))
    key = np.r_[key, outer * 700 - 1] if nnz == 1 or key[-1] != outer * 700 - 1 else key
    extra = nnz - key.size
    rows, cols = np.r_[key // 700, key[:extra] // 700], np.r_[key % 700, key[:extra] % 700]     # a few repeated
    o = rng.permutation(nnz)
    c = [rows[o].astype(np.int64), cols[o].astype(np.int64)]
    coo = I.Coo((outer, 700), c, I.uniform_pm1(1, 5, nnz)) if od == (0, 1) else I.Coo((700, outer), c[::-1], I.uniform_pm1(1, 5, nnz))
    ref = oracle.pack(coo.dims, coo.coords, coo.vals, lt, od)
    before = sp().sp_launch_count()
    A = sp().sp_pack(coo.dims, *to_dev(coo), lt, od)
    assert (sp().sp_launch_count() - before > 6) == sorted_
    assert_storage_equal(A, ref)
