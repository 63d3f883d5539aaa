"""Packing from many short-lived host threads at once: each borrows its read-back words and no two share them."""
import threading

import pytest
import torch

from gpu_util import assert_storage_equal, sp, to_dev
from paper_2202_04305_b200 import inputs as I

pytestmark = pytest.mark.gpu


def test_threads_that_come_and_go(oracle):
    coo = I.uniform_matrix(300, 280, 6000, seed=5)
    coords, vals = to_dev(coo)
    ref = oracle.pack(coo.dims, coo.coords, coo.vals, (0, 1))
    for _ in range(3):                                             # 40 at once, one after the other has ended
        gate = threading.Barrier(40)
        got, errors = [], []

        def body():
            try:
                torch.cuda.set_device(0)
                with torch.cuda.stream(torch.cuda.Stream()):
                    sp().sp_pack(coo.dims, coords, vals, (0, 1)).free()
                    gate.wait(60)                                  # all hold their words now
                    got.append(sp().sp_pack(coo.dims, coords, vals, (0, 1)))
            except BaseException as e:                             # noqa: BLE001
                errors.append(e)
                gate.abort()
        torch.cuda.synchronize()
        ts = [threading.Thread(target=body) for _ in range(40)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
        assert not errors, errors[0]
        torch.cuda.synchronize()
        for A in got:
            assert_storage_equal(A, ref)
