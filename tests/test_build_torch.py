"""The binding's torch side is rebuilt for another torch, and only then (no compiler is run here)."""
import os

import torch

from paper_2202_04305_b200 import build


def test_another_torch_gets_its_own_library(tmp_path, monkeypatch):
    lib, runs = tmp_path / "libsp_torch.so", []
    monkeypatch.setattr(build, "LIB_TORCH", str(lib))
    monkeypatch.setattr(build, "OBJ", str(tmp_path / "objects"))

    def compile_(cmd):
        runs.append(cmd)
        lib.write_bytes(b"")
    monkeypatch.setattr(build.subprocess, "check_call", compile_)
    lib.write_bytes(b"")                                           # from before, for no known torch
    build.build_torch()
    assert len(runs) == 1
    build.build_torch()
    assert len(runs) == 1
    monkeypatch.setattr(torch, "__version__", "0.0.0+other")
    build.build_torch()
    assert len(runs) == 2
    build.build_torch()
    assert len(runs) == 2
    os.utime(lib, (1, 1))                                          # older than its source
    build.build_torch()
    assert len(runs) == 3
