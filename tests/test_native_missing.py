"""A library built elsewhere, on a machine that cannot build the binding's extension module, or holds one that does not load."""
import subprocess

import pytest
import torch

from paper_2512_07503_b200 import binding as B


@pytest.mark.parametrize("error", [FileNotFoundError("g++"), subprocess.CalledProcessError(1, "g++"), RuntimeError("nvcc not found"),
                                   ImportError("undefined symbol"), PermissionError("read-only folder")])
def test_the_library_loads_without_it(monkeypatch, error):
    B.lib()

    def fail(*a, **k):
        raise error

    monkeypatch.setattr(B, "_lib", None)
    monkeypatch.setattr(B, "_native", None)
    monkeypatch.setattr(B._build, "build_native", fail)
    with pytest.warns(RuntimeWarning, match="extension module"):
        assert B.sjd_version() == 1
    p = B.sjd_params()
    for _ in range(2):  # the way through ctypes, which words the refusals
        with pytest.raises(B.SjdError, match="CUDA device"):
            B.sjd_step(torch.zeros(1, 1, 8), None, None, None, p, 0, None, None, None)
    with pytest.raises(B.SjdError, match="contiguous CUDA"):
        B.sjd_window_advance(p, 4, 0, None, torch.zeros(1, 1, dtype=torch.int32), B.DeviceProbs.empty(1, 1, 1, "cpu"), *[None] * 4,
                             B.DeviceProbs.empty(1, 1, 1, "cpu"), None)
