"""When the binding's extension module is compiled again (without a compiler: what it would be called with is recorded)."""
import os
import sysconfig

import pytest
import torch

from paper_2512_07503_b200 import build


@pytest.fixture
def compiled(monkeypatch, tmp_path):
    """The paths that the compiler was asked for, in a package folder of its own."""
    asked = []

    def compile_to(cmd):
        out = cmd[cmd.index("-o") + 1]
        open(out, "w").close()
        asked.append(out)

    source = tmp_path / "binding_native.cpp"
    source.write_text("")
    os.utime(source, (1, 1))
    monkeypatch.setattr(build, "_PKG", str(tmp_path))
    monkeypatch.setattr(build, "_INC", str(tmp_path))
    monkeypatch.setattr(build, "NATIVE_SOURCE", str(source))
    monkeypatch.setattr(build, "_nvcc", lambda: "/usr/local/cuda/bin/nvcc")
    monkeypatch.setattr(build.subprocess, "check_call", compile_to)
    return asked


def test_a_module_is_compiled_once(compiled):
    first = build.build_native()
    assert os.path.exists(first) and len(compiled) == 1
    assert build.build_native() == first and len(compiled) == 1
    os.utime(build.NATIVE_SOURCE, (2 ** 32, 2 ** 32))  # a newer source
    assert build.build_native() == first and len(compiled) == 2


@pytest.mark.parametrize("change", ["torch", "torch build", "python"])
def test_another_torch_or_python_gets_a_module_of_its_own(compiled, monkeypatch, change):
    first = build.build_native()
    if change == "torch":
        monkeypatch.setattr(torch, "__version__", "99.0")
    elif change == "torch build":
        monkeypatch.setattr(torch.version, "git_version", "0123456789abcdef")
    else:
        monkeypatch.setattr(sysconfig, "get_config_var", lambda name: "cpython-399-x86_64-linux-gnu")
    second = build.build_native()
    assert second != first and os.path.exists(first) and os.path.exists(second) and len(compiled) == 2
