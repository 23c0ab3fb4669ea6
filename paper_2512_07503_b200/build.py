"""Compile the CUDA library (libsjd.so) in-tree for sm_100a with nvcc, and the binding's extension module (_native.*.so) with the host compiler."""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
_CSRC = os.path.join(_PKG, "csrc")
_INC = os.path.join(os.path.dirname(_PKG), "include")
LIB_PATH = os.path.join(_PKG, "libsjd.so")
NATIVE_SOURCE = os.path.join(_CSRC, "binding_native.cpp")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-shared",
              "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", "--extended-lambda"]


def _nvcc() -> str:
    for c in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found: the CUDA library cannot be built")


def sources():
    return sorted(glob.glob(os.path.join(_CSRC, "*.cu")))


def _deps():
    return sources() + glob.glob(os.path.join(_CSRC, "*.cuh")) + glob.glob(os.path.join(_CSRC, "*.h")) + glob.glob(os.path.join(_INC, "*.h"))


def is_stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    return any(os.path.getmtime(p) > t for p in _deps())


def native_path() -> str:
    """Where the extension module lies that fits this interpreter and this PyTorch.  It is compiled against the layouts of both, so their versions
    are part of its name: after a change of either it is another file, and one that fits the new ones is built."""
    import torch
    fits = [sysconfig.get_config_var("SOABI"), "torch" + torch.__version__, (torch.version.git_version or "")[:8],
            "cxx11" if torch.compiled_with_cxx11_abi() else "cxx98"]
    return os.path.join(_PKG, "_native." + ".".join(str(x) for x in fits) + ".so")


def _native_command(out: str, first_includes=()) -> list:
    import torch
    at = os.path.join(os.path.dirname(torch.__file__), "include")
    libs = ["-L" + os.path.join(os.path.dirname(torch.__file__), "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10"]
    cuda = os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include")
    includes = [*first_includes, at, os.path.join(at, "torch", "csrc", "api", "include"), cuda, sysconfig.get_paths()["include"]]
    # (torch is imported before the module: the libraries named here are loaded already)
    return [shutil.which("g++") or "g++", "-O2", "-std=c++20", "-shared", "-fPIC", *[f"-I{d}" for d in includes], NATIVE_SOURCE, "-o", out, *libs]


def build_native(force: bool = False) -> str:
    """The extension module that binding.py calls the library's per-step functions through."""
    path = native_path()
    deps = [NATIVE_SOURCE] + glob.glob(os.path.join(_INC, "*.h"))
    if not force and os.path.exists(path) and all(os.path.getmtime(p) <= os.path.getmtime(path) for p in deps):
        return path
    tmp = path + f".tmp{os.getpid()}"
    subprocess.check_call(_native_command(tmp))
    os.replace(tmp, path)
    return path


def build_native_variant(out_path: str, first_includes) -> str:
    """The extension module with other headers found first (test builds: a stand-in for the CUDA device functions), written to `out_path`."""
    subprocess.check_call(_native_command(out_path, first_includes))
    return out_path


def build(force: bool = False, verbose: bool = False) -> str:
    override = os.environ.get("SJD_LIBRARY")
    if override:  # a library built elsewhere (the tests build variants with build_variant())
        return override
    if not force and not is_stale():
        return LIB_PATH
    tmp = LIB_PATH + f".tmp{os.getpid()}"
    cmd = [_nvcc(), *NVCC_FLAGS, "-I", _INC, *(["-Xptxas", "-v"] if verbose else []), *sources(), "-o", tmp]
    subprocess.check_call(cmd)
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


def build_variant(out_path: str, defines) -> str:
    """The library with extra -D definitions (test builds: short wait limits, a dropped copy), written to
    `out_path`.  Load it in a process of its own by setting SJD_LIBRARY to that path."""
    cmd = [_nvcc(), *NVCC_FLAGS, "-I", _INC, *[f"-D{d}" for d in defines], *sources(), "-o", out_path]
    subprocess.check_call(cmd)
    return out_path


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose="-v" in sys.argv))
