"""The extension module's calls for tensors on a device that is not the current one, without a GPU: the module is built against a stand-in for PyTorch's
device functions, the tensors only say that they are on a device, and the library's functions are callbacks that note which one is current."""
import ctypes as C
import importlib.util

import pytest
import torch

from paper_2512_07503_b200 import binding as B
from paper_2512_07503_b200 import build

STAND_IN = """
#pragma once
#include <c10/core/Device.h>
namespace c10::cuda {
inline int g_current = 0;
inline DeviceIndex current_device() { return (DeviceIndex)g_current; }
inline void set_device(DeviceIndex d, const bool = false) { g_current = d; }
}
extern "C" __attribute__((used, visibility("default"))) inline int stand_in_current() { return c10::cuda::g_current; }
"""


@pytest.fixture(scope="module")
def module(tmp_path_factory):
    tmp = tmp_path_factory.mktemp("native")
    (tmp / "c10" / "cuda").mkdir(parents=True)
    (tmp / "c10" / "cuda" / "CUDAFunctions.h").write_text(STAND_IN)
    path = build.build_native_variant(str(tmp / "_native.so"), [str(tmp)])
    spec = importlib.util.spec_from_file_location("stand_in._native", path)
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod, C.CDLL(path).stand_in_current


_MEMORY = C.create_string_buffer(4096)


def _tensor(shape, dtype, device):
    n = 1
    for d in shape:
        n *= d
    where = torch.device("cuda", device)
    storage = torch._C._construct_storage_from_data_pointer(C.addressof(_MEMORY), where, n * 4)
    stride = [n := n // d for d in shape]
    return torch._C._construct_CUDA_Tensor_From_Storage_And_Metadata(
        dict(nbytes=storage.nbytes(), data_ptr=C.addressof(_MEMORY), size=tuple(shape), stride=tuple(stride), dtype=dtype, device=where, storage_offset=0),
        storage)


def _probs(device):
    f, i = torch.float32, torch.int32
    return B.DeviceProbs(_tensor((1, 2), f, device), _tensor((1, 2, 4), i, device), _tensor((1, 2, 4), f, device), _tensor((1, 2), i, device))


@pytest.mark.parametrize("device", [0, 1, 3])
def test_the_tensors_device_is_current_during_the_call(module, device):
    mod, current = module
    seen = []
    note = lambda *args: seen.append((current(), args)) or -3
    step = C.CFUNCTYPE(C.c_int, *[C.c_void_p] * 5, C.c_uint64, *[C.c_void_p] * 3)(note)
    advance = C.CFUNCTYPE(C.c_int, C.c_void_p, C.c_int32, C.c_uint64, *[C.c_void_p] * 10)(note)
    mod.set_entries(C.cast(step, C.c_void_p).value, C.cast(advance, C.c_void_p).value)
    p = B.sjd_params()
    i32 = lambda *shape: _tensor(shape, torch.int32, device)
    logits = _tensor((1, 2, 8), torch.float32, device)
    at = C.addressof(_MEMORY)
    assert mod.step(C.addressof(p), logits, None, i32(1, 2), _probs(device), 7, i32(1), i32(1, 2), _probs(device)) == -3
    assert seen[-1][0] == device and seen[-1][1][:3] == (at, None, at) and seen[-1][1][4:8] == (C.addressof(p), 7, at, at)
    assert mod.advance(C.addressof(p), 9, 5, i32(1), i32(1, 2), _probs(device), i32(1), i32(1), i32(1), i32(1, 2), _probs(device), i32(1, 9), None) == -3
    assert seen[-1][0] == device and seen[-1][1][:5] == (C.addressof(p), 9, 5, at, at) and seen[-1][1][-2:] == (at, None)
    # handed back: a check that fails once the device has been switched
    assert mod.step(C.addressof(p), logits, _tensor((1, 2, 8), torch.float64, device), i32(1, 2), _probs(device), 7, i32(1),
                    i32(1, 2), _probs(device)) == 1
    assert len(seen) == 2 and current() == 0
