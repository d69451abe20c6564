"""The binding's CPython shim: what it hands to a C entry point (a callback stands in for it; no device)."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2603_16590_b200 import binding, build

P, I64, I32, SZ = C.c_void_p, C.c_int64, C.c_int32, C.c_size_t


@pytest.fixture(scope="module")
def call():
    build.build()
    binding.load()
    return binding._CALL


@pytest.mark.parametrize("dtype,code", [(torch.float32, binding.F32), (torch.bfloat16, binding.BF16)])
def test_linear_arguments(call, dtype, code):
    seen = []
    fn = C.CFUNCTYPE(C.c_int, P, P, P, I64, I64, P, I32, I64, P, SZ, P)(lambda *a: seen.append(a) or 5)
    x = torch.empty((9, 96), dtype=torch.bfloat16)[1:4, :64]      # a row stride and a pointer of its own
    y = torch.empty((3, 40), dtype=dtype)
    ws = torch.empty(2048, dtype=torch.uint8)
    big = 1 << 47
    assert call.linear(C.cast(fn, P).value, 0, big, x, y, ws, 7) == 5
    assert seen == [(None, big, x.data_ptr(), 3, 96, y.data_ptr(), code, 40, ws.data_ptr(), 2048, 7)]


def test_quantise_arguments_and_errors(call):
    seen = []
    fn = C.CFUNCTYPE(C.c_int, P, P, I64, I64, I64, P, P, I32, P)(lambda *a: seen.append(a) or 0)
    x = torch.empty((4, 64), dtype=torch.bfloat16)
    codes, addr = torch.empty(128, dtype=torch.uint8), C.cast(fn, P).value
    assert call.quantise(addr, 3, x, codes, None, binding.SF_MMA, 0) == 0
    assert seen == [(3, x.data_ptr(), 4, 64, 64, codes.data_ptr(), None, 1, None)]
    with pytest.raises(AttributeError):
        call.quantise(addr, 3, "not a tensor", codes, codes, 1, 0)
    with pytest.raises(TypeError):
        call.quantise(addr, 3, x, codes, codes, "layout", 0)
    with pytest.raises(TypeError):
        call.linear(addr, 0, 0)
    assert len(seen) == 1


def test_addresses_of_any_integer_type(call, monkeypatch):
    """An address is what int() takes (a numpy integer, as numpy's own pointers come), through the shim as through
    ctypes; x may be anything with shape, stride() and an address; a layout is a Python int."""
    seen = []
    fn = C.CFUNCTYPE(C.c_int, P, P, I64, I64, I64, P, P, I32, P)(lambda *a: seen.append(a) or 0)
    monkeypatch.setattr(binding, "_ADDRESS", {"batq_quantize_act": C.cast(fn, P).value})
    monkeypatch.setattr(binding, "_stream", lambda: 7)
    x = torch.empty((4, 64), dtype=torch.bfloat16)

    class Rows:
        shape = (4, 64)
        stride = staticmethod(lambda d: 96)
        __int__ = lambda self: 4096

    top = np.uint64((1 << 64) - 256)
    binding.batq_quantize_act(None, x, np.int64(1 << 40), top, binding.SF_MMA)
    binding.batq_quantize_act(None, Rows(), 512, -256, binding.SF_ROWMAJOR)
    assert seen == [(None, x.data_ptr(), 4, 64, 64, 1 << 40, int(top), 1, 7), (None, 4096, 4, 64, 96, 512, int(top), 0, 7)]
    with pytest.raises(TypeError):
        binding.batq_quantize_act(None, x, 256, 256, np.int32(1))
    with pytest.raises(TypeError):
        binding.batq_quantize_act(None, x, object(), 256, binding.SF_MMA)
    assert len(seen) == 2
