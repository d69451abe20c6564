"""The binding's CPython shim: what it hands to a C entry point (a callback stands in for it; no device)."""
import ctypes as C

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
