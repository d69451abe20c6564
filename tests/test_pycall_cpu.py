"""The binding's CPython shim: what it hands to a C entry point (a callback stands in for it; no device)."""
import ctypes as C
import os
import sysconfig

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


def test_without_the_shim(call, monkeypatch):
    """Where the shim has not been built, load() works and the same arguments go through ctypes."""
    monkeypatch.setattr(binding, "shim_path", lambda: __file__ + ".none")
    monkeypatch.setattr(binding, "_LIB", None)
    monkeypatch.setattr(binding, "_CALL", binding._CALL)
    binding.load()
    assert binding._CALL is None
    seen = []
    linear = C.CFUNCTYPE(C.c_int, P, P, P, I64, I64, P, I32, I64, P, SZ, P)(lambda *a: seen.append(a) or 0)
    quantise = C.CFUNCTYPE(C.c_int, P, P, I64, I64, I64, P, P, I32, P)(lambda *a: seen.append(a) or 5)

    class Fake:
        batq_linear_w4a8, batq_quantize_act = linear, quantise

    monkeypatch.setattr(binding, "_LIB", Fake)
    monkeypatch.setattr(binding, "_stream", lambda: 7)
    x = torch.empty((9, 96), dtype=torch.bfloat16)[1:4, :64]
    y, ws = torch.empty((3, 40)), torch.empty(2048, dtype=torch.uint8)

    class Handle:
        handle = P(1 << 40)

    binding.batq_linear_w4a8(None, Handle(), x, y, ws)
    with pytest.raises(binding.BatqError):
        binding.batq_quantize_act(Handle(), x, ws, np.int64(512), binding.SF_MMA)
    assert seen == [(None, 1 << 40, x.data_ptr(), 3, 96, y.data_ptr(), binding.F32, 40, ws.data_ptr(), 2048, 7),
                    (1 << 40, x.data_ptr(), 3, 64, 96, ws.data_ptr(), 512, 1, 7)]


def test_shim_is_built_for_each_interpreter():
    assert binding.shim_path() == build.CALL_LIB and sysconfig.get_config_var("EXT_SUFFIX") in build.CALL_LIB


def test_build_without_python_headers(tmp_path, monkeypatch, capsys):
    """No shim, a line on stderr, and the library as it was."""
    monkeypatch.setattr(build, "CALL_LIB", str(tmp_path / "_pycall.so"))
    monkeypatch.setenv("CC", str(tmp_path / "no-compiler"))
    assert os.path.exists(build.build())
    assert "ctypes" in capsys.readouterr().err and not os.path.exists(build.CALL_LIB)
