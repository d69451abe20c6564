"""Builds the C-ABI shared library in-tree with nvcc for sm_100a."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
LIB = os.path.join(HERE, "libbatq.so")
# CPython shim of the binding's calls, one for each interpreter that has used this tree
CALL_LIB = os.path.join(HERE, "_pycall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
CALL_SOURCE = os.path.join(HERE, "csrc", "pycall.c")
SOURCES = [os.path.join(HERE, "csrc", "batq.cu")]
DEPS = [os.path.join(HERE, "csrc", f) for f in os.listdir(os.path.join(HERE, "csrc"))] + [
    os.path.join(ROOT, "include", "batq.h")]


def nvcc_command(extra=()):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    return [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
            "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"),
            "-I", os.path.join(HERE, "csrc"), *extra, "-o", LIB, *SOURCES]


def _build_call_shim(force: bool):
    """Without the Python headers or a C compiler there is no shim: the binding then makes its calls through ctypes."""
    if not force and os.path.exists(CALL_LIB) and os.path.getmtime(CALL_SOURCE) <= os.path.getmtime(CALL_LIB):
        return
    cmd = [os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], "-o", CALL_LIB, CALL_SOURCE]
    try:
        subprocess.run(cmd, capture_output=True, text=True, check=True)
    except (OSError, subprocess.CalledProcessError) as e:
        if os.path.exists(CALL_LIB):
            os.remove(CALL_LIB)   # of an older source
        sys.stderr.write(f"{getattr(e, 'stderr', None) or e}\n{CALL_LIB} not built: calls go through ctypes, some 2 us slower\n")


def build(force: bool = False, verbose: bool = False) -> str:
    """Compiles libbatq.so (and the binding's shim) if missing or older than their sources; returns libbatq.so's path."""
    _build_call_shim(force)
    if not force and os.path.exists(LIB):
        t = os.path.getmtime(LIB)
        if all(os.path.getmtime(d) <= t for d in DEPS):
            return LIB
    cmd = nvcc_command(("-Xptxas", "-v") if verbose else ())
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed building libbatq.so")
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
