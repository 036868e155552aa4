"""Builds tests/device_functions.cu (wrappers of the library's device functions, against its headers and with its compiler
flags) into a temporary folder and loads it."""
import ctypes as C
import os
import subprocess

import pytest


def load(tmp):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_04953_gb300 import build
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "device_functions.cu")
    so = os.path.join(str(tmp), "device_functions.so")
    r = subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", src, "-o", so],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = C.CDLL(so)
    vp, i, d, n = C.c_void_p, C.c_int, C.c_double, C.c_long
    lib.dev_pow.argtypes = [n, vp, vp, vp, vp, vp]
    lib.dev_tangent.argtypes = [n, vp, d, d, d, d, d, d, d, i, vp, vp, vp]
    return torch, lib
