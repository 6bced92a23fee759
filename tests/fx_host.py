"""The kernels' arithmetic that is host code too, compiled for the host from the
sources the kernels include (tests/fx_host.cu)."""
import ctypes
import os
import subprocess

import numpy as np

from paper_2208_14703_gb300 import build as B

_HERE = os.path.dirname(os.path.abspath(__file__))


def load(tmp):
    """The entries of fx_host.cu as a ctypes library, built in the directory `tmp`."""
    so = os.path.join(str(tmp), "libfx_host.so")
    cmd = [B.nvcc(), *B.ARCH, "-std=c++17", "-O2", "-shared", "-Xcompiler", "-fPIC,-ffp-contract=off",
           "-I", B.CSRC, "-I", B.INCLUDE, os.path.join(_HERE, "fx_host.cu"), "-o", so]
    p = subprocess.run(cmd, capture_output=True, text=True)
    assert p.returncode == 0, p.stderr
    return ctypes.CDLL(so)


def ptr(a):
    kind = {np.dtype(np.float64): ctypes.c_double, np.dtype(np.int32): ctypes.c_int,
            np.dtype(np.int64): ctypes.c_longlong}[a.dtype]
    return a.ctypes.data_as(ctypes.POINTER(kind))
