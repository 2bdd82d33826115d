"""Access to a handle's fields beyond the C ABI (peek.cu, compiled on first use)."""
import ctypes
import functools
import os
import subprocess
import tempfile

import numpy as np

from paper_1601_05527_gb300 import build


@functools.lru_cache(None)
def load():
    out = os.path.join(tempfile.mkdtemp(), "peek.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "peek.cu")
    r = subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, "-shared", src, "-o", out],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(out)


def degrees(h, n):
    """(weighted degrees, whether each sum is exact in any order) of a weighted handle."""
    D, exact = np.zeros(n, np.float64), np.zeros(n, np.uint8)
    assert load().peek_degrees(h, ctypes.c_void_p(D.ctypes.data), ctypes.c_void_p(exact.ctypes.data)) == 0
    return D, exact


def set_shape(h, R, storage, lanes, chunks):
    load().peek_set_shape(h, int(R), int(storage), int(lanes), int(chunks))
