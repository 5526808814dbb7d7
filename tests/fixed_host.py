"""Builds tests/fixed_host.cu for the CPU and calls it."""
import ctypes as C
import functools
import os
import subprocess
import tempfile

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))


@functools.lru_cache(None)
def lib():
    from paper_2012_08221_gb300 import build
    out = os.path.join(tempfile.mkdtemp(prefix="fixed_host"), "libfixed_host.so")
    r = subprocess.run([build.nvcc(), "-shared", "-o", out, os.path.join(HERE, "fixed_host.cu"), "-O2", "-std=c++17",
                        "-Xcompiler", "-fPIC,-ffp-contract=off", "-I", build.INCLUDE, "-I", build.CSRC] + build.ARCH,
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return C.CDLL(out)


def _p(a):
    return a.ctypes.data_as(C.c_void_p)


def cells(lower, last, keys):
    """Cells of the keys (IEEE bits), and the size of the guide table used."""
    lower = np.ascontiguousarray(lower, dtype=np.float64).view(np.uint64)
    keys = np.ascontiguousarray(keys, dtype=np.uint64)
    out, guided = np.empty(keys.size, np.int32), C.c_int()
    lib().host_cells(_p(lower), lower.size, C.c_uint64(int(np.float64(last).view(np.uint64))), _p(keys), keys.size,
                     _p(out), C.byref(guided))
    return out, guided.value
