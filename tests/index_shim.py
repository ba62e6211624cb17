"""The kernels' own index arithmetic (csrc/internal.h), compiled for the host from index_shim.cu."""
import ctypes
import functools
import os
import subprocess
import tempfile

import numpy as np

from paper_2608_14787_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@functools.lru_cache(maxsize=None)
def lib():
    with tempfile.TemporaryDirectory() as d:
        so = os.path.join(d, "shim.so")
        subprocess.check_call([build._nvcc(), *build.ARCH, "-std=c++17", "-O2", "-shared", "-Xcompiler", "-fPIC", "-I",
                               build.INCLUDE, "-o", so, os.path.join(HERE, "index_shim.cu")])
        L = ctypes.CDLL(so)
    i64 = ctypes.c_int64
    for name, args in {"cut": None, "whole_pieces": [i64] * 4, "share_start": [i64], "share_warp": [i64],
                       "slice_start": [i64, ctypes.c_int]}.items():
        f = getattr(L, "shim_" + name)
        f.restype = i64
        if args:
            f.argtypes = args
    L.shim_slice_owner.argtypes = [i64, i64]
    L.shim_slice_half.argtypes = [i64, ctypes.c_int]
    L.shim_slice_slots.argtypes = [i64, ctypes.c_int]
    return L


def cut(kind, nb, npos0, npos1, RV, ctas=152, owners=()):
    """(start [W + 1], row, vec, the owners of the given vectors, {"whole", "units", "C"})."""
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)   # noqa: E731
    i64 = ctypes.c_int64
    cap = ctas * 16 + 1
    start, row, vec = np.empty(cap, np.int64), np.empty(cap, np.int64), np.empty(cap, np.int32)
    v = np.asarray(owners, np.int64)
    own, facts = np.empty(len(v), np.int64), np.empty(3, np.int64)
    W = lib().shim_cut(kind, nb, npos0, npos1, RV, ctas, i64(cap), p(start), p(row), p(vec), i64(len(v)), p(v), p(own),
                       p(facts))
    assert W > 0
    return start[:W + 1], row[:W + 1], vec[:W + 1], own, dict(zip(("whole", "units", "C"), facts.tolist()))
