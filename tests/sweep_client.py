"""Builds and calls sweep_client.cu (the recording sweep on its own)."""
import ctypes as C
import os
import subprocess

import numpy as np

from paper_2502_14446_gb300 import build_ext

HERE = os.path.dirname(os.path.abspath(__file__))
_lib = None


def build():
    src, out = os.path.join(HERE, "sweep_client.cu"), os.path.join(build_ext.BUILD, "sweep_client.so")
    lib = build_ext.build()
    if not os.path.exists(out) or os.path.getmtime(out) < max(os.path.getmtime(src), os.path.getmtime(lib)):
        subprocess.run([build_ext.nvcc(), *build_ext.ARCH, "-std=c++17", "-O1", "-Xcompiler", "-fPIC", "-shared",
                        "-I", build_ext.CSRC, "-I", build_ext.INCLUDE, src, lib, "-Xlinker",
                        "-rpath=" + os.path.dirname(lib), "-o", out], check=True)
    return out


def load():
    global _lib
    if _lib is None:
        _lib = C.CDLL(build())
        _lib.sweep_pairs.restype = C.c_longlong
        _lib.sweep_pairs.argtypes = [C.c_void_p, C.c_int, C.c_longlong, C.c_int, C.c_int, C.c_int, C.c_int, C.c_float,
                                     C.c_float, C.c_int, C.c_void_p, C.c_void_p, C.c_longlong]
    return _lib


def sweep(T, w, d, lo, thr, excl=None, form=0, cap=1 << 22):
    """Recorded pairs (a << 32 | b, sorted) and their approximate distances."""
    lib = load()
    T = np.ascontiguousarray(T)
    pairs, dist = np.zeros(cap, np.uint64), np.zeros(cap, np.float32)
    n = lib.sweep_pairs(T.ctypes.data, 1 if T.dtype == np.float64 else 0, T.shape[1], T.shape[0], w,
                        w // 2 if excl is None else excl, d, lo, thr, form, pairs.ctypes.data, dist.ctypes.data,
                        cap)
    assert 0 <= n <= cap, n
    o = np.argsort(pairs[:n], kind="stable")
    return pairs[:n][o], dist[:n][o]
