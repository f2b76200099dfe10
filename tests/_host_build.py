"""Compiles device headers for the host (tests/_host_kernels.cpp) and loads
them, for tests of kernel arithmetic that need no GPU."""
import ctypes
import os
import subprocess

import numpy as np

from paper_2207_05258_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


_loaded = []


def load(directory):
    """The library, compiled into `directory` by the first call of the session."""
    if _loaded:
        return _loaded[0]
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc())))
    lib = os.path.join(str(directory), "libhost_kernels.so")
    cmd = ["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-w",
           "-I", HERE, "-I", build.CSRC, "-I", build.INCLUDE, "-I", os.path.join(cuda, "include"),
           os.path.join(HERE, "_host_kernels.cpp"), "-o", lib]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    _loaded.append(ctypes.CDLL(lib))
    return _loaded[0]


def ptr(a):
    """Pointer to a contiguous numpy array's data."""
    assert a.flags.c_contiguous
    t = {np.dtype("f8"): ctypes.c_double, np.dtype("f4"): ctypes.c_float,
         np.dtype("i4"): ctypes.c_int}[a.dtype]
    return a.ctypes.data_as(ctypes.POINTER(t))
