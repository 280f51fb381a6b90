"""The library's own objects linked against a CUDA runtime that runs on the
host (host_cuda.cpp): what its host code launches, refuses and reports can be
tested without a GPU, with launches that fail on request."""
import ctypes as C
import glob
import os
import subprocess

import pytest

from paper_2504_02627_gb300 import _binding as B
from paper_2504_02627_gb300 import build as build_mod

HERE = os.path.dirname(os.path.abspath(__file__))
NOMEM = 2                        # cudaErrorMemoryAllocation
E_NOMEM, E_STATE = -2, -6        # SMC_E_*


def _objects():
    return sorted(glob.glob(os.path.join(build_mod.BUILD, "*.o")))


def load(folder):
    """Builds and loads the library in `folder`, as its own copy."""
    if not os.path.exists(build_mod.NVCC):
        pytest.skip("no nvcc")
    build_mod.build()
    want = {os.path.basename(s)[:-3] + ".o" for s in build_mod._sources()}
    if {os.path.basename(o) for o in _objects()} != want:
        build_mod.build(force=True)
    objects = [o for o in _objects() if os.path.basename(o) in want]
    so = os.path.join(str(folder), "libhostcuda.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(build_mod.NVCC)), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-I" + inc, "-o", so,
                    os.path.join(HERE, "host_cuda.cpp")] + objects, check=True)
    lib = C.CDLL(so)
    for name, (res, args) in B.EXPORTS.items():
        f = getattr(lib, name)
        f.restype, f.argtypes = res, args
    lib.host_cuda_launched.restype = C.c_char_p
    lib.host_cuda_allocated.restype = C.c_longlong
    lib.host_cuda_fail.argtypes = [C.c_char_p, C.c_int, C.c_int]
    return lib


def launches(lib):
    """Kernels launched since the last call, by their mangled names."""
    out = lib.host_cuda_launched().decode().split()
    lib.host_cuda_clear()
    return out
