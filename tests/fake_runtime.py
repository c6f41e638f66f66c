"""The solver library's objects linked against a CUDA runtime that runs on the host (fake_cudart.cpp): the
host side of the C ABI -- argument checks, copies, launches, error paths -- without a GPU and without its
kernels, which are recorded but not run."""
import ctypes
import glob
import os
import subprocess

from paper_1905_10182_gb300 import _native as nat
from paper_1905_10182_gb300 import buildlib

HERE = os.path.dirname(os.path.abspath(__file__))


def build(folder):
    objs = [os.path.join(buildlib.BUILD, os.path.basename(s)[:-3] + ".o") for s in buildlib.sources()]
    buildlib.build(force=not all(os.path.exists(o) for o in objs))
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(buildlib.nvcc()))), "include")
    if not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        cuda = glob.glob("/usr/local/cuda/include")[0]
    out = os.path.join(str(folder), "libcmlbm_host.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-I", cuda, os.path.join(HERE, "fake_cudart.cpp"), *objs,
                    "-Wl,-Bsymbolic", "-o", out], check=True)
    L = ctypes.CDLL(out)
    P = ctypes.c_void_p
    real = nat.lib()
    for name in nat.declared_symbols():  # the same prototypes as the library itself
        fn = getattr(L, name)
        fn.argtypes, fn.restype = getattr(real, name).argtypes, getattr(real, name).restype
    L.fake_alloc.argtypes, L.fake_alloc.restype = [ctypes.c_size_t], P
    L.fake_pointer.argtypes, L.fake_pointer.restype = [ctypes.c_char_p, ctypes.c_int], P
    L.fake_launches.argtypes = L.fake_calls.argtypes = L.fake_blocks.argtypes = [ctypes.c_char_p]
    L.fake_fail.argtypes = [ctypes.c_char_p, ctypes.c_int]
    L.fake_limit.argtypes = [ctypes.c_longlong]
    L.fake_used.restype = ctypes.c_longlong
    L.cudaFree.argtypes = [P]
    return L
