"""handle_shim.cpp, compiled against the loaded libhgks.so."""
import ctypes as C
import os
import subprocess

from paper_2304_09485_gb300 import _native

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA_HOME = "/usr/local/cuda"


def load(directory):
    """The shim, built into `directory`; it links to the library that the binding has open."""
    _native.load()
    out = os.path.join(str(directory), "libhandle_shim.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I", os.path.join(CUDA_HOME, "include"),
                           os.path.join(HERE, "handle_shim.cpp"), "-o", out, _native.LIB, "-Wl,-rpath," + _native.BUILD,
                           "-L", os.path.join(CUDA_HOME, "lib64"), "-lcudart", "-ldl"])
    L = C.CDLL(out)
    for f in ("hx_fill_coef", "hx_fill_batch_coef"):
        getattr(L, f).argtypes = [C.c_void_p, C.c_int]
    L.hx_batch_shape.argtypes = [C.c_void_p, C.c_int, C.c_int]
    L.hx_barrier.argtypes = [C.c_void_p, C.c_uint, C.c_uint]
    L.hx_grid_cells.argtypes = [C.c_void_p, C.c_int]
    for f in ("hx_set_stuck", "hx_captured"):
        getattr(L, f).argtypes = [C.c_void_p]
    return L


def limit_recorder(directory):
    """limit_recorder.c as a library to preload."""
    out = os.path.join(str(directory), "liblimit_recorder.so")
    subprocess.check_call(["gcc", "-O1", "-fPIC", "-shared", os.path.join(HERE, "limit_recorder.c"), "-o", out, "-ldl"])
    return out
