"""Builds launch_harness.cu against the library and loads it (GPU tests only)."""
import ctypes
import os
import subprocess

from paper_0811_4331_gb300 import build

_here = os.path.dirname(os.path.abspath(__file__))
_loaded = None


def load():
    global _loaded
    if _loaded is None:
        pkg = os.path.dirname(build.LIB)
        out = os.path.join(build.BUILD, "launch_harness.so")
        os.makedirs(build.BUILD, exist_ok=True)
        subprocess.run([build.nvcc()] + build.ARCH + ["-O2", "-std=c++17", "-shared", "-cudart", "shared", "-Xcompiler",
                        "-fPIC", "-I", build.CSRC, os.path.join(_here, "launch_harness.cu"), "-o", out, "-L", pkg,
                        "-lwilsonmg", "-Xlinker", "-rpath=" + pkg], check=True)
        _loaded = ctypes.CDLL(out)
        for f in ("t_mma_pack_bytes", "t_mma_scratch_bytes", "t_matvec_scratch_bytes"):
            getattr(_loaded, f).restype = ctypes.c_size_t
    return _loaded


def ptr(t):
    return ctypes.c_void_p(0 if t is None else t.data_ptr())


def ints(*v):
    return (ctypes.c_int * len(v))(*v)
