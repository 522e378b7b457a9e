"""The library's host code over a stand-in CUDA runtime (native/fake_cudart.cpp): which kernels a
call launches, on which device, and what it allocates, without a GPU."""
import ctypes
import glob
import os
import subprocess

import paper_2607_01735_gb300 as rb
from paper_2607_01735_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "native", "fake_cudart.cpp")
OUT = os.path.join(HERE, "native", "_build", "libfakerbgs.so")


def load():
    """The library's object files linked with the stand-in; a fresh state of it."""
    build.build_library()
    objs = sorted(glob.glob(os.path.join(build.BUILD, "*.o")))
    cuda = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    os.makedirs(os.path.dirname(OUT), exist_ok=True)
    if not os.path.exists(OUT) or os.path.getmtime(OUT) < max(os.path.getmtime(p) for p in objs + [SRC]):
        tmp = OUT + f".tmp{os.getpid()}"
        # -Bsymbolic: the stand-in's functions and not those of a runtime that torch has loaded
        subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-Wl,--no-undefined",
                               "-I", cuda, SRC, "-o", tmp] + objs + ["-lpthread"])
        os.replace(tmp, OUT)
    lib = ctypes.CDLL(OUT)
    vp, ci, cl, cd = ctypes.c_void_p, ctypes.c_int, ctypes.c_long, ctypes.c_double
    lib.fake_log.restype = ctypes.c_char_p
    lib.fake_memory_limit.argtypes = [ctypes.c_size_t]
    lib.fake_memory_in_use.restype = ctypes.c_size_t
    lib.rbgs_default_opts.argtypes = [ctypes.POINTER(rb.Opts)]
    lib.rbgs_default_opts.restype = None
    lib.rbgs_create.argtypes = [ci, cd, vp, vp, ctypes.POINTER(rb.Opts), vp, ctypes.POINTER(vp)]
    lib.rbgs_sweep.argtypes = [vp, cl]
    lib.rbgs_solve.argtypes = [vp, cd, ctypes.POINTER(cl), ctypes.POINTER(cd)]
    lib.rbgs_residual.argtypes = [vp, ctypes.POINTER(cd)]
    lib.rbgs_destroy.argtypes = [vp]
    lib.rbgs_destroy.restype = None
    lib.rbgs_last_error.restype = ctypes.c_char_p
    lib.fake_reset()
    return lib


class Context:
    """An n^2 problem's context on the current stand-in device; `stream` is a handle."""

    def __init__(self, lib, n, stream=None, **opts):
        import numpy as np
        self.lib = lib
        o = rb.Opts()
        lib.rbgs_default_opts(ctypes.byref(o))
        for k, v in opts.items():
            setattr(o, k, v)
        f, u = np.zeros((n, n)), np.zeros((n + 2, n + 2))
        self.ctx = ctypes.c_void_p()
        st = lib.rbgs_create(n, 1.0, f.ctypes.data, u.ctypes.data, ctypes.byref(o), stream, ctypes.byref(self.ctx))
        assert st == 0, lib.rbgs_last_error()

    def sweep(self, k):
        """Status and the launches of a sweep call: [(kind, kernel, blocks, device)]."""
        self.lib.fake_clear_log()
        return self.lib.rbgs_sweep(self.ctx, k), launches(self.lib)

    def close(self):
        self.lib.rbgs_destroy(self.ctx)


def launches(lib):
    rows = [l.split() for l in lib.fake_log().decode().splitlines()]
    return [(r[0], r[1], int(r[2]), int(r[3])) for r in rows]
