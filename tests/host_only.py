"""The library's host code on the CPU: its objects linked with ``fake_cudart.cpp``, a stand-in CUDA
runtime whose device memory is host memory and whose kernels only report their launches."""

import ctypes
import os
import subprocess

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
HOOK = ctypes.CFUNCTYPE(None, ctypes.c_char_p, ctypes.POINTER(ctypes.c_uint),
                        ctypes.POINTER(ctypes.c_void_p))


def link():
    """The stand-in library (objects and library are built first where they are not up to date)."""
    from paper_2105_01196_gb300 import build
    objs = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    srcs = [os.path.join(build.CSRC, f) for f in os.listdir(build.CSRC)]
    newest = max(os.path.getmtime(s) for s in srcs)
    if not all(os.path.exists(o) and os.path.getmtime(o) >= newest for o in objs):
        build.build()
    out = os.path.join(build.BUILD, "host_only.so")
    src = os.path.join(HERE, "fake_cudart.cpp")
    if not os.path.exists(out) or os.path.getmtime(out) < max(map(os.path.getmtime, objs + [src])):
        cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
        subprocess.run(["g++", "-shared", "-fPIC", "-std=c++17", "-O1", "-pthread",
                        "-Wl,-Bsymbolic", "-I", cuda, src, *objs, "-o", out], check=True)
    return out


class Library:
    """Entry points by name, with the header's argument types; launches as (kernel, grid) pairs."""

    def __init__(self):
        from paper_2105_01196_gb300 import ebic
        self.ebic = ebic
        self.raw = ctypes.CDLL(link())
        for name, (res, args) in ebic.SIGNATURES.items():
            getattr(self.raw, name).restype, getattr(self.raw, name).argtypes = res, args
        for name in ("fake_allocs", "fake_device_blocks", "fake_device_bytes", "fake_pinned_blocks", "fake_log_size",
                     "fake_calls"):
            getattr(self.raw, name).restype = ctypes.c_int64
        self.raw.fake_log_kernel.restype = ctypes.c_char_p
        self.raw.fake_log_kernel.argtypes = self.raw.fake_log_grid.argtypes = [ctypes.c_int64]
        for name in ("fake_fail_alloc", "fake_fail_copy", "fake_set_free"):
            getattr(self.raw, name).argtypes = [ctypes.c_int64]
        self.raw.fake_elapsed.argtypes = [ctypes.c_float, ctypes.c_float]
        self.raw.cudaMalloc.argtypes = [ctypes.c_void_p, ctypes.c_size_t]
        self._hook = None

    def __getattr__(self, name):
        return getattr(self.raw, name)

    def hook(self, fn):
        """fn(kernel, grid, args) at every launch (args: the addresses of the arguments)."""
        self._hook = HOOK(lambda k, g, a: fn(k.decode(), g[0], a)) if fn else None
        self.raw.fake_hook(self._hook)

    def log(self):
        return [(self.raw.fake_log_kernel(i).decode(), self.raw.fake_log_grid(i))
                for i in range(self.raw.fake_log_size())]

    def context(self):
        out = ctypes.c_void_p()
        assert self.raw.ebic_create(ctypes.byref(out), 0, None) == 0
        return out.value

    def load(self, ctx, rows, cols):
        x = np.zeros((rows, cols), np.float32)
        return self.raw.ebic_load_matrix(ctx, x.ctypes.data, rows, cols, 0)

    def device(self, n):
        """n bytes of device memory (leaked: a test needs few)."""
        p = ctypes.c_void_p()
        assert self.raw.cudaMalloc(ctypes.byref(p), n) == 0
        return p.value

    def run(self, ctx, p, n_gen):
        rep = self.ebic.RunReport()
        return self.raw.ebic_run_generations(ctx, ctypes.byref(p), n_gen, ctypes.byref(rep)), rep
