"""The library's host code on a machine without a GPU: its objects linked with the stand-in runtime of
host_runtime.cpp (device memory is host memory, kernels are recorded and not run)."""
import ctypes
import glob
import os
import subprocess

import numpy as np

from paper_2305_11566_gb300 import binding, build

HERE = os.path.dirname(os.path.abspath(__file__))


def load(folder):
    build.build()
    objs = sorted(glob.glob(os.path.join(build.BUILD, "*.o")))
    if len(objs) < len(build.units()):
        build.build(force=True)
    objs = [os.path.join(build.BUILD, o) for _, _, o in build.units()]
    cuda = os.path.dirname(os.path.dirname(build._nvcc()))
    out = os.path.join(str(folder), "libhost.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"), "-o",
                           out, os.path.join(HERE, "host_runtime.cpp"), *objs, "-Wl,-Bsymbolic", "-Wl,-z,defs"])
    L = ctypes.CDLL(out)
    for name, (args, res) in binding.API.items():
        getattr(L, name).argtypes, getattr(L, name).restype = args, res
    for name in ("host_used", "host_peak"):
        getattr(L, name).restype = ctypes.c_size_t
    L.host_limit.argtypes = [ctypes.c_size_t]
    L.host_fail_in.argtypes = L.host_launch_fail_in.argtypes = [ctypes.c_longlong]
    L.host_launch_name.restype = ctypes.c_char_p
    L.host_launch_grid.argtypes = [ctypes.c_int, ctypes.POINTER(ctypes.c_uint)]
    return L


class Host:
    """A context of the host library and buffers for n pairs of the sizes given."""

    def __init__(self, L, shape, precision, sizes, window=3, D=4):
        self.L, self.n = L, len(sizes)
        L.host_limit(256 << 30)
        L.host_fail_in(0)
        L.host_launch_fail_in(0)
        L.host_capture(0)
        cfg = binding.make_config(shape, window, precision)
        self.params = int(L.sv_param_count(ctypes.byref(cfg)))
        self.ctx = ctypes.c_void_p()
        assert L.sv_create(ctypes.byref(cfg), 0, ctypes.byref(self.ctx)) == binding.SV_OK
        self.keep = []
        side = max(max(w, h) for w, h in sizes)
        pitch = (side + 15) // 16 * 16
        image = self.buffer(pitch * side + 16)
        image += -image % 16
        self.pairs = (binding.SvPair * self.n)(*[binding.SvPair(image, image, w, h, pitch, D) for w, h in sizes])
        # (kernels do not run: every pair may share one buffer)
        self.any = self.ptrs([self.buffer(4096)] * self.n)

    def buffer(self, nbytes):
        a = np.zeros(nbytes, np.uint8)
        self.keep.append(a)
        return a.ctypes.data

    @staticmethod
    def ptrs(items):
        return (ctypes.c_void_p * len(items))(*items)

    def close(self):
        self.L.sv_destroy(self.ctx)

    def error(self):
        return self.L.sv_last_error(self.ctx).decode()

    def refine(self):
        return self.L.sv_refine(self.ctx, self.pairs, self.any, self.n, self.any, None)

    def train(self):
        return self.L.sv_refine_train(self.ctx, self.pairs, self.any, self.any, self.n, self.any, self.any, self.any,
                                      None)

    def backward(self):
        g = self.buffer(8 * self.params)
        return self.L.sv_refine_backward(self.ctx, self.any, self.any, self.any, ctypes.c_void_p(g), None, None)

    def loss(self):
        return self.L.sv_loss(self.ctx, self.pairs, self.n, self.any, self.any, self.any, self.any, 1e-3,
                              ctypes.c_void_p(self.buffer(32)), self.any, self.any, self.any, None)

    def launches(self):
        g = (ctypes.c_uint * 3)()
        out = []
        for i in range(self.L.host_launches()):
            self.L.host_launch_grid(i, g)
            out.append((self.L.host_launch_name(i).decode(), tuple(g)))
        return out
