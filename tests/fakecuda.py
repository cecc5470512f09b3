"""The library's objects linked against a CUDA runtime without a GPU
(fake_cudart.c): host-side tests see which kernels are launched, over which
grids, and what happens when an allocation fails."""
import ctypes
import glob
import os
import subprocess

import numpy as np

import paper_2510_23739_gb300 as sw
from paper_2510_23739_gb300 import build as swbuild

HERE = os.path.dirname(os.path.abspath(__file__))


def load(folder):
    """The library over the fake runtime, built in `folder`."""
    swbuild.build()
    include = os.path.join(os.path.dirname(os.path.dirname(swbuild._nvcc())), "include")
    out = os.path.join(str(folder), "libswopt_fake.so")
    objs = sorted(glob.glob(os.path.join(swbuild.BUILD, "*.o")))
    subprocess.run(["gcc", "-O1", "-fPIC", "-shared", "-I", include,
                    os.path.join(HERE, "fake_cudart.c"), *objs, "-o", out, "-lstdc++", "-lm",
                    "-Wl,-Bsymbolic"], check=True)
    L = ctypes.CDLL(out)
    for name, (args, res) in sw._SIGS.items():
        fn = getattr(L, name)
        fn.argtypes, fn.restype = args, res
    L.fake_largest.restype = ctypes.c_size_t
    L.fake_limit.argtypes = [ctypes.c_size_t]
    L.fake_fail_in.argtypes = [ctypes.c_long]
    L.fake_failed.restype = L.fake_live.restype = L.fake_launches.restype = ctypes.c_long
    L.fake_launches.argtypes = L.fake_grid.argtypes = [ctypes.c_char_p]
    L.fake_grid.restype = ctypes.c_uint
    return L


class Handle:
    """A handle of the fake library and the buffers of its calls."""

    def __init__(self, L, X=16, Y=14, Z=12, T=40, N=4, P=2, k=3, cycle=4):
        self.L = L
        rng = np.random.default_rng(0)
        self.K = rng.standard_normal((Z, k, k, T))
        vals = [np.linspace(0.1, 0.2, P), np.ones(P), np.full(P, 0.5)]
        self.keep = vals
        dp = ctypes.POINTER(ctypes.c_double)
        s = sw._Switching(*(v.ctypes.data_as(dp) for v in vals), 1.5)
        g = sw._Geometry(X, Y, Z, T, N, P, k, cycle, 0.01)
        self.h = ctypes.c_void_p()
        st = L.swopt_create(ctypes.byref(g), self.K.ctypes.data, ctypes.byref(s),
                            ctypes.byref(self.h))
        assert st == 0, L.swopt_last_error()
        self.c = np.zeros(P * Y * X * Z, np.float32)
        self.x = np.zeros(P * Y * X * Z, np.float32)
        self.y = np.zeros(N * Y * X * T, np.float32)

    def forward(self):
        return self.L.swopt_forward(self.h, self.c.ctypes.data, self.y.ctypes.data, None)

    def prox_tv(self, iters=4):
        return self.L.swopt_prox_tv(self.h, self.c.ctypes.data, self.x.ctypes.data, 0.1, iters, 0,
                                    None)

    def precision(self, name):
        return self.L.swopt_set_precision(self.h, sw.PRECISION[name])

    def pin(self):
        """Ask for the tensor-core kernels, by a pinned schedule."""
        for kernel in (0, 1):
            assert self.L.swopt_tc_schedule(self.h, kernel, 1, 0) == 0

    def adjoint(self):
        return self.L.swopt_adjoint(self.h, self.y.ctypes.data, self.x.ctypes.data, None)

    def fista_init(self, **kw):
        prm = sw.SolveParams(**kw)._c()
        return self.L.swopt_fista_init(self.h, self.y.ctypes.data, ctypes.byref(prm), None)

    def objective(self):
        F, fit = ctypes.c_double(), ctypes.c_double()
        return self.L.swopt_objective(self.h, self.c.ctypes.data, self.y.ctypes.data, 0.1, 0.1, 0.0,
                                      ctypes.byref(F), ctypes.byref(fit), None)

    def close(self):
        self.L.swopt_destroy(self.h)
