"""The library's host side on the CPU: its objects linked with a CUDA runtime that counts launches
instead of running them and fails the calls a test names (fake_cudart.cpp)."""
import ctypes
import glob
import os
import subprocess

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))


def load(tmp):
    import __graft_entry__ as g
    g.build()
    from paper_2502_17683_gb300 import _lib, build
    objs = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in glob.glob(os.path.join(build.CSRC, "*.cu"))]
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    out = os.path.join(str(tmp), "libthc_cpd_fake.so")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-Wl,--no-undefined",
                        "-I", inc, "-I", build.CSRC, os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", out, "-lpthread", "-ldl"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(out)
    for name, args in _lib._SIGS.items():
        fn = getattr(lib, name)
        fn.argtypes, fn.restype = args, ctypes.c_int
    lib.thc_cpd_last_error.restype = ctypes.c_char_p
    lib.fake_fail_launch.argtypes = [ctypes.c_char_p, ctypes.c_long]
    lib.fake_launches.argtypes, lib.fake_launches.restype = [ctypes.c_char_p], ctypes.c_long
    lib.fake_alloc_limit.argtypes = [ctypes.c_size_t]
    lib.fake_outside.restype = ctypes.c_long
    lib.fake_launched.restype = ctypes.c_char_p
    lib.fake_largest_alloc.restype = ctypes.c_size_t
    return lib


class Calls:
    """Entry points with buffers of the right sizes (host memory: no kernel runs)."""

    def __init__(self, lib):
        self.lib = lib

    def _p(self, *shape):
        a = np.zeros(shape)
        self.keep.append(a)
        return a.ctypes.data

    def _problem(self, o, v, Rt, R):
        from paper_2502_17683_gb300._lib import PTR4
        self.keep = []
        return [o, v, Rt, R, self._p(o, Rt), self._p(v, Rt), self._p(Rt, Rt),
                PTR4(*[self._p(n, R) for n in (o, v, o, v)])]

    def _opts(self, precision=0, ldl=0, products=0):
        from paper_2502_17683_gb300._lib import Opts
        o = Opts()
        o.precision, o.ldl, o.products = precision, ldl, products
        return ctypes.byref(o)

    def launched(self):
        names, i = [], 0
        while (n := self.lib.fake_launched(i)) is not None:
            names.append(n)
            i += 1
        return names

    def mttkrp(self, o, v, Rt, R, mode=0, **kw):
        return self.lib.thc_cpd_mttkrp(*self._problem(o, v, Rt, R), mode, self._p(max(o, v), R), self._opts(**kw))

    def norm2(self, o, v, Rt, **kw):
        a = self._problem(o, v, Rt, 1)
        return self.lib.thc_cpd_thc_norm2(*a[:3], *a[4:7], ctypes.byref(ctypes.c_double()), self._opts(**kw))

    def loss(self, o, v, Rt, R, normG2=1.0, **kw):
        d = ctypes.c_double()
        return self.lib.thc_cpd_loss(*self._problem(o, v, Rt, R), None, normG2, ctypes.byref(d), ctypes.byref(d),
                                     self._opts(**kw))

    def sweep(self, o, v, Rt, R, normG2=1.0, **kw):
        d = ctypes.c_double()
        return self.lib.thc_cpd_als_sweep(*self._problem(o, v, Rt, R), self._p(R), normG2, ctypes.byref(d),
                                          ctypes.byref(d), self._opts(**kw))

    def trajectory(self, o, v, Rt, R, sweeps=2, **kw):
        a, al, tl = self._problem(o, v, Rt, R), (ctypes.c_double * 2)(1.0, 1.5), (ctypes.c_double * (2 * sweeps))()
        return self.lib.thc_cpd_als_trajectory(*a, self._p(R), sweeps, al, 2, (ctypes.c_float * (40 * sweeps))(), tl,
                                               self._opts(**kw))

    def batched(self, shapes, sweeps=2, **kw):
        from paper_2502_17683_gb300._lib import Problem
        probs, keep = (Problem * len(shapes))(), []
        for q, (o, v, Rt, R) in zip(probs, shapes):
            a = self._problem(o, v, Rt, R)
            q.o, q.v, q.Rt, q.R, q.Xo, q.Xv, q.Z = a[:7]
            for k in range(4):
                q.A[k] = a[7][k]
            q.lam = self._p(R)
            keep += self.keep
        self.keep = keep
        return self.lib.thc_cpd_als_batched(len(shapes), ctypes.byref(probs), sweeps, 0.0, self._opts(**kw))

    def exchange(self, o, v, Rt, R, nalpha, **kw):
        a, d = self._problem(o, v, Rt, R), ctypes.c_double()
        return self.lib.thc_cpd_exchange(*a[:4], nalpha, *a[4:], self._p(R), self._p(nalpha, o), self._p(nalpha, v),
                                         ctypes.byref(d), ctypes.byref(d), ctypes.byref(d), self._opts(**kw))

    def core_fit(self, o, v, Rt, naux, loss=False, **kw):
        self.keep = []
        d = ctypes.c_double()
        return self.lib.thc_cpd_core_fit(o, v, Rt, naux, self._p(o, Rt), self._p(v, Rt), self._p(naux, o, v),
                                         self._p(Rt, Rt), ctypes.byref(d) if loss else None,
                                         ctypes.byref(ctypes.c_int()), self._opts(**kw))

    def df_als(self, o, v, naux, R, sweeps=1, **kw):
        from paper_2502_17683_gb300._lib import PTR4
        self.keep = []
        A = PTR4(*[self._p(n, R) for n in (o, v, o, v)])
        return self.lib.thc_cpd_df_als(o, v, naux, R, self._p(naux, o, v), A, self._p(R), sweeps, 0.0,
                                       ctypes.byref(ctypes.c_int()), ctypes.byref(ctypes.c_double()), self._opts(**kw))

    def nd_mttkrp(self, dims, dL, Rt, R, mode=0, **kw):
        self.keep = []
        d = len(dims)
        X = (ctypes.c_void_p * d)(*[self._p(n, Rt) for n in dims])
        A = (ctypes.c_void_p * d)(*[self._p(n, R) for n in dims])
        return self.lib.thc_cpd_nd_mttkrp(d, dL, (ctypes.c_int * d)(*dims), Rt, R, X, self._p(Rt, Rt), A, mode,
                                          self._p(dims[mode], R), self._opts(**kw))

    def nd_als(self, dims, dL, Rt, R, sweeps=1, **kw):
        self.keep = []
        d = len(dims)
        X = (ctypes.c_void_p * d)(*[self._p(n, Rt) for n in dims])
        A = (ctypes.c_void_p * d)(*[self._p(n, R) for n in dims])
        return self.lib.thc_cpd_nd_als(d, dL, (ctypes.c_int * d)(*dims), Rt, R, X, self._p(Rt, Rt), A, self._p(R),
                                       sweeps, 0.0, ctypes.byref(ctypes.c_int()), ctypes.byref(ctypes.c_double()),
                                       self._opts(**kw))

    def solve(self, R, n, **kw):
        self.keep = []
        return self.lib.thc_cpd_ldl_solve(R, n, self._p(R, R), self._p(n, R), self._p(n, R), None, 0,
                                          ctypes.byref(ctypes.c_int()), self._opts(**kw))
