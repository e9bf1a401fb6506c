"""The library's objects linked with a recording CUDA runtime (fake_cudart.cpp):
the host code of the entry points runs without a GPU, and what it launches can
be looked at."""
import ctypes as C
import os
import subprocess

import numpy as np

from paper_1209_0461_gb300 import build as B
from paper_1209_0461_gb300 import nupm

HERE = os.path.dirname(os.path.abspath(__file__))


class Fake:
    """The entry points of include/nupm.h and the controls of the fake runtime."""

    def __init__(self, out_dir):
        B.build()
        so = os.path.join(str(out_dir), "libnupm_fake.so")
        inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
        objs = [os.path.join(B.BUILD, s.replace(".cu", ".o")) for s in B.SOURCES]
        # -Bsymbolic: a real runtime that torch has loaded does not come first
        subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-Wl,-Bsymbolic", "-I", inc, "-o", so,
                        os.path.join(HERE, "fake_cudart.cpp")] + objs + ["-lpthread"], check=True)
        self.L = C.CDLL(so)
        nupm.lib()                                      # the declared signatures, from the binding
        for name in nupm.declared_symbols():
            fn, src = getattr(self.L, name), getattr(nupm.lib(), name)
            fn.restype, fn.argtypes = src.restype, src.argtypes
        self.L.fake_name.restype = C.c_char_p
        self.L.fake_bytes.restype = C.c_long

    def log(self):
        """[(kind, kernel name or memset bytes)] since the last clear; kind is
        "run", "set" (a memset) or "bad" (a refused or failed launch)."""
        L = self.L
        return [(("run", "set", "bad")[L.fake_kind(i)], L.fake_bytes(i) if L.fake_kind(i) == 1 else
                 L.fake_name(i).decode()) for i in range(L.fake_count())]

    def clear(self):
        self.L.fake_clear()

    def init(self, ngrid, npart=8, precision=nupm.PM_FP32, flags=0, n_kbins=8, m_nu=0.0, n_hist_max=4, quad=8):
        p = nupm.PmParams()
        self.L.pm_default_params(C.byref(p))
        p.ngrid, p.npart, p.precision, p.flags, p.n_kbins = ngrid, npart, precision, flags, n_kbins
        p.omega_nu, p.m_nu_total_eV, p.n_species = (-1.0, m_nu, 3) if m_nu else (0.0, 0.0, 0)
        p.n_hist_max, p.quad_nodes = n_hist_max, quad
        ic = np.ones(3 * n_kbins).ctypes.data_as(C.POINTER(C.c_double)) if m_nu else None
        ctx = C.c_void_p()
        rc = self.L.pm_init(C.byref(p), ic, ic, None, C.byref(ctx))
        assert rc == nupm.PM_OK, rc
        return ctx
