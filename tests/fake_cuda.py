"""The library linked against the CUDA runtime of tests/fake_cuda.cpp: its host
side runs here without a GPU, and the tests read what it asked of the runtime."""

import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
P, I, D = ctypes.c_void_p, ctypes.c_int, ctypes.c_double


def load(tmp):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2008_01966_gb300 import _lib, build
    inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    objs = [os.path.join(build.BUILD, s.replace(".cu", ".o")) for s in build.SOURCES]
    out = os.path.join(str(tmp), "libcavity_fake.so")
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", inc,
                    os.path.join(ROOT, "tests", "fake_cuda.cpp")] + objs + ["-Wl,-Bsymbolic", "-o", out],
                   check=True)
    lib = ctypes.CDLL(out)
    lib.fake_log.restype = lib.cavity_last_error.restype = ctypes.c_char_p
    lib.fake_log.argtypes = lib.fake_fail_alloc.argtypes = [ctypes.c_long]
    lib.fake_live.restype = lib.fake_peak.restype = ctypes.c_longlong
    lib.fake_allocs.restype = lib.fake_log_size.restype = ctypes.c_long
    lib.cavity_last_error.argtypes = lib.cavity_destroy.argtypes = [P]
    lib.cavity_destroy.restype = None
    return Fake(lib, _lib)


class Fake:
    def __init__(self, lib, defs):
        self.lib, self.defs = lib, defs

    def log(self, start=0):
        return [self.lib.fake_log(i).decode() for i in range(start, self.lib.fake_log_size())]

    def context(self, **kw):
        return Context(self, **kw)


class Context:
    """Calls of the C ABI with host memory for every buffer; each returns its status."""

    def __init__(self, fake, nx=32, ny=32, nz=8, precision="mixed", modes=0, solver="krylov",
                 stream=None):
        self.fake, self.lib = fake, fake.lib
        d = fake.defs.CavityDesc(1.0, 1.0, 0.5, nx, ny, nz, 0 if precision == "fp64" else 1, 0, 0.0, 0,
                                 0, 0.0, 0, modes, modes, fake.defs.SOLVERS[solver], 0)
        self.h = P()
        assert self.lib.cavity_setup(ctypes.byref(d), P(stream), ctypes.byref(self.h)) == 0
        nap, fpd = ctypes.c_longlong(), ctypes.c_longlong()
        self.lib.cavity_sizes(self.h, ctypes.byref(nap), ctypes.byref(fpd))
        self.n_ap, self.field_per_dir, self.nz = nap.value, fpd.value, nz
        self.el = 16 if precision == "fp64" else 8

    def close(self):
        self.lib.cavity_destroy(self.h)

    def layers(self, n):
        lev = [self.nz // n] * n
        lev[0] += self.nz - sum(lev)
        return (I * n)(*lev), (D * n)(*[1.0 + k for k in range(n)]), (D * n)(*[0.1 * k for k in range(n)])

    def prepare(self, kappa0=6.0, nlayers=1):
        return self.lib.cavity_prepare(self.h, D(kappa0), nlayers, *self.layers(nlayers))

    def apply(self, ndir, precision):
        x = np.empty((2, ndir * self.n_ap * 2))
        return self.lib.cavity_apply(self.h, ndir, precision, P(x[0].ctypes.data), P(x[1].ctypes.data))

    def field(self, ndir):
        ap = np.empty(ndir * self.n_ap * 2)
        out = np.empty(ndir * self.field_per_dir * self.el, np.uint8)
        return self.lib.cavity_field(self.h, ndir, P(ap.ctypes.data), P(out.ctypes.data))

    def rcs(self, ndir):
        ap, th, s = np.empty(ndir * self.n_ap * 2), np.zeros(ndir), np.empty(ndir)
        return self.lib.cavity_rcs(self.h, ndir, P(ap.ctypes.data), 0, P(th.ctypes.data),
                                   P(th.ctypes.data), 0, P(s.ctypes.data))

    def solve(self, ndir, field=True, host=False, kappa0=6.0, nlayers=1):
        ap, th = np.empty(ndir * self.n_ap * 2), np.zeros(ndir)
        out = np.empty(ndir * self.field_per_dir * self.el if field else 0, np.uint8)
        return self.lib.cavity_solve(
            self.h, D(kappa0), nlayers, *self.layers(nlayers), ndir, P(th.ctypes.data),
            P(th.ctypes.data), P(th.ctypes.data), 1 if field else 0, 1 if host else 0,
            P(ap.ctypes.data), P(out.ctypes.data) if field else None, None, None)
