"""The reciprocal of a pivot in the per-mode elimination (csrc/zquot.h), built
on its own with g++ and compared with 80-bit values and with a division: real
pivots (a lossless fill) have to come out correctly rounded, complex ones no
further off than Smith's scaled division, pivots of any size in range."""

import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2008_01966_gb300", "csrc")

SHIM = """
#include "zquot.h"
extern "C" void shim(const double* x, const double* y, double* qx, double* qy, double* n2, long n) {
  for (long i = 0; i < n; ++i) n2[i] = zquot(x[i], y[i], qx[i], qy[i]);
}
"""


@pytest.fixture(scope="module")
def quot(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("zquot")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC,
                    str(d / "shim.cpp"), "-o", str(d / "shim.so")], check=True)
    lib = ctypes.CDLL(str(d / "shim.so"))

    def f(x, y):
        out = np.empty((3, x.size))
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
        lib.shim(p(x), p(y), p(out[0]), p(out[1]), p(out[2]), ctypes.c_long(x.size))
        return out
    return f


def smith(x, y):
    big = np.abs(x) >= np.abs(y)
    r = np.where(big, y / np.where(big, x, 1), x / np.where(big, 1, y))
    d = np.where(big, x + y * r, y + x * r)
    return np.where(big, 1 / d, r / d), np.where(big, -r / d, -1 / d)


def units(x, y, qx, qy):
    """Error of q against 1 / (x + i y), in units of 2^-53 of its magnitude."""
    X, Y = x.astype(np.longdouble), y.astype(np.longdouble)
    n = X * X + Y * Y
    return np.hypot(qx - X / n, qy + Y / n) * np.sqrt(n) * 2.0 ** 53


@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 63, reason="no 80-bit type here")
@pytest.mark.parametrize("scale", [1e-12, 1e-3, 1.0, 50.0])
def test_against_80_bits(quot, scale):
    rng = np.random.default_rng(11)
    n = 200000
    x = scale * (1 + 0.9 * rng.uniform(-1, 1, n))
    # lossless
    qx, qy, n2 = quot(x, np.zeros(n))
    assert np.array_equal(qx, 1.0 / x) and np.all(qy == 0)
    assert np.allclose(n2, x * x, rtol=1e-15)
    qx, _, _ = quot(-x, np.zeros(n))
    assert np.array_equal(qx, -1.0 / x)
    # slightly lossy, lossy, nearly imaginary
    for xx, yy in ((x, 1e-3 * scale * rng.uniform(-1, 1, n)), (x, scale * rng.uniform(-1, 1, n)),
                   (1e-3 * scale * rng.uniform(-1, 1, n), x)):
        qx, qy, _ = quot(xx, yy)
        e, s = units(xx, yy, qx, qy), units(xx, yy, *smith(xx, yy))
        assert np.sqrt(np.mean(e.astype(float) ** 2)) <= np.sqrt(np.mean(s.astype(float) ** 2))
        assert e.max() < 3.0


def test_a_vanishing_pivot_is_not_finite(quot):
    qx, _, n2 = quot(np.zeros(1), np.zeros(1))
    assert n2[0] == 0 and not np.isfinite(qx[0])
