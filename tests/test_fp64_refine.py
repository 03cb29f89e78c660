"""The refined approximations of csrc/fp64_int.cuh that are not correctly
rounded, compiled for the host, against extended precision: the reciprocal of
the FP64 factorisation's pivots and the powers of 1/sqrt(rho) of the field
velocities.  The bounds are the sums of the steps' own rounding errors.
"""

import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2001_06468_gb300", "csrc")
SRC = r"""
#include "fp64_int.cuh"
using namespace nrs;
extern "C" void rcp(long n, const double *x, const double *y, double *r)
{
    for (long i = 0; i < n; ++i) r[i] = rcp_refined(x[i], y[i]);
}
extern "C" void cube(long n, const double *rho, double *r)
{
    for (long i = 0; i < n; ++i) {
        double y2, y3;
        rsqrt_powers(rho[i], y2, y3);
        r[i] = fma(1.5, y3 * fma(-rho[i], y2, 1.0), y3);
    }
}
"""
U = 2.0 ** -53


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("fp64_refine")
    (d / "t.cpp").write_text(SRC)
    subprocess.run([cxx, "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC,
                    str(d / "t.cpp"), "-o", str(d / "t.so")], check=True)
    return ctypes.CDLL(str(d / "t.so"))


def _call(f, *arrays):
    out = np.empty(len(arrays[0]))
    f(ctypes.c_long(len(out)), *(a.ctypes.data_as(ctypes.c_void_p) for a in (*arrays, out)))
    return out


def _significands(rng, n, kind):
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    if kind == "low":  # a power of two and a few units
        return m & np.uint64(0xff)
    if kind == "high":  # just below a power of two
        return np.uint64((1 << 52) - 1) - (m & np.uint64(0xff))
    return m


def _doubles(rng, n, kind, lo, hi):
    e = rng.integers(1023 + lo, 1023 + hi, n, dtype=np.uint64)
    return ((e << np.uint64(52)) | _significands(rng, n, kind)).view(np.float64)


@pytest.mark.parametrize("kind", ["any", "low", "high"])
def test_reciprocal(lib, kind):
    rng = np.random.default_rng(51)
    n = 200000
    x = _doubles(rng, n, kind, -960, 960) * rng.choice([-1.0, 1.0], n)
    # seeds of 20 bits (the low word zero) and any within 2^-19
    y = (1.0 / x) * (1.0 + rng.uniform(-1.0, 1.0, n) * 2.0 ** -19.1)
    coarse = (y.view(np.uint64) & np.uint64(0xffffffff00000000)).view(np.float64)
    for seed in (y, np.where(np.abs(coarse * x - 1.0) < 2.0 ** -19, coarse, y)):
        r = _call(lib.rcp, x, seed)
        exact = np.longdouble(1.0) / x.astype(np.longdouble)
        # e^3 <= 2^-57 = 2^-4 u of the value, at most 2^-4 units in the last place
        assert np.all(np.abs(r - exact) <= (0.5 + 2.0 ** -4) * np.spacing(np.abs(r)))


@pytest.mark.parametrize("kind", ["any", "low", "high"])
def test_inverse_cube_of_the_root(lib, kind):
    rng = np.random.default_rng(52)
    rho = _doubles(rng, 200000, kind, -100, 100)
    r = _call(lib.cube, rho)
    root = np.sqrt(rho.astype(np.longdouble))
    exact = np.longdouble(1.0) / (rho.astype(np.longdouble) * root)
    # y^3 and the result rounded once each (2 u), y^2 rounded (1.5 u), the series'
    # next term 15/8 e^2 with |e| <= 2^-27 (0.94 u)
    assert np.all(np.abs(r - exact) <= 4.45 * U * np.abs(exact))
