"""The FP64 operations on the integer pipe (csrc/fp64_int.cuh), compiled for the
host: every product, square root and reciprocal must be the correctly rounded
one, bit for bit what the processor's FP64 unit gives, over the whole range the
kernels use them in and at the edges of the significands.
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
extern "C" void run(long n, const double *p, const double *rho, const double *w, double *s,
                    double *v, unsigned char *tie, float *hi, float *lo)
{
    for (long i = 0; i < n; ++i) {
        bool t = false;
        const Sig si = inv_rho_sqrt(rho[i], t);
        const Sig sw = unpack(w[i]);
        s[i] = pack(si);
        v[i] = pack(mul_sig(mul_sig(unpack(p[i]), si.m << 1, si.f, t), sw.m << 1, sw.f, t));
        tie[i] = t;
        hi[i] = lo[i] = 0.0f;
        split_pair(p[i], hi[i], lo[i]);
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("fp64_int")
    (d / "t.cpp").write_text(SRC)
    subprocess.run([cxx, "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC,
                    str(d / "t.cpp"), "-o", str(d / "t.so")], check=True)
    return ctypes.CDLL(str(d / "t.so"))


def _significands(rng, n, kind):
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    if kind == "low":  # a power of two and a few units
        return m & np.uint64(0xff)
    if kind == "high":  # just below a power of two
        return np.uint64((1 << 52) - 1) - (m & np.uint64(0xff))
    if kind == "short":  # trailing zeros
        return m & ~((np.uint64(1) << rng.integers(0, 52, n, dtype=np.uint64)) - np.uint64(1))
    return m


def _doubles(rng, n, kind, lo, hi):
    e = rng.integers(1023 + lo, 1023 + hi, n, dtype=np.uint64)
    return ((e << np.uint64(52)) | _significands(rng, n, kind)).view(np.float64)


@pytest.mark.parametrize("kind", ["any", "low", "high", "short"])
def test_correctly_rounded(lib, kind):
    rng = np.random.default_rng(7)
    n = 400000
    p = _doubles(rng, n, kind, -69, 100) * rng.choice([-1.0, 1.0], n)
    rho = _doubles(rng, n, kind, -100, 100)
    w = _doubles(rng, n, kind, -200, 200)
    s, v = np.empty(n), np.empty(n)
    tie = np.empty(n, np.uint8)
    hi, lo = np.empty(n, np.float32), np.empty(n, np.float32)
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    lib.run(ctypes.c_long(n), *(ptr(a) for a in (p, rho, w, s, v, tie, hi, lo)))
    ok = tie == 0
    # a result that rests on a rounding tie is only ever left to the general path
    assert ok.mean() > (0.999999 if kind == "any" else 0.5)
    want = 1.0 / (rho * np.sqrt(rho))
    assert np.array_equal(s[ok], want[ok])
    assert np.array_equal(v[ok], ((p * want) * w)[ok])
    # the float pair: hi within half a unit, the sum to 2^-48
    assert np.all(np.abs(p - hi.astype(np.float64)) <= np.abs(p) * 2.0 ** -24)
    assert np.all(np.abs((p - hi.astype(np.float64)) - lo) <= np.abs(p) * 2.0 ** -48)
