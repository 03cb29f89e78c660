"""The exact product of the refinement's residual (csrc/fp64_int.cuh), compiled
for the host, against Python's integers: |x v| 2^-L truncated toward zero, for
places inside and on both sides of the range the plain placement takes, zeros,
subnormal factors, and products that have no room.
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
extern "C" void run(long n, const double *x, const double *v, const int *c, unsigned long *z,
                    unsigned char *bad)
{
    for (long i = 0; i < n; ++i) {
        const FxFactor a = fx_factor(x[i], 0), f = fx_factor(v[i], c[i]);
        int32_t s = a.s + 1075 + f.s;
        FxWords w = fx_product(a.m, f.m);
        bad[i] = (uint32_t)s > 86u && !fx_move(w, s);
        const FxPlaced p = fx_place(w, (uint32_t)s);
        z[3 * i] = p.z0, z[3 * i + 1] = p.z1, z[3 * i + 2] = p.z2;
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("fx_product")
    (d / "t.cpp").write_text(SRC)
    subprocess.run([cxx, "-O2", "-shared", "-fPIC", "-I", CSRC, str(d / "t.cpp"), "-o",
                    str(d / "t.so")], check=True)
    return ctypes.CDLL(str(d / "t.so"))


@pytest.mark.parametrize("kind", ["normal", "subnormal", "zero", "full"])
def test_placed_product(lib, kind):
    rng = np.random.default_rng(11)
    n = 20000
    m = rng.integers(0, 1 << 52, (2, n), dtype=np.uint64)
    e = rng.integers(1, 2047, (2, n), dtype=np.uint64)
    if kind == "full":
        m[:] = (1 << 52) - 1 - (m & np.uint64(3))
    if kind == "subnormal":
        e[1] = 0
        m[1] >>= rng.integers(0, 52, n, dtype=np.uint64)
    if kind == "zero":
        e[1] = m[1] = 0
    sign = rng.integers(0, 2, (2, n), dtype=np.uint64) << np.uint64(63)
    x, v = ((e << np.uint64(52)) | m | sign).view(np.float64)
    e1 = np.maximum(e, 1).astype(np.int64)
    s = rng.integers(-140, 200, n)  # the place of the product's lowest bit
    c = (e1[0] + e1[1] - 1075 - s).astype(np.int32)
    z, bad = np.zeros((n, 3), np.uint64), np.zeros(n, np.uint8)
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    x, v = np.ascontiguousarray(x), np.ascontiguousarray(v)
    lib.run(ctypes.c_long(n), ptr(x), ptr(v), ptr(c), ptr(z), ptr(bad))
    sig = [(mm + ((ee > 0).astype(np.uint64) << np.uint64(52))) for mm, ee in zip(m, e)]
    for i in range(n):
        p = int(sig[0][i]) * int(sig[1][i])
        want = p << int(s[i]) if s[i] >= 0 else p >> int(-s[i])
        if want >> 192:
            assert bad[i], i
        elif not bad[i]:
            assert sum(int(z[i, k]) << (64 * k) for k in range(3)) == want, (i, int(s[i]))
        # a product below half of the integer's range always has room
        assert not (bad[i] and want >> 191 == 0), i
