"""The integer form of a stokeslet pair (csrc/stokeslet_int.cuh), compiled for
the host, against the definition in the processor's FP64 arithmetic: a pair is
either reported for the general path or has the definition's bits, whatever its
coordinates.
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
#include "stokeslet_int.cuh"
using namespace nrs;
extern "C" void run(long n, const double *x, const double *X, const double *e2, double *out,
                    int *odd)
{
    const FmaOps op{1.0, -0.0};
    for (long i = 0; i < n; ++i) {
        const StagedX q = stage_weighted(X[4 * i], X[4 * i + 1], X[4 * i + 2], X[4 * i + 3]);
        const Acc6 v = terms_int(x[3 * i], x[3 * i + 1], x[3 * i + 2], q, e2[i], 2.0 * e2[i], op,
                                 odd[i]);
        const double t[6] = {v.xx, v.xy, v.xz, v.yy, v.yz, v.zz};
        for (int k = 0; k < 6; ++k) out[6 * i + k] = t[k];
    }
}
"""


@pytest.fixture(scope="module")
def terms(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("stokeslet_int")
    (d / "t.cpp").write_text(SRC)
    subprocess.run([cxx, "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC,
                    str(d / "t.cpp"), "-o", str(d / "t.so")], check=True)
    lib = ctypes.CDLL(str(d / "t.so"))

    def run(x, X, e2):
        x, X, e2 = (np.ascontiguousarray(a, dtype=np.float64) for a in (x, X, e2))
        out, odd = np.empty((len(x), 6)), np.empty(len(x), np.int32)
        lib.run(ctypes.c_long(len(x)), *(a.ctypes.data_as(ctypes.c_void_p)
                                         for a in (x, X, e2, out, odd)))
        return out, odd
    return run


def _definition(x, X, e2):
    with np.errstate(all="ignore"):
        r, w = x - X[:, :3], X[:, 3]
        r2 = (r[:, 0] * r[:, 0] + r[:, 1] * r[:, 1]) + r[:, 2] * r[:, 2]
        rho = r2 + e2
        s = 1.0 / (rho * np.sqrt(rho))
        dg = r2 + 2.0 * e2
        return np.stack([(r[:, j] * r[:, k] + dg if j == k else r[:, j] * r[:, k]) * s * w
                         for j, k in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))], axis=1)


def _cloud(n, seed):
    rng = np.random.default_rng(seed)
    X = np.concatenate([rng.uniform(-2.0, 2.0, (n, 3)), rng.uniform(0.01, 1.0, (n, 1))], axis=1)
    return rng, rng.uniform(-2.0, 2.0, (n, 3)), X, np.full(n, 1e-4)


def test_ordinary_pairs_have_the_bits_of_the_definition(terms):
    _, x, X, e2 = _cloud(100000, 1)
    got, odd = terms(x, X, e2)
    assert np.mean(odd == 0) > 0.9999
    assert np.array_equal(got[odd == 0], _definition(x, X, e2)[odd == 0])


@pytest.mark.parametrize("where", [(0,), (1,), (2,), (0, 2), (0, 1, 2)])
@pytest.mark.parametrize("value", ["nan", "inf", "-inf", "2**50", "2**500", "2**511", "2**512",
                                   "2**513", "2**600", "2**1000", "1e155", "1e170", "1e200"])
def test_far_and_non_finite_pairs_take_the_general_path(terms, value, where):
    rng, x, X, e2 = _cloud(2000, 2)
    for k in where:
        x[:, k] = eval(value) if "*" in value else float(value)
        if np.isfinite(x[0, k]):
            x[:, k] *= rng.uniform(1.1, 1.9, len(x)) * rng.choice([-1.0, 1.0], len(x))
    _, odd = terms(x, X, e2)
    assert np.all(odd >= 2)


def test_a_carry_in_a_product_where_the_reciprocal_is_a_power_of_two(terms):
    # r_j r_k = (1 - (i 2^-52)^2) 2^c rounds up to 2^c and rho is 4^k exactly: both
    # factors of the next product have rounded up to a power of two
    x, X, e2 = [], [], []
    for k in range(-8, 9):
        for c in range(0, 12):
            for i in (1, 2, 3, 5, 100):
                for axes in ((0, 1, 2), (1, 0, 2), (2, 0, 1), (0, 2, 1)):
                    for r3 in (0.0, 2.0 ** (k - 6)):
                        r = np.zeros(3)
                        r[axes[0]] = (1.0 + i * 2.0 ** -52) * 2.0 ** (k - 1)
                        r[axes[1]] = (1.0 - i * 2.0 ** -52) * 2.0 ** (k - 2 - c)
                        r[axes[2]] = r3
                        r2 = (r[0] * r[0] + r[1] * r[1]) + r[2] * r[2]
                        if r2 + (4.0 ** k - r2) == 4.0 ** k:
                            x.append(r)
                            X.append([0.0, 0.0, 0.0, 0.7])
                            e2.append(4.0 ** k - r2)
    x, X, e2 = np.array(x), np.array(X), np.array(e2)
    assert len(x) > 1000
    got, odd = terms(x, X, e2)
    want = _definition(x, X, e2)
    assert np.all(odd < 2)  # (a zero component: 1)
    assert np.array_equal(got, want)
