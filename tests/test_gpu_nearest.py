"""The pruned nearest-neighbour search against the oracle's exhaustive one, bit
for bit, where its pruning has least to go by: points in arbitrary order,
clusters far apart, exact ties across boxes, bodies that end inside a box of 32
points, more boxes than a block lists at a time, coordinates that are not
finite; and segments longer than a warp sorts at once.
"""

import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nrs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_06468_gb300 import nrs
    return nrs


def _clouds(kind, N, Q, rng):
    x, X = np.zeros((N, 4)), np.zeros((Q, 4))
    x[:, :3], X[:, :3] = rng.uniform(-1, 1, (N, 3)), rng.uniform(-1, 1, (Q, 3))
    if kind == "curve":  # neighbours in index order are neighbours in space
        for a, n in ((x, N), (X, Q)):
            s = np.linspace(0.0, 30.0, n)
            a[:, :3] = np.stack([np.cos(s), np.sin(s), 0.1 * s], axis=1)
    elif kind == "clusters":
        x[:, :3] = 1e-3 * x[:, :3] + rng.choice([-50.0, 0.0, 50.0], (N, 3))
        X[:, :3] = 1e-3 * X[:, :3] + rng.choice([-50.0, 0.0, 50.0], (Q, 3))
    elif kind == "lattice":  # exact ties everywhere
        x[:, :3], X[:, :3] = rng.integers(0, 4, (N, 3)), rng.integers(0, 8, (Q, 3)) * 0.5
    elif kind == "tiny":
        x[:, :3] *= 1e-21
        X[:, :3] *= 1e-21
    return x, X


def _segments(nn, N):
    perm = np.argsort(nn, kind="stable")
    return np.concatenate([[0], np.cumsum(np.bincount(nn, minlength=N))]), perm


@pytest.mark.parametrize("kind", ["random", "curve", "clusters", "lattice", "tiny"])
@pytest.mark.parametrize("n_off,q_off", [([0, 1], [0, 70]), ([0, 33, 95, 96], [0, 200, 500, 501]),
                                         ([0, 17001], [0, 1500])])
def test_exhaustive_search(nrs, kind, n_off, q_off):
    n_off, q_off = np.array(n_off), np.array(q_off)
    x, X = _clouds(kind, n_off[-1], q_off[-1], np.random.default_rng(3))
    xd, Xd = torch.from_numpy(x).cuda(), torch.from_numpy(X).cuda()
    for glob in (False, True):
        one = (np.array([0, n_off[-1]]), np.array([0, q_off[-1]])) if glob else (n_off, q_off)
        want = O.nearest(x, X, *one)
        seg, perm = _segments(want, n_off[-1])
        got = [t.cpu().numpy() for t in nrs.nearest_build_static(xd, Xd, n_off, q_off, glob)]
        if n_off[-1] < 1000:
            ctx = nrs.Context(n_off, q_off, [nrs.PRESCRIBED] * (len(n_off) - 1), eps=0.1,
                              nn_global=glob)
            for a, b in zip(ctx.nearest_build(xd, Xd), got):
                assert np.array_equal(a.cpu().numpy(), b)
        assert np.array_equal(got[0], want)
        assert np.array_equal(got[1], seg) and np.array_equal(got[2], perm)


def test_coordinates_that_are_not_finite(nrs):
    rng = np.random.default_rng(4)
    x, X = _clouds("random", 100, 300, rng)
    x[5, 0], x[40, 1], x[77, 2] = np.nan, np.inf, -np.inf
    X[17, 0], X[200, 1] = np.nan, np.inf
    nn, seg, perm = nrs.nearest_build_static(torch.from_numpy(x).cuda(), torch.from_numpy(X).cuda(),
                                             [0, 100], [0, 300], check=False)
    torch.cuda.synchronize()
    nn = nn.cpu().numpy()
    fine = np.ones(300, bool)
    fine[[17, 200]] = False
    ok = np.all(np.isfinite(x), axis=1)
    back = np.flatnonzero(ok)
    assert np.all(nn[~fine] < 0)
    assert np.array_equal(nn[fine], back[O.nearest(x[ok], X[fine], [0, len(back)], [0, fine.sum()])])
    assert seg[-1].item() == fine.sum()
