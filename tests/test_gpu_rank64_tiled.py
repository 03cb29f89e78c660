"""The rank-64 update where its tiles of the matrix go through shared memory (more
than a wave of tiles): whole and ragged last tiles, a matrix whose column stride
no tensor map takes, and a one-level factorisation, whose tiles on the block row
and column being finished are left to the plain path.
"""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nrs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_06468_gb300 import nrs
    return nrs


def _sphere(nrs, N, **kw):
    k = np.arange(N) + 0.5
    phi, z = np.pi * (1 + 5 ** 0.5) * k, 1 - 2 * k / N
    x = np.zeros((N, 4))
    x[:, :3] = np.stack([np.sqrt(1 - z * z) * np.cos(phi), np.sqrt(1 - z * z) * np.sin(phi), z], 1)
    h = (4 * np.pi / N) ** 0.5
    X = np.repeat(x, 4, axis=0)
    X[:, :3] += np.random.default_rng(N).uniform(-0.1 * h, 0.1 * h, (4 * N, 3))
    X[:, 3] = 0.25
    return nrs.Context([0, N], [0, 4 * N], [nrs.PRESCRIBED], eps=0.3 * h, **kw), x, X


@pytest.mark.parametrize("n,lda", [(2816, 2816), (2689, 2720), (3001, 3001), (3001, 3002), (2700, 2700)])
def test_update(nrs, n, lda):
    ctx, _, _ = _sphere(nrs, 8)
    rng = np.random.default_rng(n + lda)
    M = rng.normal(size=(n, lda)).astype(np.float32)  # Mt[j, i] = M[i, j]
    C, R = (rng.normal(size=(n, 64)).astype(np.float32) for _ in range(2))
    Mt = torch.from_numpy(M).cuda()
    ctx.rank64_update(Mt, torch.from_numpy(C).cuda(), torch.from_numpy(R).cuda(), "tf32")
    got = Mt.cpu().numpy().astype(np.float64)
    want = M[:, :n].astype(np.float64) - (C.astype(np.float64) @ R.astype(np.float64).T).T
    bound = (np.abs(C).astype(np.float64) @ np.abs(R).astype(np.float64).T).T
    # as for the other sizes: the split form's 1e-5 of the absolute product
    assert np.all(np.abs(got[:, :n] - want) <= 1e-5 * bound + 1e-6 * np.abs(want))
    assert np.array_equal(got[:, n:], M[:, n:].astype(np.float64))


@pytest.mark.parametrize("N", [900, 939, 981])
def test_factor(nrs, N):
    ctx, x, X = _sphere(nrs, N, factor_prec="tf32")
    xd, Xd = torch.from_numpy(x).cuda(), torch.from_numpy(X).cuda()
    ctx.nearest_build(xd, Xd)
    ctx.assemble(xd, Xd, want_matrix=False)
    assert ctx.factor("tf32") == 0
    b = torch.from_numpy(np.random.default_rng(1).normal(size=3 * N)).cuda()
    _, rep = ctx.solve(b)
    # an inverse with a wrong tile still converges, but takes many iterations
    assert rep[0]["converged"] and rep[0]["outer"] <= 4, rep
    assert rep[0]["inner"] <= 2 * rep[0]["outer"], rep
    assert rep[0]["backward_err"] < 1e-15, rep
