"""The FP64 matrix with a force point that is not finite or very far away, in
both forms of its kernel, against the oracle: the rows of that point hold what
the definition gives there (NaN or zero), the others are unaffected.
"""

import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf, 2.0 ** 49, 2.0 ** 51, 2.0 ** 513,
                                   -(2.0 ** 600), 1e200])
@pytest.mark.parametrize("N,Q,axis", [(37, 211, 0), (129, 700, 1), (130, 700, 2)])
def test_matrix_with_a_far_force_point(N, Q, axis, value):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_06468_gb300 import nrs
    rng = np.random.default_rng(21)
    x, X, eps = np.zeros((N, 4)), np.zeros((Q, 4)), 0.05
    x[:, :3] = rng.uniform(-1.0, 1.0, (N, 3))
    X[:, :3] = rng.uniform(-1.0, 1.0, (Q, 3))
    X[:, 3] = rng.uniform(0.01, 0.02, Q)
    m = N // 2
    x[m, axis] = value
    ctx = nrs.Context([0, N], [0, Q], [nrs.PRESCRIBED], eps=eps, factor_prec="tf32")
    xd, Xd = torch.from_numpy(x).cuda(), torch.from_numpy(X).cuda()
    nn = ctx.nearest_build(xd, Xd)[0].cpu().numpy()
    assert np.all(nn >= 0) and not np.any(nn == m)
    want = O.assemble_stokeslet(x, X, nn, eps, 1.0)
    # with the matrix to return: the integer form
    got = ctx.assemble(xd, Xd).cpu().numpy().T
    assert np.array_equal(got, want, equal_nan=True)
    # beside the factorisation of a small system: the FP64 form, seen through A v
    ctx.assemble(xd, Xd, want_matrix=False)
    v = rng.normal(size=3 * N)
    b = torch.zeros(3 * N, dtype=torch.float64, device="cuda")
    r = ctx.residual(b, torch.from_numpy(v).cuda()).cpu().numpy()
    rows = np.isfinite(want).all(axis=1)
    bound = 3 * N * 2.0 ** -52 * (np.abs(want[rows]) @ np.abs(v))
    assert np.all(np.abs(r[rows] + want[rows] @ v) <= bound)
    assert np.all(np.isnan(r[~rows]))
