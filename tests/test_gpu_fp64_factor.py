"""The FP64 factor and its triangular solves at sizes around their blocks of 64,
halves of 32 and panel strips of 16, against numpy's dense solve.
"""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 10, 11, 21, 22, 26, 27, 32, 43, 64, 85, 86, 107, 171, 299])
def test_fp64_factor_and_solve(N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_06468_gb300 import nrs
    n, copies = 3 * N, 4
    rng = np.random.default_rng(N)
    k = np.arange(N) + 0.5
    phi, z = np.pi * (1 + 5 ** 0.5) * k, 1 - 2 * k / N
    x = np.zeros((N, 4))
    x[:, :3] = np.stack([np.sqrt(1 - z * z) * np.cos(phi), np.sqrt(1 - z * z) * np.sin(phi), z], 1)
    h = (4 * np.pi / N) ** 0.5
    X = np.repeat(x, copies, axis=0)
    X[:, :3] += rng.uniform(-0.1 * h, 0.1 * h, (N * copies, 3))
    X[:, 3] = 1.0 / copies
    ctx = nrs.Context([0, N], [0, N * copies], [nrs.PRESCRIBED], eps=0.3 * h, factor_prec="fp64")
    xd, Xd = torch.from_numpy(x).cuda(), torch.from_numpy(X).cuda()
    ctx.nearest_build(xd, Xd)
    A = ctx.assemble(xd, Xd).cpu().numpy().T
    b = rng.normal(size=n)
    assert ctx.factor("fp64") == 0
    got, rep = ctx.solve(torch.from_numpy(b).cuda())
    want = np.linalg.solve(A, b)
    # an FP64 factor leaves one iteration a correction at most; both solutions
    # are within cond(A) n 2^-52 of the exact one
    assert rep[0]["converged"] and rep[0]["inner"] <= rep[0]["outer"] <= 3, rep
    assert rep[0]["backward_err"] < 1e-15, rep
    bound = 2 * np.linalg.cond(A) * n * 2.0 ** -52
    assert np.abs(got.cpu().numpy() - want).max() <= bound * np.linalg.norm(want)
