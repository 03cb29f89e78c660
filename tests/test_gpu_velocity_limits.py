"""Field velocities where the kernel's arrangement meets its limits, against the
oracle's: numbers of field points around a warp and a block, points on the
quadrature points, scales inside and beyond the range of the integer seed of
1/sqrt, zero and negative weights.
"""

import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [0, -46, -60, 46, 60])
@pytest.mark.parametrize("P", [1, 32, 33, 128, 130])
def test_velocity_at_the_limits(P, scale):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_06468_gb300 import nrs
    rng = np.random.default_rng(P)
    N, Q, eps = 20, 333, 0.05
    x, X, xp = np.zeros((N, 4)), np.zeros((Q, 4)), np.zeros((P, 4))
    for a in (x, X, xp):
        a[:, :3] = rng.uniform(-1.0, 1.0, (len(a), 3))
    X[:, 3] = rng.choice([0.0, -0.01, 0.02, 0.03], Q)
    xp[: P // 2, :3] = X[: P // 2, :3]
    s = 2.0 ** scale
    for a in (x, X, xp):
        a[:, :3] *= s
    ctx = nrs.Context([0, N], [0, Q], [nrs.PRESCRIBED], eps=eps * s)
    xd, Xd = torch.from_numpy(x).cuda(), torch.from_numpy(X).cuda()
    nn, _, _ = ctx.nearest_build(xd, Xd)
    f = rng.normal(size=3 * N)
    u = ctx.velocity(torch.from_numpy(xp).cuda(), torch.from_numpy(f).cuda(), Xd).cpu().numpy()
    want = O.velocity(xp, X, nn.cpu().numpy(), f, eps * s, 1.0)
    # as for the other sizes: 1e-13 of the largest velocity
    assert np.abs(u - want).max() <= 1e-13 * np.abs(want).max()
    assert np.all(u[:, 3] == 0.0)
