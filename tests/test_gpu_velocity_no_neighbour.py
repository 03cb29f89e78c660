"""Velocities where some quadrature point has no nearest force point (its
coordinates are not finite, or too far for a finite distance): the definition
has no density for it, so every velocity is NaN, and nothing outside the density
is read.
"""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("where", ["quadrature nan", "quadrature far", "all force points nan"])
def test_velocity_without_a_neighbour(where):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_06468_gb300 import nrs
    N, Q, P = 20, 333, 130
    rng = np.random.default_rng(41)
    x, X, xp = (np.concatenate([rng.uniform(-1.0, 1.0, (k, 3)), np.full((k, 1), 0.02)], axis=1)
                for k in (N, Q, P))
    bad = np.zeros(Q, bool)
    if where == "quadrature nan":
        X[[0, 200], 1] = np.nan
        bad[[0, 200]] = True
    elif where == "quadrature far":
        X[332, 0] = 1e200
        bad[332] = True
    else:
        x[:, 2] = np.nan
        bad[:] = True
    ctx = nrs.Context([0, N], [0, Q], [nrs.PRESCRIBED], eps=0.05)
    Xd = torch.from_numpy(X).cuda()
    nn = ctx.nearest_build(torch.from_numpy(x).cuda(), Xd)[0].cpu().numpy()
    assert np.array_equal(nn < 0, bad)
    f = torch.from_numpy(rng.normal(size=3 * N)).cuda()
    u = ctx.velocity(torch.from_numpy(xp).cuda(), f, Xd).cpu().numpy()
    assert np.all(np.isnan(u[:, :3])) and np.all(u[:, 3] == 0.0)
    with pytest.raises(nrs.NrsError) as e:
        ctx.sync()
    assert e.value.status == nrs.NRS_ENONFINITE
