"""The learned start's network at numbers of points around a warp's four and a
gradient block's 32, against the FP64 oracle; tolerances as derived there for
the other sizes (FP32 layers within 3e-5 of their absolute sums, gradients
within 1e-4 of theirs).
"""

import numpy as np
import pytest
import torch

import oracle.mlp as OM
from synth import geometry as g
from synth import mlp_batch, mlp_init, mlp_perturb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npts", [2, 3, 4, 5, 15, 16, 17, 31, 32, 33, 63, 65, 257, 797])
def test_network_and_gradient(npts):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_06468_gb300 import nrs
    P = mlp_perturb(1, mlp_init(2), 0.1)
    ctx = nrs.Context.from_problem(g.swimmer_config())
    ctx.mlp_set_params(P)
    X, T = mlp_batch(900 + npts, npts)
    Y, G, loss = ctx.mlp_eval(torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda(), grad=True,
                              loss=True)
    P, X, T = (a.astype(np.float64) for a in (P, X, T))
    assert np.all(np.abs(Y.cpu().numpy() - OM.forward(P, X)[0]) <= 3e-5 * OM.forward_abs(P, X))
    want, want_loss = OM.grad(P, X, T)
    assert np.all(np.abs(G.cpu().numpy() - want) <= 1e-4 * OM.grad_abs(P, X, T) + 1e-30)
    assert abs(loss - want_loss) <= 1e-5 * want_loss
