"""A solve that meets a value that is not finite says so in its whole report: the
status, no convergence, and a backward error that is not finite either (a norm
that leaves NaN out would report zero).
"""

import numpy as np
import pytest
import torch

from synth import geometry as g

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("residual", ["extended", "fp64"])
@pytest.mark.parametrize("prec,mode", [("fp64", "device"), ("tf32", "device"), ("tf32", "host"),
                                       ("fp32", "host")])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_right_hand_side(bad, prec, mode, residual):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_06468_gb300 import nrs
    pr = g.swimmer_config(ns_f=20, nth_f=4, ns_q=100, nth_q=8)
    ctx = nrs.Context.from_problem(pr, factor_prec=prec, solve_mode=mode, residual=residual)
    Y = g.initial_state(pr)
    ctx.set_state(Y["x0"], Y["B"])
    xi, Xiw, xidot = nrs.shapes_to_device(g.pack_shapes(pr, 0.2))
    x, Xw, b = ctx.kinematics(xi, Xiw, xidot)
    ctx.nearest_build(xi, Xiw)
    ctx.assemble(x, Xw, want_matrix=False)
    ctx.factor(prec)
    _, rep = ctx.solve(b, check=False)
    assert rep[0]["status"] == nrs.NRS_OK and rep[0]["converged"]
    b[pr.n // 3] = bad
    _, rep = ctx.solve(b, check=False)
    assert rep[0]["status"] == nrs.NRS_ENONFINITE, rep
    assert not rep[0]["converged"] and not np.isfinite(rep[0]["backward_err"]), rep
