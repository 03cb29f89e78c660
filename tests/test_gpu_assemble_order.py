"""The FP64 matrix is formed on a side stream beside what the caller does next:
calls that rewrite its inputs (another nearest-neighbour map, another assembly,
a recorded step) must not reach it.
"""

import numpy as np
import pytest
import torch

from synth import geometry as g

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nrs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_06468_gb300 import nrs
    return nrs


def _cloud(seed, N=1500, Q=15000):
    rng = np.random.default_rng(seed)
    x, X = np.zeros((N, 4)), np.zeros((Q, 4))
    x[:, :3], X[:, :3] = rng.uniform(-1.0, 1.0, (N, 3)), rng.uniform(-1.0, 1.0, (Q, 3))
    X[:, 3] = rng.uniform(0.01, 0.02, Q)
    return torch.from_numpy(x).cuda(), torch.from_numpy(X).cuda()


@pytest.mark.parametrize("other", ["map", "assembly"])
def test_calls_after_an_assembly(nrs, other):
    (x0, X0), (x1, X1) = _cloud(31), _cloud(32)
    N, Q = x0.shape[0], X0.shape[0]
    v = torch.from_numpy(np.random.default_rng(33).normal(size=3 * N)).cuda()
    b = torch.zeros_like(v)
    got = []
    for disturbed in (False, True):
        ctx = nrs.Context([0, N], [0, Q], [nrs.PRESCRIBED], eps=0.05, factor_prec="tf32")
        if other == "map":
            ctx.nearest_build(x0, X0)
            ctx.assemble(x0, X0, want_matrix=False)
            if disturbed:
                ctx.nearest_build(x1, X1)
        else:
            ctx.nearest_build(x1, X1)
            if disturbed:
                ctx.assemble(x0, X0, want_matrix=False)
            ctx.assemble(x1, X1, want_matrix=False)
        ctx.factor("tf32")
        got.append(ctx.residual(b, v).cpu().numpy())
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("recorded", [False, True])
def test_a_recorded_step_after_an_assembly(nrs, recorded):
    pr = g.swimmer_config(ns_f=20, nth_f=4, ns_q=100, nth_q=8)
    Y = g.initial_state(pr)
    s0, sh = (nrs.shapes_to_device(g.pack_shapes(pr, t)) for t in (0.1, 0.105))
    s0, sh = nrs.Context.shapes(*s0), nrs.Context.shapes(*sh)
    got = []
    for disturbed in (False, True):
        ctx = nrs.Context.from_problem(pr, factor_prec="tf32", graph=True)
        sol = torch.empty(2 * pr.n, dtype=torch.float64, device="cuda")
        ctx.set_state(Y["x0"], Y["B"])
        # the first step is not recorded, the second records, the third replays
        steps = 3 if recorded else 2
        for k in range(steps):
            if disturbed and k == steps - 1:
                x = torch.zeros((pr.N, 4), dtype=torch.float64, device="cuda")
                Xw = torch.ones((pr.Q, 4), dtype=torch.float64, device="cuda")
                ctx.assemble(x, Xw, want_matrix=False)
            ctx.step(s0, sh, 0.01, sol=sol)
        got.append(sol.cpu().numpy())
    assert np.array_equal(got[0], got[1])


def test_a_map_captured_after_an_assembly(nrs):
    # the capture of a call that rewrites the segments, with an assembly from
    # before it still unjoined
    (x0, X0), (x1, X1) = _cloud(34), _cloud(35)
    N, Q = x0.shape[0], X0.shape[0]
    stream = torch.cuda.Stream()
    ctx = nrs.Context([0, N], [0, Q], [nrs.PRESCRIBED], eps=0.05, factor_prec="tf32", stream=stream)
    with torch.cuda.stream(stream):
        want = [t.cpu() for t in ctx.nearest_build(x1, X1)]
        ctx.nearest_build(x0, X0)
        ctx.assemble(x0, X0, want_matrix=False)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        got = ctx.nearest_build(x1, X1)
    graph.replay()
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a.cpu(), b)
