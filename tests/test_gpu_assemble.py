"""The FP64 matrix where the integer products of its kernel meet their limits,
bit for bit against the oracle: points in common planes and coincident points
(zero components), short significands (rounding ties), scales and weights
beyond the integer path's range, tile remainders.
"""

import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


def _cloud(kind, N, Q, rng):
    x = np.zeros((N, 4))
    X = np.zeros((Q, 4))
    x[:, :3] = rng.uniform(-1.0, 1.0, (N, 3))
    X[:, :3] = rng.uniform(-1.0, 1.0, (Q, 3))
    X[:, 3] = rng.uniform(0.01, 0.02, Q)
    eps = 0.05
    if kind == "planes":
        x[:, 2] = 0.25
        X[: Q // 2, 2] = 0.25
        X[::3, 0] = x[np.arange(len(X[::3])) % N, 0]
        X[: min(N, Q), :3] = x[: min(N, Q), :3]
    elif kind == "short":  # differences of 27 bits: their products may end in a tie
        x[:, :3] = rng.integers(1 << 26, 1 << 27, (N, 3)) * 2.0 ** -20
        X[:, :3] = rng.integers(-(1 << 26), 0, (Q, 3)) * 2.0 ** -20
        eps = 2.0 ** -3
    elif kind == "weights":
        X[:, 3] = rng.choice([0.0, -0.5, 2.0 ** -210, 2.0 ** 210, 1e-308 / 7, 1.0], Q)
    elif kind == "tiny_component":
        x[:, 0] = 0.0
        X[:, 0] = rng.choice([0.0, -0.0, 2.0 ** -160, 2.0 ** -140], Q)
    elif kind.startswith("scale"):
        f = 2.0 ** float(kind[5:])
        x[:, :3] *= f
        X[:, :3] *= f
        eps *= f
    return x, X, eps


@pytest.mark.parametrize("kind", ["plain", "planes", "short", "weights", "tiny_component",
                                  "scale-48", "scale-60", "scale47", "scale60"])
@pytest.mark.parametrize("N,Q", [(1, 3), (37, 211), (129, 700)])
def test_matrix_bits_at_the_limits(N, Q, kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_06468_gb300 import nrs
    x, X, eps = _cloud(kind, N, Q, np.random.default_rng(11))
    ctx = nrs.Context([0, N], [0, Q], [nrs.PRESCRIBED], eps=eps)
    xd, Xd = torch.from_numpy(x).cuda(), torch.from_numpy(X).cuda()
    nn, _, _ = ctx.nearest_build(xd, Xd)
    got = ctx.assemble(xd, Xd).cpu().numpy().T
    want = O.assemble_stokeslet(x, X, nn.cpu().numpy(), eps, 1.0)
    assert np.array_equal(got, want)


def test_the_callers_points_may_be_overwritten_in_stream_order():
    # the FP64 matrix is assembled beside the caller's stream: what that does to
    # its buffers after nrs_assemble must not reach it
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_06468_gb300 import nrs
    N, Q = 1500, 15000
    x, X, eps = _cloud("plain", N, Q, np.random.default_rng(12))
    v = torch.from_numpy(np.random.default_rng(13).normal(size=3 * N)).cuda()
    b = torch.zeros_like(v)
    got = []
    for overwrite in (False, True):
        ctx = nrs.Context([0, N], [0, Q], [nrs.PRESCRIBED], eps=eps, factor_prec="tf32")
        xd, Xd = torch.from_numpy(x).cuda(), torch.from_numpy(X).cuda()
        ctx.nearest_build(xd, Xd)
        ctx.assemble(xd, Xd, want_matrix=False)
        if overwrite:
            xd.zero_()
            Xd.zero_()
        got.append(ctx.residual(b, v).cpu().numpy())
    assert np.array_equal(got[0], got[1])
