"""The pruned nearest-neighbour search where boxes do not tell points apart and
where many force points lie at one distance, against the oracle's exhaustive
search, bit for bit: more equally distant candidates than a lane keeps, in one
chunk of boxes and in several, and clouds in no spatial order.
"""

import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["shuffled curve", "duplicates", "one place", "near ties"])
@pytest.mark.parametrize("N,Q", [(63, 130), (700, 400), (2500, 700), (17001, 300)])
def test_exhaustive_search(N, Q, kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_06468_gb300 import nrs
    rng = np.random.default_rng(N + Q)
    x, X = np.zeros((N, 4)), np.zeros((Q, 4))
    if kind == "shuffled curve":
        for a in (x, X):
            s = rng.permutation(np.linspace(0.0, 30.0, len(a)))
            a[:, :3] = np.stack([np.cos(s), np.sin(s), 0.1 * s], axis=1)
    elif kind == "duplicates":  # each place many times over, in no order
        x[:, :3], X[:, :3] = rng.integers(0, 3, (N, 3)), rng.integers(0, 6, (Q, 3)) * 0.5
    elif kind == "one place":
        x[:, :3], X[:, :3] = 0.25, rng.uniform(-1, 1, (Q, 3))
    else:  # distances that FP32 does not tell apart, in descending order of the index
        d = rng.normal(size=(N, 3))
        d /= np.linalg.norm(d, axis=1)[:, None]
        x[:, :3] = d * (1.0 + 1e-12 * np.arange(N, 0, -1))[:, None]
        X[:, :3] = 1e-14 * rng.normal(size=(Q, 3))
    want = O.nearest(x, X, [0, N], [0, Q])
    got = nrs.nearest_build_static(torch.from_numpy(x).cuda(), torch.from_numpy(X).cuda(), [0, N],
                                   [0, Q])[0].cpu().numpy()
    assert np.array_equal(got, want)
