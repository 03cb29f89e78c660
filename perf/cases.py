"""Workloads whose speed matters to a user of this library, each one pass
through its public entry points (``paper_2001_06468_gb300.nrs``).

Kinds of cases (``case["kind"]``):

* ``resistance``  the quasi-static rigid-body problem: lab frame, nearest
                  neighbours, matrix, factor and six right-hand sides.
* ``matrix``      the stages up to the FP64 matrix, handed to the caller.
* ``solve``       factor and refined solution of an assembled system, in the
                  mixed-precision or the plain FP64 path.
* ``nearest``     the nearest-neighbour map and its segments.
* ``velocity``    the fluid velocity at field points (particle tracking).
* ``learn``       one training iteration of the learned starting vector.
* ``replay``      one time step of free tubes, recorded as a CUDA graph.
* ``tubes``       one time step of several free tubes, with factor reuse.
* ``channel``     three time steps of sperm-like cells in a closed channel,
                  with factor reuse and warm starts.
* ``batch``       one time step of many uneven problems as one graph.

Inputs come from the synthetic generators in ``synth``; the seed moves the
bodies, their phases of the beat, the loads and the random points, never the
sizes.
"""

import math

import numpy as np
import torch

from paper_2001_06468_gb300 import nrs
from synth import geometry as geo
from synth import mlp_inputs

DT = 0.01


def listed():
    return [
        # the smallest problems: a coarse rigid sphere in the default precision, where the
        # latency of launches and of short dependent kernels counts
        dict(name="sphere_coarse", kind="resistance", cells_f=4, cells_q=16, prec="fp32"),
        # the paper's sphere (Sec. 3): 864 force and 3456 quadrature points
        dict(name="sphere_paper", kind="resistance", cells_f=12, cells_q=24, prec="tf32"),
        # a user who wants the FP64 matrix itself: one tube of 2000 / 20000 points
        dict(name="matrix_tube", kind="matrix", ns_f=200, nth_f=10, ns_q=1000, nth_q=20),
        # mixed-precision factor and solve of an ill-conditioned system of odd order
        dict(name="solve_mixed", kind="solve", ns_f=131, nth_f=13, ns_q=524, nth_q=26, prec="tf32"),
        # the plain FP64 factor and solve on the single swimmer
        dict(name="solve_fp64", kind="solve", ns_f=80, nth_f=10, ns_q=400, nth_q=20, prec="fp64"),
        # nearest neighbours and segments of the whole channel, over all bodies
        dict(name="nearest_channel", kind="nearest", cells=8, wall=90, scope="global"),
        # 2000 tracers in the channel's flow
        dict(name="velocity_tracers", kind="velocity", cells=8, wall=90, points=2000),
        # one full-batch training iteration on the channel's force points
        dict(name="learn_channel", kind="learn", points=9200),
        # the single swimmer, one recorded time step
        dict(name="swimmer_replay", kind="replay", count=1, ns_f=80, nth_f=10, ns_q=400, nth_q=20),
        # four swimmers (14064 unknowns, ill-conditioned), one time step
        dict(name="swimmers4_step", kind="tubes", count=4, ns_f=117, nth_f=10, ns_q=468, nth_q=20),
        # eight cells in a closed channel (27648 unknowns), a stretch of three time steps
        dict(name="channel_steps", kind="channel", cells=8, wall=90),
        # thirty-two uneven ventral-node problems as one graph
        dict(name="node_batch", kind="batch", count=32, first=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["resistance", "matrix", "solve", "solve", "nearest", "velocity", "learn",
                       "replay", "replay", "tubes", "channel", "batch"])
    if kind == "resistance":
        c = rng.randint(4, 13)
        return dict(kind=kind, cells_f=c, cells_q=c * rng.randint(2, 3), prec=rng.choice(["fp32", "tf32"]))
    if kind in ("matrix", "solve", "replay"):
        prec = rng.choice(["tf32", "tf32", "fp64"]) if kind == "solve" else "tf32"
        top = 1000 if prec == "fp64" or kind == "replay" else 1700
        N = _log(rng, 100, top)
        # rings closer than eps along the tube leave systems no FP32 inverse preconditions
        nth = rng.randint(6, 10) if N < 800 else 13
        ns = max(12, N // nth)
        c = dict(kind=kind, ns_f=ns, nth_f=nth, ns_q=ns * rng.randint(3, 5), nth_q=2 * nth)
        if kind == "solve":
            c["prec"] = prec
        if kind == "replay":
            c["count"] = 1
        return c
    if kind == "nearest":
        return dict(kind=kind, cells=rng.randint(2, 8), wall=rng.randint(20, 90),
                    scope=rng.choice(["global", "body", "static"]))
    if kind == "velocity":
        return dict(kind=kind, cells=rng.randint(2, 8), wall=rng.randint(20, 80), points=_log(rng, 40, 2000))
    if kind == "learn":
        return dict(kind=kind, points=_log(rng, 98, 9200))
    if kind == "tubes":
        ns = rng.randint(40, 120)
        return dict(kind=kind, count=rng.randint(2, 4), ns_f=ns, nth_f=10, ns_q=4 * ns + 1, nth_q=20)
    if kind == "channel":
        return dict(kind=kind, cells=rng.randint(2, 7), wall=rng.randint(24, 80))
    return dict(kind=kind, count=rng.randint(8, 32), first=rng.randint(0, 96))


# ---- inputs -------------------------------------------------------------------


def _channel(case, seed):
    w = int(case["wall"])
    return geo.sperm_channel_config(count=int(case["cells"]), seed=seed,
                                    wall_f=(w, max(6, w * 21 // 90), max(3, w * 10 // 90)),
                                    wall_q=(w * 31 // 10, max(18, w * 70 // 90), max(9, w * 30 // 90)))


def _tubes(case, seed):
    grid = [int(case[k]) for k in ("ns_f", "nth_f", "ns_q", "nth_q")]
    if case.get("count", 1) == 1:
        return geo.swimmer_config(*grid)
    return geo.swimmers_config(int(case["count"]), *grid, seed=seed)


def _rotation(axis, angle):
    a = np.asarray(axis, float) / np.linalg.norm(axis)
    K = np.array([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]])
    return np.eye(3) + math.sin(angle) * K + (1.0 - math.cos(angle)) * (K @ K)


def _problems(case, seed):
    """The case's problems, each with its state, its loads and a start time."""
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    if kind == "resistance":
        prs = [geo.sphere_cells_config(int(case["cells_f"]), int(case["cells_q"]))]
    elif kind in ("nearest", "velocity", "channel"):
        prs = [_channel(case, seed)]
    elif kind == "batch":
        prs = [geo.node_config(int(case["first"]) + i, cilia=(4, 12), floor=(160, 500), n_rod=10,
                               q_rod=100, n_sphere=2, q_sphere=8) for i in range(int(case["count"]))]
    else:
        prs = [_tubes(case, seed)]
    out = []
    for pr in prs:
        Y = geo.initial_state(pr)
        for i, body in enumerate(pr.bodies):
            if body.kind == geo.PRESCRIBED and kind == "resistance":
                Y["x0"][i] = rng.uniform(-1.0, 1.0, 3)
                Y["B"][i] = _rotation(rng.normal(size=3), rng.uniform(0.0, 3.0))
            elif body.kind == geo.PRESCRIBED:
                Y["B"][i] = _rotation(body.Omega, rng.uniform(0.0, 2.0 * math.pi)) @ Y["B"][i]
            elif body.kind == geo.FREE and kind == "batch":
                Y["x0"][i] += rng.uniform(-0.02, 0.02, 3)
            elif body.kind == geo.FREE and kind != "channel":
                Y["B"][i] = _rotation(rng.normal(size=3), rng.uniform(0.0, 0.1)) @ Y["B"][i]
        ext = None
        if kind == "batch":  # sinking spheres
            ext = np.zeros((pr.n_free, 6))
            ext[:, 2] = -rng.uniform(0.1, 1.0, pr.n_free)
        out.append((pr, Y, ext, float(rng.uniform(0.0, 1.0))))
    return out


def _host_shapes(pr, t):
    s = geo.pack_shapes(pr, t)
    return tuple(s[k] for k in ("x", "Xw", "xidot"))


def _device_shapes(pr, t):
    return tuple(torch.from_numpy(a).cuda() for a in _host_shapes(pr, t))


def _rigid_motions(xi, Y):
    """Velocities of the force points for the six unit rigid motions, (6, 3N)."""
    B = torch.as_tensor(Y["B"][0], device=xi.device)
    r = xi[:, :3] @ B.T
    e = torch.eye(3, dtype=torch.float64, device=xi.device)
    rows = [e[c].expand(r.shape).reshape(-1) for c in range(3)]
    rows += [torch.linalg.cross(e[c].expand(r.shape), r).reshape(-1) for c in range(3)]
    return torch.stack(rows).contiguous()


# a factor serves six stages at most: one factorisation in three time steps
REUSE_CHANNEL = dict(reuse_factor=True, warm_start=True, reuse_max_inner=40, reuse_max_stages=5,
                     inner_tol=1e-5, arnoldi="df")
REUSE_TUBES = dict(inner_tol=1e-6, max_inner=64, max_outer=20, reuse_factor=True, warm_start=True,
                   reuse_max_inner=60, reuse_max_stages=32, arnoldi="df")


def _tracers(points, seed):
    rng = np.random.default_rng(seed)
    xp = np.zeros((points, 4))
    xp[:, :3] = rng.uniform([0.1, 0.1, 0.05], [3.9, 0.9, 0.45], size=(points, 3))
    return torch.from_numpy(xp).cuda()


def _density(N, seed):
    rng = np.random.default_rng(seed + 1)
    return torch.from_numpy(rng.normal(size=3 * N)).cuda()


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "learn":
        points = int(case["points"])
        # any problem with that many force points carries the network
        ctx = nrs.Context([0, points], [0, 2 * points], [nrs.PRESCRIBED], 0.01)
        ctx.mlp_set_params(mlp_inputs.mlp_perturb(seed, mlp_inputs.mlp_init(seed), 0.05))
        X, T = mlp_inputs.mlp_batch(seed, points)
        st.update(ctx=ctx, X=torch.from_numpy(X).cuda(), T=torch.from_numpy(T).cuda())
        return st
    problems = _problems(case, seed)
    pr, Y, ext, t0 = problems[0]
    if kind == "batch":
        batch = nrs.Batch([p[0] for p in problems], factor_prec="tf32")
        pairs, sols = [], []
        for c, (p, y, e, t) in zip(batch.contexts, problems):
            c.set_state(y["x0"], y["B"])
            c.set_external(e)
            pairs.append((_device_shapes(p, t), _device_shapes(p, t + 0.5 * DT)))
            sols.append(torch.empty(2 * p.n, dtype=torch.float64, device="cuda"))
        st.update(batch=batch, pairs=pairs, sols=sols)
        return st
    options = {"resistance": dict(factor_prec=case.get("prec", "tf32")),
               "solve": dict(factor_prec=case.get("prec", "tf32")),
               "replay": dict(factor_prec="tf32", graph=True),
               "tubes": dict(factor_prec="tf32", **REUSE_TUBES),
               "channel": dict(factor_prec="tf32", **REUSE_CHANNEL)}.get(kind, dict(factor_prec="tf32"))
    if kind == "nearest":
        xi, Xiw, xidot = _device_shapes(pr, t0)
        n_off = np.cumsum([0] + [b.N for b in pr.bodies])
        q_off = np.cumsum([0] + [b.Q for b in pr.bodies])
        if case["scope"] == "global":
            pr.nn_global = True
        st.update(scope=case["scope"], n_off=n_off, q_off=q_off)
    ctx = nrs.Context.from_problem(pr, **options)
    ctx.set_state(Y["x0"], Y["B"])
    st.update(ctx=ctx, Y=Y)
    if kind == "nearest":
        st["x"], st["Xw"] = xi, Xiw
        if case["scope"] == "global":
            st["x"], st["Xw"], _ = ctx.kinematics(xi, Xiw, xidot)
        return st
    if kind in ("replay", "tubes", "channel"):
        steps = 3 if kind == "channel" else 1
        st["shapes"] = []
        for s in range(steps):
            pair = [_device_shapes(pr, t0 + (s + h) * DT) for h in (0.0, 0.5)]
            st["shapes"].append(tuple(nrs.Context.shapes(*p) for p in pair))
        st["sol"] = [torch.empty(2 * pr.n, dtype=torch.float64, device="cuda") for _ in range(steps)]
        return st
    st["shapes"] = _device_shapes(pr, t0)
    if kind == "resistance":
        st["b"] = _rigid_motions(st["shapes"][0], Y)
        st["prec"] = case["prec"]
    if kind in ("solve", "velocity"):
        x, st["Xw"], st["b"] = ctx.kinematics(*st["shapes"])
        ctx.nearest_build(*st["shapes"][:2])
    if kind == "solve":
        ctx.assemble(x, st["Xw"], want_matrix=False)
        st["prec"] = case["prec"]
    if kind == "velocity":
        st["xp"] = _tracers(int(case["points"]), seed)
        st["f"] = _density(pr.N, seed)
    return st


# ---- one pass -------------------------------------------------------------------


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["batch"].step(state["pairs"], DT, sols=state["sols"])
        return state["sols"]
    ctx = state["ctx"]
    if kind == "learn":
        out, grad, _ = ctx.mlp_eval(state["X"], state["T"], grad=True)
        ctx.mlp_adam(grad, 1e-3)
        return out, grad
    if kind == "nearest":
        if state["scope"] == "static":
            return nrs.nearest_build_static(state["x"], state["Xw"], state["n_off"], state["q_off"])
        return ctx.nearest_build(state["x"], state["Xw"])
    if kind == "velocity":
        return ctx.velocity(state["xp"], state["f"], state["Xw"])
    if kind == "solve":
        ctx.factor(state["prec"])
        return ctx.solve(state["b"])[0]
    if kind == "replay":
        s0, sh = state["shapes"][0]
        ctx.step(s0, sh, DT, sol=state["sol"][0], report=False)
        return state["sol"][0], ctx.get_state()
    if kind in ("tubes", "channel"):
        ctx.set_state(state["Y"]["x0"], state["Y"]["B"])
        for (s0, sh), sol in zip(state["shapes"], state["sol"]):
            ctx.step(s0, sh, DT, sol=sol, report=False)
        return state["sol"], ctx.get_state()
    xi, Xiw, xidot = state["shapes"]
    x, Xw, b = ctx.kinematics(xi, Xiw, xidot)
    nn, _, _ = ctx.nearest_build(xi, Xiw)
    if kind == "matrix":
        return ctx.assemble(x, Xw), b, nn
    ctx.assemble(x, Xw, want_matrix=False)
    ctx.factor(state["prec"])
    return ctx.solve(state["b"])[0]


# ---- what a pass cannot do without ------------------------------------------------


def work(case):
    """Bytes: inputs read once, outputs written once.  Flops: 40 per
    (force point, quadrature point) pair of the matrix, 2/3 n^3 per
    factorisation, 2 n^2 per right-hand side."""
    kind = case["kind"]
    if kind == "learn":
        p = int(case["points"])
        weights = 64 * 17 + 64 * 64 + 3 * 64
        return {"bytes": 4 * p * (17 + 3 + 3) + 24 * mlp_inputs.NPARAM, "flops": 6 * p * weights}
    bytes_, flops = 0.0, 0.0
    for pr, _, _, _ in _problems(case, 0):
        N, Q, n = pr.N, pr.Q, pr.n
        cloud, pairs, factor = 32 * (2 * N + Q), 40.0 * N * Q, 2.0 / 3.0 * n ** 3
        if kind == "resistance":
            bytes_ += cloud + 12 * 8 * n
            flops += pairs + factor + 12 * n * n
        elif kind == "matrix":
            bytes_ += cloud + 8 * n * n + 8 * n + 4 * Q
            flops += pairs
        elif kind == "solve":
            bytes_ += 8 * n * n + 16 * n
            flops += factor + 2 * n * n
        elif kind == "nearest":
            per_body = sum(b.N * b.Q for b in pr.bodies)
            bytes_ += 32 * (N + Q) + 4 * (2 * Q + N)
            flops += 8.0 * (N * Q if case["scope"] == "global" else per_body)
        elif kind == "velocity":
            p = int(case["points"])
            bytes_ += 32 * Q + 24 * N + 64 * p
            flops += 40.0 * p * Q
        else:
            steps = 3 if kind == "channel" else 1
            bytes_ += steps * (2 * cloud + 16 * n)
            # with factor reuse one factorisation serves the pass
            factors = 1.0 if kind in ("channel", "tubes") else 2.0
            flops += steps * (2 * pairs + 4 * n * n) + factors * factor
    return {"bytes": bytes_, "flops": flops}


# ---- the same values in 64 bits ---------------------------------------------------

ROWS = 1 << 22  # pairs evaluated at a time


def _body_of(sizes):
    return torch.repeat_interleave(torch.arange(len(sizes)), torch.tensor(sizes)).cuda()


def _nearest(xi, Xi, bx, bX):
    step = max(1, ROWS // len(xi))
    out = []
    for q in range(0, len(Xi), step):
        d = Xi[q:q + step, None, :] - xi[None, :, :]
        d2 = d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1] + d[..., 2] * d[..., 2]
        d2 = torch.where(bX[q:q + step, None] == bx[None, :], d2, torch.inf)
        first = d2 == d2.min(dim=1, keepdim=True).values
        out.append(first.to(torch.int8).argmax(dim=1))
    return torch.cat(out)


def _stokeslet_terms(x, X, w, eps, mu):
    """S_jk(x_m - X_q) w_q / (8 pi mu) for j <= k, one (points, Q) array each."""
    r = [x[:, None, k] - X[None, :, k] for k in range(3)]
    r2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2]
    rho = r2 + eps * eps
    s = w[None, :] / (rho * torch.sqrt(rho)) / (8.0 * math.pi * mu)
    for j in range(3):
        for k in range(j, 3):
            v = r[j] * r[k] * s
            yield j, k, v + (r2 + 2.0 * eps * eps) * s if j == k else v


def _lab(pr, Y, host):
    xi, Xiw, xidot = (torch.from_numpy(a).cuda() for a in host)
    bx, bX = _body_of([b.N for b in pr.bodies]), _body_of([b.Q for b in pr.bodies])
    x0 = torch.as_tensor(Y["x0"]).cuda()
    B = torch.as_tensor(Y["B"]).cuda()
    x = x0[bx] + (B[bx] @ xi[:, :3, None])[..., 0]
    X = x0[bX] + (B[bX] @ Xiw[:, :3, None])[..., 0]
    v = (B[bx] @ xidot[:, :3, None])[..., 0]
    nn = _nearest(xi[:, :3], Xiw[:, :3], bx, bX)
    return x, X, Xiw[:, 3], v, nn, bx, bX, x0


def _cross_matrix(r):
    z = torch.zeros_like(r[..., 0])
    return torch.stack([torch.stack([z, -r[..., 2], r[..., 1]], -1),
                        torch.stack([r[..., 2], z, -r[..., 0]], -1),
                        torch.stack([-r[..., 1], r[..., 0], z], -1)], -2)


def _system(pr, Y, ext, host):
    """Matrix, right-hand side and nearest-neighbour map of one stage."""
    x, X, w, v, nn, bx, bX, x0 = _lab(pr, Y, host)
    N, n = pr.N, pr.n
    A = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    step = max(1, ROWS // pr.Q)
    for m in range(0, N, step):
        e = min(N, m + step)
        for j, k, val in _stokeslet_terms(x[m:e], X, w, pr.eps, pr.mu):
            blk = torch.zeros((e - m, N), dtype=torch.float64, device="cuda").index_add_(1, nn, val)
            A[3 * m + j:3 * e + j:3, k:3 * N:3] = blk
            if j != k:
                A[3 * m + k:3 * e + k:3, j:3 * N:3] = blk
    b = torch.zeros(n, dtype=torch.float64, device="cuda")
    W = torch.zeros(N, dtype=torch.float64, device="cuda").index_add_(0, nn, w)
    R = torch.zeros((N, 3), dtype=torch.float64, device="cuda").index_add_(
        0, nn, w[:, None] * (X - x0[bX]))
    free = 0
    for i, body in enumerate(pr.bodies):
        own = torch.nonzero(bx == i)[:, 0]
        r = x[own] - x0[i]
        vb = v[own]
        if body.kind == geo.PRESCRIBED:
            Om = torch.as_tensor(body.Omega, dtype=torch.float64, device="cuda")
            vb = vb + torch.as_tensor(body.U, dtype=torch.float64, device="cuda") \
                + torch.linalg.cross(Om.expand(r.shape), r)
        elif body.kind == geo.STATIC:
            vb = torch.zeros_like(vb)
        lo, hi = 3 * int(own[0]), 3 * int(own[-1]) + 3
        b[lo:hi] = vb.reshape(-1)
        if body.kind == geo.FREE:
            c = 3 * N + 6 * free
            eye = torch.eye(3, dtype=torch.float64, device="cuda").expand(len(own), 3, 3)
            A[lo:hi, c:c + 3] = -eye.reshape(-1, 3)
            A[lo:hi, c + 3:c + 6] = _cross_matrix(r).reshape(-1, 3)
            A[c:c + 3, lo:hi] = (W[own, None, None] * eye).permute(1, 0, 2).reshape(3, -1)
            A[c + 3:c + 6, lo:hi] = _cross_matrix(R[own]).permute(1, 0, 2).reshape(3, -1)
            if ext is not None:
                b[c:c + 6] = torch.as_tensor(ext[free], device="cuda")
            free += 1
    return A, b, nn


def _refined(A, b):
    """A x = b (b with columns) by LU and a few steps of refinement."""
    LU, piv = torch.linalg.lu_factor(A)
    x = torch.linalg.lu_solve(LU, piv, b)
    for _ in range(3):
        x = x + torch.linalg.lu_solve(LU, piv, b - A @ x)
    return x


def _orthonormal(B):
    Q = np.array(B)
    for j in range(3):
        for i in range(j):
            Q[:, j] -= (Q[:, i] @ Q[:, j]) * Q[:, i]
        Q[:, j] /= math.sqrt(Q[:, j] @ Q[:, j])
    return Q


def _moved(pr, Y0, Y, sol, h):
    """Y0 + h dY/dt at the state Y with the solution's rigid velocities."""
    x0, B = Y0["x0"].copy(), Y0["B"].copy()
    free = 0
    for i, body in enumerate(pr.bodies):
        if body.kind == geo.STATIC:
            continue
        U, Om = body.U, body.Omega
        if body.kind == geo.FREE:
            c = 3 * pr.N + 6 * free
            U, Om = sol[c:c + 3], sol[c + 3:c + 6]
            free += 1
        x0[i] = Y0["x0"][i] + h * U
        K = np.array([[0, -Om[2], Om[1]], [Om[2], 0, -Om[0]], [-Om[1], Om[0], 0]])
        B[i] = _orthonormal(Y0["B"][i] + h * (K @ Y["B"][i]))
    return {"x0": x0, "B": B}


def _step(pr, Y, ext, t):
    sols, Yh = [], Y
    for stage in range(2):
        A, b, _ = _system(pr, Yh, ext, _host_shapes(pr, t + 0.5 * DT * stage))
        x = _refined(A, b[:, None])[:, 0]
        sols.append(x)
        Yh = _moved(pr, Y, Yh, x.cpu().numpy(), DT * (stage + 1) / 2.0)
    return torch.cat(sols), Yh


def exact(case, seed):
    kind = case["kind"]
    if kind in ("nearest", "tubes", "channel"):
        return None  # whole numbers, or dense systems too large for 64 bits here
    if kind == "learn":
        p = mlp_inputs.mlp_perturb(seed, mlp_inputs.mlp_init(seed), 0.05)
        X, T = (torch.from_numpy(a).cuda().double() for a in mlp_inputs.mlp_batch(seed, int(case["points"])))
        p = torch.from_numpy(p).cuda().double().requires_grad_(True)
        at, parts = 0, []
        for shape in ((64, 17), (64,), (64, 64), (64,), (3, 64), (3,)):
            size = math.prod(shape)
            parts.append(p[at:at + size].view(shape))
            at += size
        W1, b1, W2, b2, W3, b3 = parts
        silu = torch.nn.functional.silu
        out = silu(silu(X @ W1.T + b1) @ W2.T + b2) @ W3.T + b3
        torch.mean((out - T) ** 2).backward()
        return out.detach(), p.grad
    problems = _problems(case, seed)
    pr, Y, ext, t0 = problems[0]
    if kind == "batch":
        return [_step(p, y, e, t)[0] for p, y, e, t in problems]
    if kind == "replay":
        sol, Yn = _step(pr, Y, ext, t0)
        return sol, Yn
    host = _host_shapes(pr, t0)
    if kind == "velocity":
        _, X, w, _, nn, _, _, _ = _lab(pr, Y, host)
        f = _density(pr.N, seed).view(-1, 3)[nn]
        xp = _tracers(int(case["points"]), seed)
        u = torch.zeros_like(xp)
        step = max(1, ROWS // pr.Q)
        for m in range(0, len(xp), step):
            for j, k, val in _stokeslet_terms(xp[m:m + step, :3], X, w, pr.eps, pr.mu):
                u[m:m + step, j] += val @ f[:, k]
                if j != k:
                    u[m:m + step, k] += val @ f[:, j]
        return u
    A, b, nn = _system(pr, Y, ext, host)
    if kind == "matrix":
        return A.T.contiguous(), b, None
    if kind == "resistance":
        rhs = _rigid_motions(torch.from_numpy(host[0]).cuda(), Y)
        return _refined(A, rhs.T.contiguous()).T.contiguous()
    return _refined(A, b[:, None])[:, 0]
