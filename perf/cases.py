"""Performance cases of the damped least-squares solves, through the library's public entry points.

Each case is one call sequence that a user of the library makes: the batched block solve, Moré's
two factorizations, the composed factor + solve of [blkdiag(J_i) | S] with a dense S (generic
horizontal concatenations, ellipse fits, bundle adjustment), banded instances and
Levenberg-Marquardt iterations of the curve-fit model.  Inputs are drawn on the GPU from the seed
alone; sizes are those of the workloads, tests and benchmark of this repository.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1802_03773_gb300 import Context, qrkit

DEV = torch.device("cuda", 0)
F64 = torch.float64


def listed():
    return [
        # a caller's small batch of uneven blocks: launch latency counts
        dict(name="blocks_500", kind="blocks", precision="fp32_refined", blocks=500, lam=0.0),
        # the benchmark's headline: one million uneven blocks, float with refinement
        dict(name="blocks_1m", kind="blocks", precision="fp32_refined", blocks=1_000_000, lam=0.0),
        # the two factorizations of Moré's LM step (J = QR, then [R; lambda^(1/2) D]) per block
        dict(name="more_250k", kind="blocks", precision="fp32", blocks=250_000, lam=1e-2),
        # the smallest horizontal concatenation of the benchmark, all in double
        dict(name="hcat_fp64_200", kind="hcat", precision="fp64", blocks=200, rows=4, cols=2, shared=30, lam=1e-2),
        # one LM step of an ellipse fit (2 x 1 blocks and five shared parameters), in double
        dict(name="ellipse_100k", kind="ellipse", precision="fp64", blocks=100_000, lam=1e-3),
        # a dense shared block of 128 columns below 100,000 blocks, float with one refinement step
        dict(name="hcat_s128", kind="hcat", precision="fp32_refined", blocks=100_000, rows=4, cols=2, shared=128,
             lam=1e-2),
        # the widest shared block the float path takes
        dict(name="hcat_s512", kind="hcat", precision="fp32_refined", blocks=100_000, rows=4, cols=2, shared=512,
             lam=1e-2),
        # one LM step of a bundle adjustment: 100,000 points seen by 2 to 6 of 14 cameras
        dict(name="ba_14_cameras", kind="ba", precision="fp32_refined", blocks=100_000, cameras=14, lam=1e-3),
        # one banded system of a million columns
        dict(name="banded_1e6", kind="banded", precision="fp32_refined", instances=1, cols_lo=1_000_000,
             cols_hi=1_000_000, lam=1e-3),
        # a batch of independent banded systems of uneven sizes
        dict(name="banded_batch", kind="banded", precision="fp32_refined", instances=256, cols_lo=1000, cols_hi=100_000,
             lam=1e-3),
        # a few LM iterations of one large curve fit, as the graph-replayed loop runs them
        dict(name="lm_fit_200k", kind="lm", precision="fp32_refined", problems=1, points_lo=200_000,
             points_hi=200_000, control_lo=2048, control_hi=2048, iterations=3),
        # one LM iteration of a thousand curve fits at once
        dict(name="lm_batch_1024", kind="lm", precision="fp32_refined", problems=1024, points_lo=500,
             points_hi=20_000, control_lo=16, control_hi=256, iterations=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["blocks", "blocks", "more", "hcat", "hcat", "hcat64", "ellipse", "ba", "banded", "banded", "lm",
                       "lm"])
    if kind == "blocks":
        return dict(kind="blocks", precision=rng.choice(["fp32_refined", "fp32_refined", "fp64"]),
                    blocks=_log_int(rng, 64, 1_000_000), lam=0.0)
    if kind == "more":
        return dict(kind="blocks", precision="fp32", blocks=_log_int(rng, 1000, 1_000_000),
                    lam=10.0 ** rng.uniform(-3.0, 0.0))
    if kind == "hcat":
        s = rng.choice([rng.randint(3, 64), 32 * rng.randint(2, 16), 32 * rng.randint(2, 16)])
        m = rng.randint(1, 3)
        n = rng.randint(m + 1, 6)
        most = min(100_000, int(4e5 * 512.0 / (n * s)), int(4e5 * 512.0 ** 2 / (n * s * s)))
        return dict(kind="hcat", precision="fp32_refined", blocks=_log_int(rng, 400, most), rows=n, cols=m, shared=s,
                    lam=1e-2)
    if kind == "hcat64":
        m = rng.randint(1, 3)
        return dict(kind="hcat", precision="fp64", blocks=_log_int(rng, 100, 20_000), rows=rng.randint(m + 1, 6),
                    cols=m, shared=rng.randint(3, 64), lam=1e-2)
    if kind == "ellipse":
        return dict(kind="ellipse", precision="fp64", blocks=_log_int(rng, 500, 500_000), lam=1e-3)
    if kind == "ba":
        return dict(kind="ba", precision="fp32_refined", blocks=_log_int(rng, 500, 100_000),
                    cameras=rng.randint(7, 30), lam=1e-3)
    if kind == "banded":
        count = _log_int(rng, 1, 256)
        hi = _log_int(rng, 1000, 1_000_000 if count < 13 else 13_000_000 // count)
        return dict(kind="banded", precision="fp32_refined", instances=count, cols_lo=max(500, hi // 20), cols_hi=hi,
                    lam=1e-3)
    count = _log_int(rng, 1, 1024)
    hi = _log_int(rng, 2000, 200_000 if count < 50 else 10_000_000 // count)
    kc = max(16, min(2048, hi // 40))
    return dict(kind="lm", precision="fp32_refined", problems=count, points_lo=max(500, hi // 4), points_hi=hi,
                control_lo=max(8, kc // 4), control_hi=kc, iterations=rng.randint(1, 3))


# ---- inputs (what a user's program has in hand before the call) ----

def _gens(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(20180209 + 1000003 * seed)
    return np.random.default_rng([20180209, seed]), g


def _shapes():
    """The generator of uneven sizes: a case's structure is the same for every seed, only its values are new."""
    return np.random.default_rng(20180209)


def _dtype(case):
    return F64 if case["precision"] == "fp64" else torch.float32


def _offsets(counts):
    return np.concatenate([[0], np.cumsum(counts, dtype=np.int64)])


def _padded(n, m):
    """Index maps of packed column-major blocks padded to (max n, max m): value and row positions and their masks."""
    n, m = torch.as_tensor(n, dtype=torch.int64, device=DEV), torch.as_tensor(m, dtype=torch.int64, device=DEV)
    nm = n * m
    v0, r0 = nm.cumsum(0) - nm, n.cumsum(0) - n
    r, j = torch.arange(int(n.max()), device=DEV), torch.arange(int(m.max()), device=DEV)
    val = v0[:, None, None] + j[None, None, :] * n[:, None, None] + r[None, :, None]
    vmask = (r[None, :, None] < n[:, None, None]) & (j[None, None, :] < m[:, None, None])
    row = r0[:, None] + r[None, :]
    return val, vmask, row, r[None, :] < n[:, None], j[None, :] < m[:, None]


def _block_inputs(case, seed):
    """n ~ U{2..16}, m ~ U{1..min(n, 6)}, N(0, 1) values."""
    h, (_, g) = _shapes(), _gens(case, seed)
    K, dt = case["blocks"], _dtype(case)
    n = h.integers(2, 17, size=K)
    m = 1 + (h.random(K) * np.minimum(n, 6)).astype(np.int64)
    J = torch.randn(int((n * m).sum()), generator=g, device=DEV, dtype=dt)
    b = torch.randn(int(n.sum()), generator=g, device=DEV, dtype=dt)
    return n, m, J, b


def _hcat_inputs(case, seed):
    """K blocks n x m and a dense S (column-major), N(0, 1), columns scaled over two decades."""
    _, g = _gens(case, seed)
    K, n, m, s, dt = case["blocks"], case["rows"], case["cols"], case["shared"], _dtype(case)
    N = K * m + s
    scale = 10.0 ** (2.0 * torch.arange(N, device=DEV, dtype=F64) / (N - 1))
    J = (torch.randn((K, m, n), generator=g, device=DEV, dtype=dt) * scale[:K * m].reshape(K, m, 1)).to(dt).reshape(-1)
    S = torch.randn((s, K * n), generator=g, device=DEV, dtype=dt)
    S *= scale[K * m:, None].to(dt)
    b = torch.randn(K * n, generator=g, device=DEV, dtype=dt)
    return np.full(K, n), np.full(K, m), J, S, b


def _ellipse_inputs(case, seed):
    """The linear system of one LM step of an ellipse fit at a perturbed start."""
    h, g = _gens(case, seed)
    K, dt = case["blocks"], _dtype(case)
    true = np.array([0.5 * h.standard_normal(), 0.5 * h.standard_normal(), 1.5 + h.random(), 0.0, math.pi * h.random()])
    true[3] = true[2] * (0.3 + 0.5 * h.random())
    at = true + 0.02 * h.standard_normal(5)
    t = 2.0 * math.pi * torch.rand(K, generator=g, device=DEV, dtype=F64)
    t0 = t + 0.05 * torch.randn(K, generator=g, device=DEV, dtype=F64)

    def curve(t, x):
        c, s = math.cos(x[4]), math.sin(x[4])
        u, v = x[2] * torch.cos(t), x[3] * torch.sin(t)
        return torch.stack([x[0] + c * u - s * v, x[1] + s * u + c * v], 1)

    y = curve(t, true) + 0.01 * torch.randn((K, 2), generator=g, device=DEV, dtype=F64)
    c, s = math.cos(at[4]), math.sin(at[4])
    ct, st = torch.cos(t0), torch.sin(t0)
    u, v, du, dv = at[2] * ct, at[3] * st, -at[2] * st, at[3] * ct
    J = torch.stack([c * du - s * dv, s * du + c * dv], 1).reshape(-1)
    one, zero = torch.ones_like(t0), torch.zeros_like(t0)
    S = torch.stack([torch.stack([one, zero], 1), torch.stack([zero, one], 1), torch.stack([c * ct, s * ct], 1),
                     torch.stack([-s * st, c * st], 1), torch.stack([-s * u - c * v, c * u - s * v], 1)])
    b = (y - curve(t0, at)).reshape(-1)
    return np.full(K, 2), np.full(K, 1), J.to(dt), S.reshape(5, -1).to(dt).contiguous(), b.to(dt)


def _rotate(w, X):
    th = w.norm(dim=-1, keepdim=True)
    k = w / th.clamp_min(1e-300)
    return X * th.cos() + torch.linalg.cross(k, X) * th.sin() + k * (k * X).sum(-1, keepdim=True) * (1 - th.cos())


def _project(cam, X):
    """Angle-axis, translation, focal length and two radial terms per camera."""
    Xc = _rotate(cam[:, :3], X) + cam[:, 3:6]
    q = -Xc[:, :2] / Xc[:, 2:3]
    r2 = (q * q).sum(-1, keepdim=True)
    return cam[:, 6:7] * (1.0 + cam[:, 7:8] * r2 + cam[:, 8:9] * r2 * r2) * q


def _ba_inputs(case, seed):
    """The linear system of one LM step of a bundle adjustment: cameras on a circle around a ball of points."""
    h, g = _gens(case, seed)
    P, C, dt = case["blocks"], case["cameras"], _dtype(case)
    rn = lambda *size: torch.randn(size, generator=g, device=DEV, dtype=F64)  # noqa: E731
    X = rn(P, 3)
    X *= torch.rand((P, 1), generator=g, device=DEV, dtype=F64) ** (1.0 / 3.0) / X.norm(dim=1, keepdim=True)
    cams = np.zeros((C, 9))
    for c, th in enumerate(2.0 * np.pi * (np.arange(C) + 0.5 * h.random(C)) / C):
        centre = 4.0 * np.array([math.sin(th), 0.2 * h.standard_normal(), math.cos(th)])
        z = centre / np.linalg.norm(centre)
        x = np.cross([0.0, 1.0, 0.0], z)
        x /= np.linalg.norm(x)
        R = np.stack([x, np.cross(z, x), z])
        ang = math.acos(min(1.0, max(-1.0, (np.trace(R) - 1.0) / 2.0)))
        axis = np.array([R[2, 1] - R[1, 2], R[0, 2] - R[2, 0], R[1, 0] - R[0, 1]])
        cams[c, :3] = ang * axis / max(np.linalg.norm(axis), 1e-12)
        cams[c, 3:6] = -R @ centre
    cams[:, 6] = 500.0 + 300.0 * h.random(C)
    cams[:, 7:9] = h.standard_normal((C, 2)) * [0.05, 0.01]
    near = cams.copy()
    near[:, :3] += 0.001 * h.standard_normal((C, 3))
    near[:, 3:6] += 0.01 * h.standard_normal((C, 3))
    near[:, 6] *= 1.0 + 0.005 * h.standard_normal(C)
    near[:, 7:9] += 0.001 * h.standard_normal((C, 2))
    k = h.integers(2, 7, size=P)
    seen = torch.rand((P, C), generator=g, device=DEV).argsort(1)[:, :6]
    kd = torch.as_tensor(k, device=DEV)
    seen = torch.where(torch.arange(6, device=DEV)[None, :] < kd[:, None], seen, C).sort(1).values
    cam = seen[seen < C]
    point = torch.arange(P, device=DEV).repeat_interleave(kd)
    true, at = torch.as_tensor(cams, device=DEV), torch.as_tensor(near, device=DEV)
    obs = _project(true[cam], X[point]) + 0.5 * rn(cam.numel(), 2)
    X0 = X + 0.01 * rn(P, 3)
    ca, xa = at[cam], X0[point]
    b = (obs - _project(ca, xa)).reshape(-1)
    Jp, Jc = torch.empty((cam.numel(), 2, 3), device=DEV, dtype=F64), torch.empty((cam.numel(), 2, 9), device=DEV, dtype=F64)
    for j in range(3):
        d = torch.zeros(3, device=DEV, dtype=F64)
        d[j] = 1e-6
        Jp[:, :, j] = (_project(ca, xa + d) - _project(ca, xa - d)) / 2e-6
    for j in range(9):
        d = torch.zeros(9, device=DEV, dtype=F64)
        d[j] = 1e-6 * max(1.0, float(at[:, j].abs().max()))
        Jc[:, :, j] = (_project(ca + d, xa) - _project(ca - d, xa)) / (2.0 * float(d[j]))
    n, m = 2 * k, np.full(P, 3)
    val, vmask, row, rmask, _ = _padded(n, m)
    J = torch.empty(int((n * m).sum()), device=DEV, dtype=dt)
    rows = Jp.reshape(-1, 3)
    J[val[vmask]] = rows[row.clamp_max(rows.shape[0] - 1)][vmask].to(dt)
    s = (9 * C + 31) // 32 * 32
    S = torch.zeros((s, rows.shape[0]), device=DEV, dtype=dt)
    cols = (9 * cam[:, None] + torch.arange(9, device=DEV)[None, :]).repeat_interleave(2, 0)
    S[cols, torch.arange(rows.shape[0], device=DEV)[:, None]] = Jc.reshape(-1, 9).to(dt)
    return n, m, J, S, b.to(dt)


def _banded_inputs(case, seed):
    """Four rows per column, eight values per row, N(0, 1); entries past an instance's last column are zero."""
    h, (_, g) = _shapes(), _gens(case, seed)
    cols = h.integers(case["cols_lo"], case["cols_hi"] + 1, size=case["instances"])
    M, dt = 4 * int(cols.sum()), _dtype(case)
    J = torch.randn((M, 8), generator=g, device=DEV, dtype=dt)
    b = torch.randn(M, generator=g, device=DEV, dtype=dt)
    ends = torch.as_tensor(4 * np.cumsum(cols), device=DEV)
    for t in range(1, 8):   # entry t of the last t columns' rows
        J[(ends[:, None] - 1 - torch.arange(4 * t, device=DEV)[None, :]).reshape(-1), t] = 0
    return cols, J, b


def _spline(u):
    v = 1.0 - u
    return torch.stack([v ** 3, 3 * u ** 3 - 6 * u ** 2 + 4, -3 * u ** 3 + 3 * u ** 2 + 3 * u + 1, u ** 3], -1) / 6.0


def _dspline(u):
    v = 1.0 - u
    return torch.stack([-3 * v ** 2, 9 * u ** 2 - 12 * u, -9 * u ** 2 + 6 * u + 3, 3 * u ** 2], -1) / 6.0


def _segment(t, kc):
    seg = torch.minimum(t.floor().clamp_min(0), (kc - 4).to(F64))
    return seg.long(), t - seg


def _lm_inputs(case, seed):
    """Points on uniform cubic B-splines with noise, and a perturbed start [t of all points | control points]."""
    h, (_, g) = _shapes(), _gens(case, seed)
    npts = h.integers(case["points_lo"], case["points_hi"] + 1, size=case["problems"])
    kcs = h.integers(case["control_lo"], case["control_hi"] + 1, size=case["problems"])
    kd, nd = torch.as_tensor(kcs, device=DEV), torch.as_tensor(npts, device=DEV)
    ki = torch.arange(int(kcs.sum()), device=DEV) - (kd.cumsum(0) - kd).repeat_interleave(kd)
    th = 2.0 * math.pi * ki / kd.repeat_interleave(kd)
    rad = 1.0 + 0.1 * torch.randn(th.numel(), generator=g, device=DEV, dtype=F64)
    ctrl = torch.stack([th.cos() * rad, th.sin() * rad], 1)
    kp, first = kd.repeat_interleave(nd), (kd.cumsum(0) - kd).repeat_interleave(nd)
    t = torch.rand(kp.numel(), generator=g, device=DEV, dtype=F64) * (kp - 3)
    seg, u = _segment(t, kp)
    B = _spline(u)
    data = 0.01 * torch.randn((t.numel(), 2), generator=g, device=DEV, dtype=F64)
    for q in range(4):
        data += B[:, q:q + 1] * ctrl[first + seg + q]
    t0 = t + 0.05 * torch.randn(t.numel(), generator=g, device=DEV, dtype=F64)
    P0 = ctrl + 0.01 * torch.randn(ctrl.shape, generator=g, device=DEV, dtype=F64)
    return npts, kcs, data, torch.cat([t0, P0.reshape(-1)])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lm":
        npts, kcs, data, x0 = _lm_inputs(case, seed)
        torch.cuda.synchronize()   # the context's stream is its own: the iterations are captured in a graph
        stream = torch.cuda.Stream(DEV)
        ctx = Context(0, stream=stream, precision=case["precision"])
        ctx.lm_plan(npts, kcs, data)
        start = ctx.lm_states(1e-3)
        return dict(case=case, ctx=ctx, stream=stream, x0=x0, x=x0.clone(), start=start, states=ctx.lm_states(1e-3))
    ctx = Context(0, precision=case["precision"])
    if kind == "blocks":
        n, m, J, b = _block_inputs(case, seed)
        ctx.plan_blocks(n, m)
        N, S = int(m.sum()), None
    elif kind == "banded":
        cols, J, b = _banded_inputs(case, seed)
        ctx.plan_banded(cols, rows_per_col=4, window=8)
        N, S = int(cols.sum()), None
    else:
        n, m, J, S, b = {"hcat": _hcat_inputs, "ellipse": _ellipse_inputs, "ba": _ba_inputs}[kind](case, seed)
        ctx.plan_blocks(n, m, qrkit.COUPLED_DENSE, shared_cols=S.shape[0])
        N = int(m.sum()) + S.shape[0]
    return dict(case=case, ctx=ctx, J=J, S=S, b=b, p=torch.empty(N, device=DEV, dtype=_dtype(case)))


def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "lm":
        st, x = state["states"], state["x"]
        ctypes.memmove(st, state["start"], ctypes.sizeof(st))
        with torch.cuda.stream(state["stream"]):
            x.copy_(state["x0"])
        if case["iterations"] == 1:
            ctx.lm_step(x, st, refine_steps=1)
        else:
            ctx.lm_run(x, st, max_iter=case["iterations"], refine_steps=1, use_graph=True)
        # the states' scalars in the precision of the context's arithmetic
        rec = np.frombuffer(st, dtype=_STATE)
        out = {f: rec[f].astype(np.float32) for f in ("lambda", "cost", "cost_new", "pred", "rho")}
        out["accepted"] = rec["accepted"].copy()
        out["x"] = x
        return out
    if case["kind"] == "banded":
        ctx.factor_solve(state["J"], state["b"], state["p"], lam=case["lam"], refine_steps=2)
    elif case["kind"] == "blocks":
        ctx.factor_solve(state["J"], state["b"], state["p"], lam=case["lam"], refine_steps=2)
    else:
        ctx.factor(state["J"], state["S"], lam=case["lam"])
        ctx.solve(state["b"], state["p"], refine_steps=0 if case["precision"] == "fp64" else 1)
    return state["p"]


_STATE = np.dtype([("lambda", "f8"), ("nu", "f8"), ("cost", "f8"), ("cost_new", "f8"), ("pred", "f8"), ("rho", "f8"),
                   ("accepted", "i4"), ("done", "i4"), ("iteration", "i8")])


def work(case):
    """Inputs once, outputs once; Householder QR and the orthogonal applications as operations (means of the draws)."""
    e, kind = (8 if case["precision"] == "fp64" else 4), case["kind"]
    if kind == "blocks":
        K = case["blocks"]
        return dict(bytes=e * K * (30.5 + 9.0 + 3.2), flops=K * 2.0 * (130.0 + 2 * 30.5 + 6.0))
    if kind == "banded":
        N = case["instances"] * (case["cols_lo"] + case["cols_hi"]) / 2.0
        return dict(bytes=e * N * (4 * 9 + 1), flops=N * 2.0 * (4 + 1) * (8 * 8 + 2 * 8))
    if kind == "lm":
        pts = case["problems"] * (case["points_lo"] + case["points_hi"]) / 2.0
        # data (2), the parameter in and out, per iteration; a 2 x 1 block, its window of 8 and the banded rows
        return dict(bytes=case["iterations"] * 8.0 * 4 * pts, flops=case["iterations"] * pts * 2.0 * (60 + 3 * 8 + 2 * 64))
    K = case["blocks"]
    n, m, s = {"hcat": lambda: (case["rows"], case["cols"], case["shared"]), "ellipse": lambda: (2, 1, 5),
               "ba": lambda: (8, 3, (9 * case["cameras"] + 31) // 32 * 32)}[kind]()
    M = K * n + s
    return dict(bytes=float(e) * (K * n * (m + s + 1) + K * m + s),
                flops=K * 4.0 * (n + m) * m * (s + 1) + 2.0 * M * s * s - 2.0 / 3.0 * s ** 3 + 4.0 * M * s)


# ---- what run returns, in 64 bits ----

def _householder(A, cols):
    """The first `cols` reflectors of a stack A (B, r, c) applied to the whole of it, in place."""
    for k in range(cols):
        x = A[:, k:, k]
        norm = x.norm(dim=1)
        v = x.clone()
        v[:, 0] += torch.where(x[:, 0] >= 0, norm, -norm)
        vv = (v * v).sum(1)
        w = torch.einsum("bi,bij->bj", v, A[:, k:, k:]) * (2.0 / torch.where(vv == 0, 1.0, vv))[:, None]
        A[:, k:, k:] -= v[:, :, None] * w[:, None, :]


def _backsub(R, y):
    x = torch.zeros_like(y)
    for k in reversed(range(y.shape[1])):
        x[:, k] = (y[:, k] - (R[:, k, k + 1:y.shape[1]] * x[:, k + 1:]).sum(1)) / R[:, k, k]
    return x


def _exact_blocks(case, seed):
    n, m, J, b = _block_inputs(case, seed)
    out, step, vo, ro = [], 250_000, _offsets(n * m), _offsets(n)
    for k0 in range(0, len(n), step):
        sl = slice(k0, min(k0 + step, len(n)))
        val, vmask, row, rmask, cmask = _padded(n[sl], m[sl])
        Jk, bk = J[vo[k0]:vo[sl.stop]].to(F64), b[ro[k0]:ro[sl.stop]].to(F64)
        K, N, Mc = vmask.shape
        A = torch.zeros((K, N + Mc, Mc + 1), device=DEV, dtype=F64)
        A[:, :N, :Mc] = torch.where(vmask, Jk[torch.where(vmask, val, 0)], 0.0)
        A[:, :N, Mc] = torch.where(rmask, bk[torch.where(rmask, row, 0)], 0.0)
        D = A[:, :N, :Mc].norm(dim=1)
        D = math.sqrt(case["lam"]) * torch.where(D == 0, 1.0, D)
        idx = torch.arange(Mc, device=DEV)
        A[:, N + idx, idx] = torch.where(cmask, D, 1.0)   # unit rows in the columns a block lacks
        _householder(A, Mc)
        out.append(_backsub(A, A[:, :Mc, Mc])[cmask])
    return torch.cat(out)


def _exact_dense(case, seed):
    n, m, J, S, b = {"hcat": _hcat_inputs, "ellipse": _ellipse_inputs, "ba": _ba_inputs}[case["kind"]](case, seed)
    lam, s = case["lam"], S.shape[0]
    val, vmask, row, rmask, _ = _padded(n, m)
    K, N, m = vmask.shape
    A = torch.zeros((K, N + m, m + s + 1), device=DEV, dtype=F64)
    A[:, :N, :m] = torch.where(vmask, J.to(F64)[torch.where(vmask, val, 0)], 0.0)
    row = torch.where(rmask, row, 0)
    for c in range(s):
        A[:, :N, m + c] = torch.where(rmask, S[c].to(F64)[row], 0.0)
    A[:, :N, m + s] = torch.where(rmask, b.to(F64)[row], 0.0)
    D = A[:, :N, :m].norm(dim=1)
    idx = torch.arange(m, device=DEV)
    A[:, N + idx, idx] = math.sqrt(lam) * torch.where(D == 0, 1.0, D)
    DS = torch.stack([S[c].to(F64).norm() for c in range(s)])
    _householder(A, m)
    damp = torch.zeros((s, s + 1), device=DEV, dtype=F64)
    damp[:, :s] = torch.diag(math.sqrt(lam) * torch.where(DS == 0, 1.0, DS))
    rows = torch.cat([A[:, m:, m:].reshape(-1, s + 1), damp])
    while rows.shape[0] > 4 * (s + 1):   # triangles of row chunks, stacked
        chunk = max(4 * (s + 1), 1 << 15)
        rows = torch.cat([torch.linalg.qr(rows[i:i + chunk], mode="r").R for i in range(0, rows.shape[0], chunk)])
    R = torch.linalg.qr(rows, mode="r").R
    xs = torch.linalg.solve_triangular(R[:s, :s], R[:s, s:], upper=True)[:, 0]
    x = _backsub(A[:, :m, :m], A[:, :m, m + s] - A[:, :m, m:m + s] @ xs)
    return torch.cat([x.reshape(-1), xs])


def _gauss(A, B):
    """A^{-1} B for stacks of symmetric positive definite 8 x 8 matrices."""
    W = torch.cat([A, B], 2)
    for k in range(8):
        W[:, k] /= W[:, k, k:k + 1].clone()
        f = W[:, :, k].clone()
        f[:, k] = 0
        W -= f[:, :, None] * W[:, k][:, None, :]
    return W[:, :, 8:]


def _tridiagonal(D, U, f):
    """Block cyclic reduction of a symmetric block tridiagonal system: U[i] couples block i to block i + 1."""
    n = D.shape[0]
    if n == 1:
        return _gauss(D, f[:, :, None])[:, :, 0]
    ne, no = (n + 1) // 2, n // 2
    De, fe = D[0::2].clone(), f[0::2].clone()
    L, R = U[0:2 * no:2].transpose(1, 2), U[1::2]          # odd block's couplings to its left and right
    X = _gauss(D[1::2], torch.cat([L, R, f[1::2][:, :, None]], 2))
    XL, XR, Xf = X[:, :, :8], X[:, :, 8:16], X[:, :, 16]
    De[:no] -= L.transpose(1, 2) @ XL
    fe[:no] -= (L.transpose(1, 2) @ Xf[:, :, None])[:, :, 0]
    k = ne - 1                                              # even blocks that have an odd block to their left
    De[1:] -= R[:k].transpose(1, 2) @ XR[:k]
    fe[1:] -= (R[:k].transpose(1, 2) @ Xf[:k, :, None])[:, :, 0]
    Ue = torch.zeros((ne, 8, 8), device=DEV, dtype=F64)
    Ue[:no] = -L.transpose(1, 2) @ XR
    xe = _tridiagonal(De, Ue, fe)
    x = torch.empty((n, 8), device=DEV, dtype=F64)
    x[0::2] = xe
    nxt = torch.zeros((no, 8), device=DEV, dtype=F64)
    nxt[:k] = xe[1:]
    x[1::2] = Xf - (XL @ xe[:no, :, None])[:, :, 0] - (XR @ nxt[:, :, None])[:, :, 0]
    return x


def _solve_band(band, f):
    """The symmetric banded system with band[i, t] = A[i, i + t], t < 8."""
    n = f.numel()
    P = (n + 7) // 8
    full = torch.zeros((8 * P, 8), device=DEV, dtype=F64)
    full[:n] = band
    full[n:, 0] = 1.0
    rhs = torch.zeros(8 * P, device=DEV, dtype=F64)
    rhs[:n] = f
    full = full.reshape(P, 8, 8)
    D, U = torch.zeros_like(full), torch.zeros_like(full)
    for i in range(8):
        for t in range(8):
            if i + t < 8:
                D[:, i, i + t] = full[:, i, t]
                D[:, i + t, i] = full[:, i, t]
            else:
                U[:, i, i + t - 8] = full[:, i, t]
    return _tridiagonal(D, U, rhs.reshape(P, 8)).reshape(-1)[:n]


def _exact_banded(case, seed):
    cols, J, b = _banded_inputs(case, seed)
    n = int(cols.sum())
    band, f = torch.zeros((n + 8, 8), device=DEV, dtype=F64), torch.zeros(n + 8, device=DEV, dtype=F64)
    step = 1 << 20
    for c0 in range(0, n, step):
        c1 = min(c0 + step, n)
        V = J[4 * c0:4 * c1].to(F64).reshape(c1 - c0, 4, 8)
        G = V.transpose(1, 2) @ V
        g = (V.transpose(1, 2) @ b[4 * c0:4 * c1].to(F64).reshape(-1, 4, 1))[:, :, 0]
        for a in range(8):
            band[c0 + a:c1 + a, :8 - a] += G[:, a, a:]
            f[c0 + a:c1 + a] += g[:, a]
    band, f = band[:n], f[:n]
    band[:, 0] += case["lam"] * torch.where(band[:, 0] == 0, 1.0, band[:, 0])
    return _solve_band(band, f)


def _exact_lm(case, seed):
    npts, kcs, data, x = _lm_inputs(case, seed)
    B, P = len(npts), data.shape[0]
    nd, kd = torch.as_tensor(npts, device=DEV), torch.as_tensor(kcs, device=DEV)
    prob = torch.arange(B, device=DEV).repeat_interleave(nd)
    cprob = torch.arange(B, device=DEV).repeat_interleave(2 * kd)
    kp, first = kd[prob], (kd.cumsum(0) - kd)[prob]
    lam = torch.full((B,), 1e-3, device=DEV, dtype=F64)
    nu = torch.full_like(lam, 2.0)
    done = torch.zeros(B, device=DEV, dtype=torch.bool)
    last = {k: torch.zeros_like(lam) for k in ("cost", "cost_new", "pred", "rho", "accepted")}

    def residual(x):
        seg, u = _segment(x[:P], kp)
        w, ctrl, f = _spline(u), x[P:].reshape(-1, 2), -data
        for q in range(4):
            f = f + w[:, q:q + 1] * ctrl[first + seg + q]
        return f

    def sums(v, index):
        return torch.zeros(B, device=DEV, dtype=F64).index_add_(0, index, v)

    for it in range(case["iterations"]):
        f = residual(x)
        cost = 0.5 * sums((f * f).sum(1), prob)
        seg, u = _segment(x[:P], kp)
        w, dw, ctrl = _spline(u), _dspline(u), x[P:].reshape(-1, 2)
        j = sum(dw[:, q:q + 1] * ctrl[first + seg + q] for q in range(4))
        g0 = 2 * (first + seg)                               # first shared column of a point's window
        jj = (j * j).sum(1)
        dt2 = lam[prob] * torch.where(jj == 0, 1.0, jj)      # lambda D^2 of the point's own column
        n = x.numel() - P
        band, rhs = torch.zeros((n + 8) * 8, device=DEV, dtype=F64), torch.zeros(n + 8, device=DEV, dtype=F64)
        diag, jtb = torch.zeros(n + 8, device=DEV, dtype=F64), torch.zeros(n + 8, device=DEV, dtype=F64)
        jb = -(j * f).sum(1)
        for c0 in range(0, P, 1 << 21):
            c = slice(c0, min(P, c0 + (1 << 21)))
            S = torch.zeros((c.stop - c0, 2, 8), device=DEV, dtype=F64)
            S[:, 0, 0::2] = w[c]
            S[:, 1, 1::2] = w[c]
            Sj = (S * j[c][:, :, None]).sum(1)
            q = jj[c] + dt2[c]
            Sb = -(S * f[c][:, :, None]).sum(1)
            for a in range(8):
                at = g0[c] + a
                diag.index_add_(0, at, (S[:, :, a] ** 2).sum(1))
                jtb.index_add_(0, at, Sb[:, a])
                rhs.index_add_(0, at, Sb[:, a] - Sj[:, a] * jb[c] / q)
                for t in range(8 - a):
                    band.index_add_(0, at * 8 + t, (S[:, :, a] * S[:, :, a + t]).sum(1) - Sj[:, a] * Sj[:, a + t] / q)
        band = band.reshape(-1, 8)[:n]
        dS2 = lam[cprob] * torch.where(diag[:n] == 0, 1.0, diag[:n])
        band[:, 0] += dS2
        pS = _solve_band(band, rhs[:n])
        Sp = sum(w[:, q:q + 1] * pS.reshape(-1, 2)[first + seg + q] for q in range(4))
        pt = (jb - (j * Sp).sum(1)) / (jj + dt2)
        pred = 0.5 * (sums(pt * (dt2 * pt + jb), prob) + sums(pS * (dS2 * pS + jtb[:n]), cprob))
        step = torch.cat([pt, pS])
        fn = residual(x + step)
        cost_new = 0.5 * sums((fn * fn).sum(1), prob)
        rho = torch.where(pred > 0, (cost - cost_new) / pred, -1.0)
        ok = (rho > 0) & ~done
        for k, v in (("cost", cost), ("cost_new", cost_new), ("pred", pred), ("rho", rho), ("accepted", ok.to(F64))):
            last[k] = torch.where(done, last[k], v)
        x = torch.where(torch.cat([ok[prob], ok[cprob]]), x + step, x)
        grow = torch.maximum(torch.full_like(lam, 1.0 / 3.0), 1.0 - (2.0 * rho - 1.0) ** 3)
        lam, nu = (torch.where(done, lam, torch.where(ok, lam * grow, lam * nu)),
                   torch.where(done, nu, torch.where(ok, torch.full_like(nu, 2.0), nu * 2.0)))
        if case["iterations"] > 1:
            done = done | (ok & (cost - cost_new <= 1e-12 * cost)) | (lam > 1e16)
    out = {k: last[k] for k in ("cost", "cost_new", "pred", "rho")}
    return dict(out, **{"lambda": lam, "accepted": None, "x": x})


def exact(case, seed):
    return {"blocks": _exact_blocks, "banded": _exact_banded, "lm": _exact_lm}.get(case["kind"], _exact_dense)(case, seed)
