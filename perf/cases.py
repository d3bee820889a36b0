"""The measured cases: what a user of this package has it do, through its public entry points.

A case names one call (or one training step) of the package:
  solve      fbsde.Solver.solve, the solve of Q query points (the main path);
  host       fbsde.fbsde_solve_host, the same from and to host buffers;
  grad       fbsde.fbsde_value with torch.autograd: u forward, then the reverse sweep to x0
             (and theta);
  plan       autotune.Batch, many uneven instances in one plan (one launch);
  anchored   fbsde.fbsde_solve_anchored, one regression per particle anchor;
  batch      fbsde.fbsde_solve_batch, each anchor's regression over K particles (CG);
  direct     fbsde.fbsde_solve_batch_direct, the same solved directly.
Sizes are those of workloads.py, the benchmark and the tests (fewer time steps where a whole
solve would be long), or ragged sizes of the same ranges.  The inputs (x0, theta, the Philox
seed) come from the case's seed with the workloads' own laws.

The FP32 path holds its rows, products and sums in 32 bits and returns them widened; a
program that asked for it keeps its results in that type, as run() does here.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_02635_gb300 import autotune, fbsde
from paper_2510_02635_gb300 import workloads as W

# kind (or the forward SDE with a drift) -> (sigma, T, x0 law) as in workloads.py
LAWS = {
    "ac_manufactured": (lambda d: 1.0, 0.5, "normal_1/d"),
    "logistic_grad": (lambda d: float(d), 1.0, "normal_1/d"),
    "hjb_logquad": (lambda d: math.sqrt(2.0), 1.0, "normal_1/d"),
    "ac_doublewell": (lambda d: math.sqrt(2.0), 0.3, "normal_1/d"),
    "drift": (lambda d: 0.5, 0.6, "normal_1/d"),
}
DRIFT = {"mu0": 0.1, "mu1": -0.8, "sig1": 0.2}


def listed():
    return [
        # the smallest call: one query of a small cloud, where launches and latency count
        {"name": "solve_small_d64", "call": "solve", "kind": "ac_manufactured", "d": 64,
         "M": 512, "N": 6, "Q": 1, "precision": "fp32", "cg_tol": 1e-7, "max_iter": 100},
        # the plain scheme in FP64 throughout (workloads.C0_AC_D100)
        {"name": "solve_fp64_d100", "call": "solve", "kind": "ac_manufactured", "d": 100,
         "M": 2048, "N": 10, "Q": 1, "precision": "fp64", "cg_tol": 1e-12, "max_iter": 0},
        # FP64 with wider rows, as a user runs what FP32 rows do not carry
        {"name": "solve_fp64_d1203", "call": "solve", "kind": "logistic_grad", "d": 1203,
         "M": 2048, "N": 5, "Q": 1, "precision": "fp64", "cg_tol": 1e-12, "max_iter": 3000},
        # an ordinary cloud of one query, from and to host buffers, ragged d
        {"name": "host_d2503", "call": "host", "kind": "ac_manufactured", "d": 2503,
         "M": 8192, "N": 10, "Q": 1, "precision": "fp32", "cg_tol": 1e-6, "max_iter": 0},
        # many queries at once, gradient-dependent driver (workloads.C1_LOGISTIC_D1000)
        {"name": "solve_logistic_d1000_q64", "call": "solve", "kind": "logistic_grad",
         "d": 1000, "M": 4096, "N": 20, "Q": 64, "precision": "fp32", "cg_tol": 1e-6,
         "max_iter": 0},
        # the largest: the benchmark's workload (workloads.C2_AC_D10000) over five of its
        # fifty time steps
        {"name": "solve_d10000_q16", "call": "solve", "kind": "ac_manufactured", "d": 10000,
         "M": 16384, "N": 5, "Q": 16, "precision": "fp32", "cg_tol": 1e-6, "max_iter": 0,
         "T": 1.0, "x0": "uniform_pm1"},
        # value and derivatives through autograd (workloads.C4_HJB_D1000)
        {"name": "grad_hjb_d1000", "call": "grad", "kind": "hjb_logquad", "d": 1000,
         "M": 4096, "N": 20, "Q": 1, "precision": "fp32", "cg_tol": 1e-6, "max_iter": 0},
        # a forward SDE with the drift and diffusion of workloads.F4_DRIFT_AC_D1000
        {"name": "solve_drift_d1000_q16", "call": "solve", "kind": "ac_manufactured",
         "d": 1000, "M": 4096, "N": 20, "Q": 16, "precision": "fp32", "cg_tol": 1e-6,
         "max_iter": 0, "drift": True},
        # uneven instances in one plan: the first of workloads.batch_instances whose
        # regressions are well determined in the type they are routed to, ten time steps each
        {"name": "plan_24", "call": "plan", "n": 24, "first": 0, "N": 10},
        # literal Algorithm 1 at the benchmark's size
        {"name": "anchored_d100", "call": "anchored", "kind": "logistic_grad", "d": 100,
         "M": 2048, "N": 10, "Q": 1, "precision": "fp32", "cg_tol": 1e-6, "max_iter": 0},
        # the same where its contractions carry the time
        {"name": "anchored_d500", "call": "anchored", "kind": "logistic_grad", "d": 500,
         "M": 4096, "N": 2, "Q": 1, "precision": "fp32", "cg_tol": 1e-6, "max_iter": 0},
        # each anchor's regression over 256 particles, solved directly
        {"name": "direct_d100_k256", "call": "direct", "kind": "logistic_grad", "d": 100,
         "M": 2048, "N": 10, "Q": 1, "K": 256, "precision": "fp32", "cg_tol": 1e-6,
         "max_iter": 0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A drawn case that costs no more than the largest listed one (FP64 arithmetic counted
    eight times, about its rate on this part)."""
    most = max(work(c)["flops"] for c in listed())
    while True:
        c = _draw(rng)
        if work(c)["flops"] * (8.0 if c.get("precision") == "fp64" else 1.0) <= 0.5 * most:
            return c


def _draw(rng):
    call = rng.choice(["solve"] * 6 + ["host", "grad", "grad", "drift", "plan", "anchored",
                                       "batch", "direct"])
    if call == "plan":
        return {"call": "plan", "n": rng.randint(2, 24), "first": rng.randint(0, 200),
                "N": rng.choice([4, 7, 10])}
    if call in ("anchored", "batch", "direct"):
        d = _log(rng, 10, 500 if call == "anchored" else 100)
        c = {"call": call, "kind": "logistic_grad" if call == "anchored" else "ac_doublewell",
             "d": d, "M": max(_log(rng, 150, 4096), 4 * d), "N": rng.randint(2, 8),
             "Q": rng.choice([1, 1, 2]),
             "precision": "fp64" if rng.random() < 0.2 else "fp32"}
        if call != "anchored":
            c["K"] = min(c["M"], max(4 * d, _log(rng, 64, 512)))
    else:
        Q = rng.choice([1, 1, 1, 2, 3, 5, 16, 33])
        M = _log(rng, 500, 16384)
        d = _log(rng, 50, min(10000, M // (2 if call in ("solve", "host") else 4)))
        c = {"call": "solve" if call == "drift" else call, "d": d, "M": M,
             "N": rng.randint(2, 12), "Q": Q,
             "kind": rng.choice({"grad": ["hjb_logquad"], "drift": ["ac_manufactured"]}.get(
                 call, ["ac_manufactured", "logistic_grad"])),
             "precision": "fp64" if rng.random() < 0.2 else "fp32"}
        if call == "drift":
            c["drift"] = True
    c["cg_tol"] = 1e-12 if c["precision"] == "fp64" else rng.choice([1e-6, 1e-7])
    c["max_iter"] = 3000
    return c


def _workload(case, seed):
    sigma, T, law = LAWS["drift" if case.get("drift") else case["kind"]]
    return W.Workload("case", case["kind"], d=case["d"], sigma=sigma(case["d"]),
                      T=case.get("T", T), N=case["N"], M=case["M"], Q=case["Q"], seed=seed,
                      x0_law=case.get("x0", law), precision=case["precision"],
                      cg_tol=case["cg_tol"], cg_max_iter=case["max_iter"],
                      theta_law="uniform_0.5_1.5" if case["kind"] == "hjb_logquad" else None,
                      extra=dict(DRIFT) if case.get("drift") else {})


def _instances(case, seed):
    """The plan's instances with the case's number of steps and a seed of their own: those
    of the batch in FP64, or in FP32 with at least two particles a dimension (closer to
    M = d, FP32 rows leave the slopes themselves undetermined at their type's precision)."""
    every = [w for w in autotune.route_precision(W.batch_instances())
             if w.precision == "fp64" or w.M >= 2 * w.d]
    every = [w.with_(N=case["N"], seed=seed)
             for w in every[case["first"]:case["first"] + case["n"]]]
    x0s = W.batch_x0(every, seed=seed)
    return every, x0s


def prepare(case, seed):
    call = case["call"]
    if call == "plan":
        inst, x0s = _instances(case, seed)
        return {"call": call, "batch": autotune.Batch(inst, x0s, None),
                "precision": [w.precision for w in inst]}
    w = _workload(case, seed)
    inp = W.inputs(w)
    x0 = torch.tensor(inp["x0"], device="cuda")
    s = {"call": call, "w": w, "x0": x0, "seed": seed, "precision": w.precision}
    params = {"h": w.h, "ridge_rel": w.ridge_rel, "cg_tol": w.cg_tol,
              "cg_max_iter": w.cg_max_iter}
    if call in ("solve", "grad"):
        s["solver"] = fbsde.Solver(w.kind, w.d, w.N, w.M, w.sigma, w.T, Q=w.Q,
                                   precision=w.precision, theta=inp["theta"], **params,
                                   **w.extra)
        if call == "grad":
            x0.requires_grad_(True)
            s["theta"] = None
            if inp["theta"] is not None:
                s["theta"] = torch.tensor(inp["theta"], device="cuda", requires_grad=True)
        return s
    if call == "host":
        s["x0"] = inp["x0"]
        s["theta"] = None if inp["theta"] is None else np.ascontiguousarray(inp["theta"])
        p = fbsde.make_problem(w.kind, w.d, w.N, w.M, w.sigma, w.T, w.precision,
                               theta=s["theta"], **params)
        n = fbsde.fbsde_workspace_bytes(p, w.Q) + fbsde.fbsde_host_staging_bytes(p, w.Q)
        s["u"], s["g"] = np.zeros(w.Q), np.zeros((w.Q, w.d))
    else:
        s["theta"] = None if inp["theta"] is None else torch.tensor(inp["theta"], device="cuda")
        p = fbsde.make_problem(w.kind, w.d, w.N, w.M, w.sigma, w.T, w.precision,
                               theta=s["theta"], **params)
        n = fbsde.fbsde_anchored_workspace_bytes(p)
        s["K"] = case.get("K")
        s["u"] = torch.empty(w.Q, dtype=torch.float64, device="cuda")
        s["g"] = torch.empty(w.Q, w.d, dtype=torch.float64, device="cuda")
    s["problem"], s["ws"] = p, torch.empty(n, dtype=torch.uint8, device="cuda")
    return s


def _kept(t, precision):
    """A result in the type of the path that computed it."""
    if precision == "fp64":
        return t
    return t.astype(np.float32) if isinstance(t, np.ndarray) else t.to(torch.float32)


def run(s):
    call, prec = s["call"], s["precision"]
    if call == "plan":
        plan = s["batch"].plan
        plan.launch()
        return {"u": [_kept(u, p) for u, p in zip(plan.u0, prec)],
                "g": [_kept(g, p) for g, p in zip(plan.grad, prec)]}
    if call == "solve":
        out = s["solver"].solve(s["x0"], seed=s["seed"])
        return {"u": _kept(out["u0"], prec), "g": _kept(out["grad"], prec),
                "status": out["status"]}
    if call == "grad":
        x0, theta = s["x0"], s["theta"]
        u = fbsde.fbsde_value(s["solver"], x0, s["seed"], theta=theta)
        grads = torch.autograd.grad(u.sum(), [x0] if theta is None else [x0, theta])
        return {"u": _kept(u.detach(), prec), "d": [_kept(g, prec) for g in grads]}
    w, p = s["w"], s["problem"]
    if call == "host":
        fbsde.check(fbsde.fbsde_solve_host(p, w.Q, s["x0"], s["seed"], 0, s["u"], s["g"],
                                           s["ws"]))
        return {"u": _kept(s["u"], prec), "g": _kept(s["g"], prec)}
    if call == "anchored":
        st = fbsde.fbsde_solve_anchored(p, w.Q, s["x0"], s["seed"], 0, s["u"], s["g"], s["ws"])
    else:
        entry = fbsde.fbsde_solve_batch if call == "batch" else fbsde.fbsde_solve_batch_direct
        st = entry(p, s["K"], w.Q, s["x0"], s["seed"], 0, s["u"], s["g"], s["ws"])
    fbsde.check(st)
    return {"u": _kept(s["u"], prec), "g": _kept(s["g"], prec)}


# ------------------------------------------------------------------------------- work
# Bytes of cache and shared memory a working set can stay in between two passes over it.
ON_CHIP = 150e6


def _passes(d, m, tol, ridge=1e-3):
    """CG passes of one regression of m particles in d dimensions: the Chebyshev bound of
    the Marchenko-Pastur spectrum, halved for the starting guess."""
    q = d / m
    hi = (1.0 + math.sqrt(q)) ** 2 + ridge
    lo = ((1.0 - math.sqrt(q)) ** 2 if q <= 1.0 else 0.0) + ridge
    return max(1.0, 0.25 * math.sqrt(hi / lo) * math.log(2.0 / tol))


def _work_solve(d, M, N, Q, precision, tol, adjoint=False):
    cells = float(Q) * M * d
    size = 8.0 if precision == "fp64" else 4.0
    passes = _passes(d, M, tol)
    # a level: the path step and its normal, the prediction and the three moments, then the
    # two contractions of every pass; the reverse sweep has a solve and two sums of its own
    flops = N * cells * (30.0 + 4.0 * passes * (3.0 if adjoint else 1.0))
    io = 8.0 * Q * (2.0 * d + 1.0)
    rows = size * cells
    if rows > ON_CHIP:   # rows that fit no cache: read and written by a step, read by a pass
        io += N * (rows - ON_CHIP) * (2.0 + passes * (3.0 if adjoint else 1.0))
    return {"bytes": io, "flops": flops}


def work(case):
    if case["call"] == "plan":
        total = {"bytes": 0.0, "flops": 0.0}
        for w in _instances(case, 0)[0]:
            one = _work_solve(w.d, w.M, w.N, w.Q, w.precision, w.cg_tol)
            total = {k: total[k] + one[k] for k in total}
        return total
    d, M, N, Q = case["d"], case["M"], case["N"], case["Q"]
    if case["call"] in ("solve", "host", "grad"):
        return _work_solve(d, M, N, Q, case["precision"], case["cg_tol"], case["call"] == "grad")
    K = case.get("K") or M
    pairs = float(Q) * N * M * K
    size = 8.0 if case["precision"] == "fp64" else 4.0
    if case["call"] == "direct":   # second moments (half of a symmetric matrix), L D L^T
        flops = pairs * d * (d + 1.0) + Q * N * M * d ** 3 / 3.0
    else:
        flops = pairs * d * (6.0 + 4.0 * _passes(d, K, case["cg_tol"]))
    return {"bytes": 8.0 * Q * (2.0 * d + 1.0) + size * Q * N * 2.0 * M * d, "flops": flops}


# ------------------------------------------------------------------------------ exact
# The scheme in 64 bits with plain torch: the Philox4x32-10 normals and the Brownian bridge
# (or Euler-Maruyama) paths, the Gaussian weights, each level's ridge regression solved to
# 1e-13, Newton to rounding.  None where it would take long.

def _normals(dev, seed, s, k, M, d):
    """xi_{s,k,j,i} [M, d] of the documented counter layout (i // 4, j, k, s)."""
    m32 = 0xFFFFFFFF
    nb = (d + 3) // 4
    i64 = {"dtype": torch.int64, "device": dev}
    c0 = torch.arange(nb, **i64).repeat(M, 1)
    c1 = torch.arange(M, **i64)[:, None].expand(M, nb).clone()
    c2, c3 = torch.full((M, nb), k, **i64), torch.full((M, nb), s, **i64)
    k0, k1 = seed & m32, (seed >> 32) & m32
    for _ in range(10):
        # products of two 32-bit words, split so that they stay below 2^63
        def halves(x, mul):
            a, b = x * (mul & 0xFFFF), x * (mul >> 16)
            lo = a + ((b & 0xFFFF) << 16)
            return (b >> 16) + (lo >> 32), lo & m32
        h0, l0 = halves(c0, 0xD2511F53)
        h1, l1 = halves(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    def u01(x):
        return ((x >> 9).double() + 0.5) * 2.0 ** -23
    out = torch.empty(M, nb, 4, dtype=torch.float64, device=dev)
    for o, (a, b) in ((0, (c0, c1)), (2, (c2, c3))):
        r = torch.sqrt(-2.0 * torch.log(u01(a)))
        t = 2.0 * math.pi * u01(b)
        out[:, :, o], out[:, :, o + 1] = r * torch.cos(t), r * torch.sin(t)
    return out.reshape(M, 4 * nb)[:, :d].contiguous()


def _g(w, x, theta):
    if w.kind == "ac_manufactured":
        return torch.cos(x).mean(-1)
    if w.kind == "logistic_grad":
        return 1.0 / (1.0 + torch.exp(-(w.T + x.mean(-1))))
    if w.kind == "ac_doublewell":
        return 1.0 / (2.0 + 0.4 * (x * x).sum(-1))
    return torch.log(0.5 * (1.0 + (theta * x * x).sum(-1)))


def _source(w, t, x, ax):
    """What f takes besides y: the source at x, sum z or |z|^2 (z = sigma alpha_x, or
    sigma(x) alpha_x)."""
    if w.kind == "ac_manufactured":
        us = math.exp(t - w.T) * torch.cos(x).mean(-1)
        return us ** 3 - (2.0 - 0.5 * w.sigma ** 2) * us
    if w.kind == "ac_doublewell":
        return torch.zeros_like(x[..., 0])
    z = (w.sigma + w.extra.get("sig1", 0.0) * x) * ax
    return z.sum(-1) if w.kind == "logistic_grad" else (z * z).sum(-1)


def _newton(w, E, feat, dt):
    """The root Y of Y - E - dt f(Y); the last step carries the derivatives."""
    def f(y, ft):
        if w.kind == "logistic_grad":
            return (y - (2.0 + w.d) / (2.0 * w.d)) * ft, ft
        if w.kind == "hjb_logquad":
            return -0.5 * ft + 0.0 * y, torch.zeros_like(ft)
        return y - y ** 3 + ft, 1.0 - 3.0 * y * y
    with torch.no_grad():
        y = E.detach().clone()
        for _ in range(12):
            v, dv = f(y, feat.detach())
            y = y - (y - E.detach() - dt * v) / (1.0 - dt * dv)
    v, dv = f(y, feat)
    return y - (y - E - dt * v) / (1.0 - dt * dv).detach()


class _Solve(torch.autograd.Function):
    """x = (sum_j wn_j D_j D_j^T - S S^T + lam I)^-1 b, constant in everything but b."""

    @staticmethod
    def forward(ctx, b, D, wn, S, lam):
        def mul(v):
            return D.T @ (wn * (D @ v)) - S * (S @ v) + lam * v
        x, r = torch.zeros_like(b), b.clone()
        p, rr, stop = r.clone(), float(r @ r), 1e-26 * float(b @ b)
        for _ in range(6000):
            if rr <= stop:
                break
            q = mul(p)
            a = rr / float(p @ q)
            x, r = x + a * p, r - a * q
            new = float(r @ r)
            p, rr = r + (new / rr) * p, new
        ctx.save_for_backward(D, wn, S)
        ctx.lam = lam
        return x

    @staticmethod
    def backward(ctx, g):
        return _Solve.apply(g, *ctx.saved_tensors, ctx.lam), None, None, None, None


def _exact_query(w, x0, theta, seed, s):
    """(u, grad u) of one query with one anchor per level; differentiable in x0, theta."""
    dev, d, M, N = x0.device, w.d, w.M, w.N
    dt = w.T / N
    sde = bool(w.extra.get("mu1"))
    mu0, mu1, sg1 = (w.extra.get(k, 0.0) for k in ("mu0", "mu1", "sig1"))
    if sde:
        rows, c = [torch.zeros(M, d, dtype=torch.float64, device=dev)], [torch.zeros_like(x0)]
        for k in range(N):
            x = x0 + rows[-1]
            rows.append(rows[-1] + (mu0 + mu1 * x) * dt +
                        (w.sigma + sg1 * x) * math.sqrt(dt) * _normals(dev, seed, s, k, M, d))
            c.append(c[-1] + (mu0 + mu1 * (x0 + c[-1])) * dt)
        D = rows[N]
    else:
        D = w.sigma * math.sqrt(w.T) * _normals(dev, seed, s, N, M, d)
    Y, ax = _g(w, x0 + D, theta), None
    for k in range(N - 1, -1, -1):
        # the rows against the anchor, the weights and the regression of Y on them
        R = D - c[k] if sde else D
        rho = (R * R).sum(1)
        ref = float(rho.mean()) if sde else w.sigma ** 2 * d * (k + 1) * dt
        wn = torch.exp(-(rho - ref) / (w.h ** 2 * ref))
        wn = wn / wn.sum()
        S = D.T @ wn
        cm = wn @ Y
        b = D.T @ (wn * (Y - cm))
        lam = w.ridge_rel * float((wn * (D * D).sum(1)).sum() - S @ S) / d
        ax = _Solve.apply(b, D, wn, S, lam)
        al = cm - S @ ax
        t = k * dt
        if k == 0:
            X, off = x0[None], torch.zeros(1, d, dtype=torch.float64, device=dev)
        else:
            if sde:
                D = rows[k]
            else:
                a = k / (k + 1.0)
                D = a * D + w.sigma * math.sqrt(dt * a) * _normals(dev, seed, s, k, M, d)
            X, off = x0 + D, D
        E = al + (off + (mu0 + mu1 * X) * dt) @ ax if sde else al + off @ ax
        feat = _source(w, t, X, ax)
        Y = _newton(w, E, feat if feat.dim() else feat.expand_as(E), dt)
    return Y.mean(), ax


def _exact_anchored(w, x0, theta, seed, s, K):
    """(u, grad u) of one query with one regression per particle anchor."""
    dev, d, M, N = x0.device, w.d, w.M, w.N
    dt = w.T / N
    P = w.sigma * math.sqrt(w.T) * _normals(dev, seed, s, N, M, d)
    Y = _g(w, x0 + P, theta)
    j = torch.arange(M, device=dev)
    window = ((j[:, None] - j[None, :]) % M) < (K or M)
    x = None
    for k in range(N - 1, -1, -1):
        a = k / (k + 1.0)
        A = torch.zeros_like(P) if k == 0 else (
            a * P + w.sigma * math.sqrt(dt * a) * _normals(dev, seed, s, k, M, d))
        rho = (P * P).sum(1)[:, None] + (A * A).sum(1)[None, :] - 2.0 * P @ A.T
        ref = w.sigma ** 2 * d * (2 * k + 1) * dt
        wn = torch.exp(-(rho - ref) / (w.h ** 2 * ref)) * window
        wn = wn / wn.sum(0)
        G = wn.T @ P
        S, c = G - A, wn.T @ Y
        b = wn.T @ (Y[:, None] * P) - c[:, None] * G
        lam = w.ridge_rel * ((wn * rho).sum(0) - (S * S).sum(1)) / d
        x, r = torch.zeros_like(b), b.clone()
        p, rr = r.clone(), (r * r).sum(1)
        stop = 1e-26 * (b * b).sum(1)
        for _ in range(3000):
            on = rr > stop
            if not bool(on.any()):
                break
            T = wn * (P @ p.T - (A * p).sum(1)[None, :])
            q = (T.T @ P - T.sum(0)[:, None] * A - S * (S * p).sum(1)[:, None]
                 + lam[:, None] * p)
            al = torch.where(on, rr / (p * q).sum(1), torch.zeros_like(rr))[:, None]
            x, r = x + al * p, r - al * q
            new = (r * r).sum(1)
            beta = torch.where(on, new / rr, torch.zeros_like(rr))[:, None]
            p, rr = torch.where(on[:, None], r + beta * p, p), torch.where(on, new, rr)
        E = c - (S * x).sum(1)
        Y = _newton(w, E, _source(w, k * dt, x0 + A, x), dt)
        P = A
    return Y.mean(), x[0]


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["call"] == "plan":
        us, gs = [], []
        for i, (w, x0) in enumerate(zip(*_instances(case, seed))):
            u = g = None
            if w.M * w.d <= 2.5e7:
                with torch.no_grad():
                    u, g = _exact_query(w, torch.tensor(x0[0], device=dev), None, w.seed,
                                        w.extra["index"])
                u, g = u[None], g[None]
            us.append(u)
            gs.append(g)
        return {"u": us, "g": gs}
    w = _workload(case, seed)
    inp = W.inputs(w)
    theta = None if inp["theta"] is None else torch.tensor(inp["theta"], device=dev)
    if case["call"] in ("anchored", "batch", "direct"):
        with torch.no_grad():
            got = [_exact_anchored(w, torch.tensor(x, device=dev), theta, seed, q, case.get("K"))
                   for q, x in enumerate(inp["x0"])]
        return {"u": torch.stack([u for u, _ in got]), "g": torch.stack([g for _, g in got])}
    us, gs = [], []
    if case["call"] == "grad":
        total = None if theta is None else torch.zeros_like(theta)
        for q, x in enumerate(inp["x0"]):
            x = torch.tensor(x, device=dev, requires_grad=True)
            th = None if theta is None else theta.clone().requires_grad_(True)
            u, _ = _exact_query(w, x, th, seed, q)
            d = torch.autograd.grad(u, [x] if th is None else [x, th])
            us.append(u.detach())
            gs.append(d[0])
            if th is not None:
                total += d[1]
        out = [torch.stack(gs)] + ([] if total is None else [total])
        return {"u": torch.stack(us), "d": out}
    with torch.no_grad():
        for q, x in enumerate(inp["x0"]):
            u, g = _exact_query(w, torch.tensor(x, device=dev), theta, seed, q)
            us.append(u)
            gs.append(g)
    out = {"u": torch.stack(us), "g": torch.stack(gs)}
    return out if case["call"] == "host" else {**out, "status": None}
