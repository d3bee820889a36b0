"""The CG's launch forms for the shapes that the cooperative loop does not take: more queries than
it holds (two launches a pass), several queries whose rows stream from HBM (two launches, and
three for rows above 16 KB), and the FP32 forward SDE (three launches).  Eagerly the passes run in
a cached CUDA graph; its replay, the first passes one by one under the profiler, every pass one by
one on a captured stream, and a plan of several branches give the same bits, and the oracle's
values (FP32 bar 1e-4)."""
import math

import numpy as np
import pytest

import oracle
from helpers import TOL_FP32

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DRIFT = {"mu0": 0.1, "mu1": -0.8, "sig1": 0.2}
# (kind, d, M, N, Q, drift)
CASES = [("ac_manufactured", 101, 503, 3, 65, {}),
         ("logistic_grad", 1003, 9001, 2, 17, {}),
         ("ac_manufactured", 4203, 6007, 2, 6, {}),
         ("ac_manufactured", 300, 1203, 4, 3, DRIFT)]


def _setup(fb, kind, d, M, N, Q, drift, cg_max_iter=60):
    sigma, T = (float(d), 1.0) if kind == "logistic_grad" else (0.5 if drift else 1.0, 0.5)
    p = fb.make_problem(kind, d, N, M, sigma, T, "fp32", cg_tol=1e-6, cg_max_iter=cg_max_iter,
                        ridge_rel=0.05, **drift)
    x0 = np.random.default_rng(d).standard_normal((Q, d)) / math.sqrt(d)
    ws = torch.empty(fb.fbsde_workspace_bytes(p, Q), dtype=torch.uint8, device="cuda")
    return p, torch.tensor(x0, device="cuda"), ws, sigma, T


def _solve(fb, p, Q, x0, ws, stream=None):
    u = torch.empty(Q, dtype=torch.float64, device="cuda")
    g = torch.empty(Q, p.d, dtype=torch.float64, device="cuda")
    fb.check(fb.fbsde_solve(p, Q, x0, 9, 0, u, g, ws, stream=stream))
    return u, g


@pytest.mark.parametrize("kind,d,M,N,Q,drift", CASES)
def test_forms_agree_bitwise_and_with_the_oracle(kind, d, M, N, Q, drift):
    from paper_2510_02635_gb300 import fbsde as fb
    p, x0, ws, sigma, T = _setup(fb, kind, d, M, N, Q, drift)
    u0, g0 = _solve(fb, p, Q, x0, ws)            # captured into the cached graph
    assert fb.fbsde_diagnostics(p, Q, ws).status == 0
    forms = [_solve(fb, p, Q, x0, ws)]           # its replay
    fb.fbsde_profile_start(1 << 16)
    fb.fbsde_profile_select(["matvec"])
    forms.append(_solve(fb, p, Q, x0, ws))       # the first passes one by one
    torch.cuda.synchronize()
    prof = fb.fbsde_profile_stop()
    assert prof["matvec"]["launches"] == N * fb.FBSDE_PROFILED_EAGER_PASSES
    graph = torch.cuda.CUDAGraph()               # every pass one by one, captured
    with torch.cuda.graph(graph, stream=torch.cuda.Stream(), capture_error_mode="thread_local"):
        u = torch.empty(Q, dtype=torch.float64, device="cuda")
        g = torch.empty(Q, d, dtype=torch.float64, device="cuda")
        fb.check(fb.fbsde_solve(p, Q, x0, 9, 0, u, g, ws, stream=torch.cuda.current_stream()))
    graph.replay()
    torch.cuda.synchronize()
    forms.append((u.clone(), g.clone()))
    plan = fb.Plan([{"problem": p, "Q": Q, "x0": x0, "seed": 9, "solve_index0": 0}] * 2, branches=2)
    plan.launch()
    torch.cuda.synchronize()
    forms += list(zip(plan.u0, plan.grad))
    for u, g in forms:
        assert torch.equal(u, u0) and torch.equal(g, g0)
    plan.close()
    prob = oracle.Problem(kind, d, sigma, T, N, M, ridge_rel=0.05, cg_tol=1e-12)
    for q in {0, Q - 1}:
        xq = x0[q].cpu().numpy()
        ref = oracle.solve_sde(prob, xq, 9, q, **drift) if drift else oracle.solve(prob, xq, 9, q)
        scale = max(np.linalg.norm(ref["grad"]), abs(ref["u0"]))
        assert abs(float(u0[q]) - ref["u0"]) <= TOL_FP32 * abs(ref["u0"])
        assert np.linalg.norm(g0[q].cpu().numpy() - ref["grad"]) <= TOL_FP32 * scale
