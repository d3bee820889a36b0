"""The conjugate gradients in one cooperative launch (k_cg_loop) against the FP64 oracle, and
against the same passes launched phase by phase (bit for bit), at the edges of its geometry:
rows that stay in shared memory (one stage, two stages) and rows that stream through the ring
(several teams, one team per row), every tile width, the shares of few tiles (one thread) and
of many (a warp), the most queries the loop takes and one more (the two-launch form), and a
pass count that runs out.  The bars are those of the two paths (FP32 1e-4, FP64 1e-10)."""
import math

import pytest

import oracle
from helpers import TOL_FP32, TOL_FP64, gpu_solver, oracle_problem, rel_errors
from paper_2510_02635_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (kind, d, M, N, Q, precision); M < d takes a ridge of the mean eigenvalue
CASES = [
    ("ac_manufactured", 3, 5, 2, 1, "fp32"),          # one tile of four coordinates
    ("ac_manufactured", 64, 13, 2, 3, "fp32"),        # fewer rows than teams
    ("ac_manufactured", 612, 2129, 3, 1, "fp32"),     # 153 tiles of four: eight-wide ones
    ("logistic_grad", 1021, 4099, 2, 1, "fp32"),      # resident, two stages, ragged
    ("ac_manufactured", 130, 700, 3, 64, "fp32"),     # the most queries; serial shares
    ("ac_manufactured", 130, 700, 3, 65, "fp32"),     # beyond: two launches a pass
    ("logistic_grad", 1205, 6011, 2, 1, "fp32"),      # streams, several teams
    ("ac_manufactured", 4999, 1501, 2, 1, "fp32"),    # streams, one team per row (pairs)
    ("logistic_grad", 2501, 3001, 2, 2, "fp32"),      # streams, two queries
    ("ac_manufactured", 101, 2047, 3, 1, "fp64"),     # resident FP64
    ("logistic_grad", 1301, 2503, 2, 1, "fp64"),      # FP64 rows that stream
]


def _workload(kind, d, M, N, Q, prec):
    sigma, T = (float(d), 1.0) if kind == "logistic_grad" else (1.0, 0.5)
    ridge = {"ridge_rel": 1.0} if M < 1.25 * d else {}
    return W.Workload(f"loop_{d}_{M}", kind, d=d, sigma=sigma, T=T, N=N, M=M, Q=Q, seed=17,
                      x0_law="normal_1/d", precision=prec,
                      cg_tol=1e-13 if prec == "fp64" else 1e-7, cg_max_iter=1000, **ridge)


@pytest.mark.parametrize("kind,d,M,N,Q,prec", CASES)
def test_loop_matches_oracle_and_single_phases(kind, d, M, N, Q, prec):
    from paper_2510_02635_gb300 import fbsde
    w = _workload(kind, d, M, N, Q, prec)
    x0 = W.inputs(w)["x0"]
    solver = gpu_solver(w)
    xd = torch.tensor(x0, device="cuda")
    out = solver.solve(xd, seed=w.seed)
    assert out["status"] == 0
    fbsde.fbsde_profile_start(1 << 16)   # the first passes of each level phase by phase
    fbsde.fbsde_profile_select(["matvec"])
    split = solver.solve(xd, seed=w.seed)
    torch.cuda.synchronize()
    fbsde.fbsde_profile_stop()
    assert torch.equal(out["u0"], split["u0"]) and torch.equal(out["grad"], split["grad"])
    tol = TOL_FP64 if prec == "fp64" else TOL_FP32
    for q in {0, Q // 2, Q - 1}:
        ref = oracle.solve(oracle_problem(w), x0[q], w.seed, q)
        ru, rg = rel_errors(float(out["u0"][q]), out["grad"][q].cpu().numpy(), ref)
        assert ru <= tol and rg <= tol, (q, ru, rg)


@pytest.mark.parametrize("Q", [1, 3])
def test_loop_reports_exhausted_passes(Q):
    """cg_max_iter passes in the loop and one by one: the same iterate and status."""
    from paper_2510_02635_gb300 import fbsde
    w = _workload("ac_manufactured", 300, 900, 3, Q, "fp32")
    xd = torch.tensor(W.inputs(w)["x0"], device="cuda")
    solver = gpu_solver(w, cg_max_iter=3)
    a = solver.solve(xd, seed=w.seed)
    fbsde.fbsde_profile_start(1 << 12)
    fbsde.fbsde_profile_select(["matvec"])
    b = solver.solve(xd, seed=w.seed)
    torch.cuda.synchronize()
    fbsde.fbsde_profile_stop()
    assert a["status"] == b["status"] == 5 and a["solves_cg_exhausted"] == Q
    assert torch.equal(a["u0"], b["u0"]) and torch.equal(a["grad"], b["grad"])
    assert math.isfinite(float(a["u0"][0]))
