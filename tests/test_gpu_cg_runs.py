"""Regressions whose chunks of rows are longer than a run of the FP32 sums (32 rows a team): one
team per row streaming through the ring (two rows of two stages at a time), several teams
streaming, rows in shared memory, several queries, the two-launch form, and FP64 rows that stream
with one team per row (no runs).  Against the FP64 oracle (FP32 bar 1e-4, FP64 1e-10), and bit for
bit between the loop and the same passes launched phase by phase, whose stages differ."""
import pytest

import oracle
from helpers import TOL_FP32, TOL_FP64, gpu_solver, oracle_problem, rel_errors
from paper_2510_02635_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,d,M,N,Q,prec", [("ac_manufactured", 5003, 6007, 2, 1, "fp32"),
                                               ("logistic_grad", 8001, 4999, 2, 1, "fp32"),
                                               ("ac_manufactured", 4201, 2503, 2, 3, "fp32"),
                                               ("ac_manufactured", 40, 200003, 2, 1, "fp32"),
                                               ("logistic_grad", 12, 300007, 2, 1, "fp32"),
                                               ("ac_manufactured", 701, 30011, 2, 2, "fp32"),
                                               ("logistic_grad", 33, 5003, 2, 65, "fp32"),
                                               ("logistic_grad", 3001, 4003, 2, 1, "fp64")])
def test_long_chunks_match_oracle_and_single_phases(kind, d, M, N, Q, prec):
    from paper_2510_02635_gb300 import fbsde
    sigma, T = (float(d), 1.0) if kind == "logistic_grad" else (1.0, 0.5)
    ridge = {"ridge_rel": 1.0} if M < 1.25 * d else {}
    w = W.Workload(f"runs_{d}_{M}", kind, d=d, sigma=sigma, T=T, N=N, M=M, Q=Q, seed=31,
                   x0_law="normal_1/d", precision=prec,
                   cg_tol=1e-13 if prec == "fp64" else 1e-7, cg_max_iter=2000, **ridge)
    x0 = W.inputs(w)["x0"]
    solver = gpu_solver(w)
    xd = torch.tensor(x0, device="cuda")
    out = solver.solve(xd, seed=w.seed)
    assert out["status"] == 0
    fbsde.fbsde_profile_start(1 << 16)
    fbsde.fbsde_profile_select(["matvec"])
    split = solver.solve(xd, seed=w.seed)
    torch.cuda.synchronize()
    fbsde.fbsde_profile_stop()
    assert torch.equal(out["u0"], split["u0"]) and torch.equal(out["grad"], split["grad"])
    tol = TOL_FP64 if prec == "fp64" else TOL_FP32
    for q in {0, Q - 1}:
        ref = oracle.solve(oracle_problem(w), x0[q], w.seed, q)
        ru, rg = rel_errors(float(out["u0"][q]), out["grad"][q].cpu().numpy(), ref)
        assert ru <= tol and rg <= tol, (q, ru, rg)
