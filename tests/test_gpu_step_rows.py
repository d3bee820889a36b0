"""The fused level step where its geometry changes: rows per stage from 32 down to one, one to
five chunks per thread, rings of three to eight stages with either lag of the column pass, and
small clouds spread over one wave of CTAs, against the FP64 oracle (FP32 bar 1e-4)."""
import pytest

import oracle
from helpers import TOL_FP32, gpu_solver, oracle_problem, rel_errors
from paper_2510_02635_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,d,M,Q", [("ac_manufactured", 256, 947, 1),
                                        ("logistic_grad", 257, 403, 2),
                                        ("ac_manufactured", 512, 707, 1),
                                        ("logistic_grad", 513, 691, 1),
                                        ("ac_manufactured", 1536, 2141, 1),
                                        ("logistic_grad", 1537, 2003, 1),
                                        ("ac_manufactured", 2560, 3201, 1),
                                        ("logistic_grad", 3412, 3607, 1),
                                        ("ac_manufactured", 3416, 3601, 1),
                                        ("ac_manufactured", 50, 3001, 1),
                                        ("logistic_grad", 340, 457, 3)])
def test_step_rows_match_oracle(kind, d, M, Q):
    sigma, T = (float(d), 1.0) if kind == "logistic_grad" else (1.0, 0.5)
    w = W.Workload(f"rows_{d}", kind, d=d, sigma=sigma, T=T, N=3, M=M, Q=Q, seed=29,
                   x0_law="normal_1/d", precision="fp32", cg_tol=1e-7, cg_max_iter=1000)
    x0 = W.inputs(w)["x0"]
    out = gpu_solver(w).solve(torch.tensor(x0, device="cuda"), seed=w.seed)
    assert out["status"] == 0
    for q in range(Q):
        ref = oracle.solve(oracle_problem(w), x0[q], w.seed, q)
        ru, rg = rel_errors(float(out["u0"][q]), out["grad"][q].cpu().numpy(), ref)
        assert ru <= TOL_FP32 and rg <= TOL_FP32, (q, ru, rg)
