"""The FP32 path at small diffusions: r . A r leaves the FP32 range after a few passes (its terms
are the squares of dot products near 1e-20) while the rows, r and the products stay in it, so
the solves converge (status 0) to the value of the FP64 path (FP32 bar 1e-4)."""
import math

import numpy as np
import pytest

from helpers import TOL_FP32

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# the loop with its rows in shared memory and streaming, one team per row, separate launches
@pytest.mark.parametrize("d,M,Q", [(64, 512, 1), (1000, 4096, 2), (5003, 5501, 1), (130, 700, 65)])
@pytest.mark.parametrize("sigma", [1e-5, 1e-7])
def test_small_diffusions_converge(d, M, Q, sigma):
    from paper_2510_02635_gb300 import fbsde as fb
    x0 = torch.tensor(np.random.default_rng(1).standard_normal((Q, d)) / math.sqrt(d),
                      device="cuda")
    out = {}
    for prec in ("fp32", "fp64"):
        solver = fb.Solver("ac_manufactured", d, 3, M, sigma, 0.5, Q=Q, precision=prec,
                           cg_tol=1e-6, cg_max_iter=500, ridge_rel=0.1 if M < 2 * d else 1e-3)
        out[prec] = solver.solve(x0, seed=3)
        assert out[prec]["status"] == 0
    u32, u64 = out["fp32"]["u0"], out["fp64"]["u0"]
    assert bool(((u32 - u64).abs() <= TOL_FP32 * u64.abs()).all())
