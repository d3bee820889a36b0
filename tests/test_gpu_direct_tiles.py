"""The FP32 direct solve of each anchor's batch regression on 8 x 8 register tiles, against the
oracle's subset loop at the edges of its tiling: one tile, a ragged last tile, block sizes of
two to five warps, the widest row, and windows of one row, a whole stage, one more and one
less than a stage, and every particle (FP32 bar 1e-4)."""
import numpy as np
import pytest

import oracle
from helpers import TOL_FP32

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,M,K", [(1, 40, 15), (8, 60, 16), (9, 64, 17), (33, 150, 150),
                                   (57, 200, 128), (80, 260, 161), (100, 301, 256),
                                   (104, 300, 239), (121, 320, 255), (128, 330, 272)])
def test_direct_tiles_match_oracle(d, M, K):
    from paper_2510_02635_gb300 import fbsde as fb
    sigma, T, N, seed = 1.4142135623730951, 0.3, 2, 23
    x0 = np.random.default_rng(d).normal(scale=0.3, size=(1, d))
    p = fb.make_problem("ac_doublewell", d, N, M, sigma, T, "fp32")
    out = fb.solve_anchored(p, torch.tensor(x0, device="cuda"), seed, 0, K=K, direct=True)
    torch.cuda.synchronize()
    ref = oracle.solve_batch(oracle.Problem("ac_doublewell", d, sigma, T, N, M, cg_tol=1e-13,
                                            cg_max_iter=1000), K, x0[0], seed, 0)
    assert out["status"] == 0 and ref["status"] == 0
    u, g = float(out["u0"][0]), out["grad"][0].cpu().numpy()
    assert abs(u - ref["u0"]) <= TOL_FP32 * abs(ref["u0"])
    assert np.linalg.norm(g - ref["grad"]) <= TOL_FP32 * max(np.linalg.norm(ref["grad"]),
                                                             abs(ref["u0"]))
