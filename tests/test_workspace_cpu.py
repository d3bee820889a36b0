"""Workspace sizes (host side): problems whose clouds alone nearly fill the fixed scratch of
fbsde_solve_noalloc.  The tiling of the level step may not put them beyond it: each of these
fits with the partial vectors of the streaming passes' own CTAs."""
import pytest

from paper_2510_02635_gb300 import fbsde

SDE = {"mu0": 0.1, "mu1": -0.8, "sig1": 0.2}

# (d, Q, M, ctas, forward SDE)
CASES = [
    (2000, 2, 3620, 0, False),
    (9461, 65, 2, 0, False),
    (656, 5, 4681, 304, False),
    (7061, 65, 6, 76, False),
    (1662, 2, 1231, 1, True),
    (2987, 8, 161, 304, True),
    (4161, 64, 7, 0, True),
    (4489, 16, 46, 5000, True),
    (3060, 1, 1301, 608, True),
]


@pytest.mark.parametrize("d,Q,M,ctas,sde", CASES)
def test_step_tiling_keeps_problems_within_the_fixed_scratch(d, Q, M, ctas, sde):
    p = fbsde.make_problem("drift_ac" if sde else "ac_manufactured", d, 5, M, 1.0, 1.0, "fp32",
                           ctas=ctas, **(SDE if sde else {}))
    assert 0 < fbsde.fbsde_workspace_bytes(p, Q) <= fbsde.FBSDE_NOALLOC_MAX_BYTES


@pytest.mark.parametrize("d,M", [(3802, 133), (4291, 151), (7842, 113)])
def test_small_wide_clouds_take_no_more_partials_than_rows(d, M):
    """The level step's three partial vectors a CTA stay within the bytes of the rows, beside
    what the other sections take (vectors of d, a few values a row)."""
    p = fbsde.make_problem("ac_manufactured", d, 5, M, 1.0, 1.0, "fp32")
    ld = (d + 3) // 4 * 4
    rows, other = 4 * M * ld, (9 * 8 + 5 * 4) * ld + M * (8 + 4 + 12 + 24 * (ld // 512 + 1))
    assert fbsde.fbsde_workspace_bytes(p, 1) <= 2 * rows + other + (64 << 10)
