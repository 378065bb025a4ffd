"""Residual norms near the end of the floats' range: a complex64 solve whose data are scaled by a
power of two such that a residual tile's |r|^2 sums to more than a float holds, while each warp's
share does not, gives the scaled iterates and the history of the unscaled solve."""
import numpy as np
import pytest

from oracle import fd

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("one_launch", [True, False])
def test_history_does_not_depend_on_the_scale(one_launch):
    from paper_2308_11469_gb300 import binding as B
    n, k, steps = 31, 3.0, 6                     # one residual tile, its level solved exactly
    h = 1.0 / (n + 1)
    f = np.ones((n, n), dtype=complex)
    g = np.zeros((n + 2, n + 2), dtype=complex)
    r1 = k * k * fd.solve_exact_dst(f, g, h, 0.0)[1:-1, 1:-1]          # r_1 = -k^2 A^-1 f
    rows = (np.abs(r1) ** 2).sum(axis=1)
    j = int(np.ceil(0.5 * np.log2(1.3 * 2.0 ** 128 / rows.sum())))
    warps = [rows[w::8].sum() * 4.0 ** j for w in range(8)]
    assert sum(warps) >= 1.3 * 2.0 ** 128 and max(warps) <= 0.9 * 2.0 ** 128
    gd, out = torch.from_numpy(g).cuda(), []
    for s in (1.0, 2.0 ** j):
        plan = B.helm_plan_create(2, n, h, k, prec=B.HELM_PREC_MIXED)
        B.helm_plan_set_coarse_mode(plan, B.HELM_COARSE_AUTO if one_launch else B.HELM_COARSE_CTA)
        u = torch.zeros_like(gd)
        out.append(B.helm_solve(plan, torch.from_numpy(f * s).cuda(), gd, u, 0.0, steps) + (u / s,))
        B.helm_plan_destroy(plan)
    (st, it, hist, u), (st2, it2, hist2, u2) = out
    assert (st2, it2) == (st, it) == (B.HELM_MAXITER, steps)
    assert torch.equal(u, u2)
    # (the two ways of adding eight floats: eight roundings of 2^-53, half of them after the root)
    assert np.abs(hist2 / hist - 1.0).max() <= 8 * 2.0 ** -53
