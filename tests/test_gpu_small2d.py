"""Whole solves of small 2D grids in one launch (clusters of CTAs): the same bits as the
launch-by-launch path (HELM_COARSE_CTA keeps it) for every schedule, cluster size, damping
and step budget."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _problem(n, k, seed):
    import torch
    rng = np.random.default_rng(seed)
    h = 1.0 / (n + 1)
    f = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    g = rng.standard_normal((n + 2, n + 2)) + 1j * rng.standard_normal((n + 2, n + 2))
    return h, torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda()


@pytest.mark.parametrize("n", [31, 63])
@pytest.mark.parametrize("sched", [(2, 2, 1), (0, 1, 1), (1, 2, 2), (3, 0, 1)])
@pytest.mark.parametrize("damp", [0.0, 1.5])
def test_solve_equals_launch_by_launch(n, sched, damp):
    import torch
    from paper_2308_11469_gb300 import binding as B
    k = 3.0
    h, f, g = _problem(n, k, n + sched[0])
    out = []
    for mode in (B.HELM_COARSE_CTA, B.HELM_COARSE_AUTO):
        plan = B.helm_plan_create(2, n, h, k, prec=B.HELM_PREC_MIXED)
        B.helm_plan_set_cycle(plan, *sched)
        B.helm_plan_set_coarse_mode(plan, mode)
        if damp:
            B.helm_plan_set_cavity(plan, k * k + 1.0, damp)
        for cap in (60, 3, 0):                   # to convergence, and out of steps
            u = torch.zeros_like(g)
            st, it, hist, einf = B.helm_solve_ex(plan, f, g, u, 1e-9, cap)
            out.append((mode, cap, st, it, hist, einf, u.cpu().numpy()))
        B.helm_plan_destroy(plan)
    for a, b in zip(out[:3], out[3:]):
        assert a[1:4] == b[1:4]
        assert np.array_equal(a[4], b[4]) and np.array_equal(a[5], b[5])
        assert np.array_equal(a[6], b[6])


@pytest.mark.parametrize("n,count", [(63, 1), (63, 13), (63, 33), (63, 97), (31, 3), (31, 33)])
@pytest.mark.parametrize("chunk", [0, 3])
def test_batch_equals_single(n, count, chunk):
    """Cluster sizes by the number of solves; run to completion or in bounded chunks."""
    import torch
    from paper_2308_11469_gb300 import binding as B
    ks = np.linspace(0.5, 4.0, count)
    h, f, g = _problem(n, 0.0, 7)
    batch = B.helm_batch_create(0)
    B.helm_batch_set_lanes(batch, 1)
    us = [torch.zeros_like(g) for _ in ks]
    ts = B.helm_batch_submit_many(batch, [(2, n, h, float(k), f, g, u) for k, u in zip(ks, us)],
                                  B.HELM_PREC_MIXED, 1e-8, 200)
    for _ in range(100):
        B.helm_batch_step(batch, chunk)
        res = B.helm_batch_poll_many(batch, ts, release=False)
        if all(r[0] for r in res):
            break
    hists = [B.helm_batch_poll(batch, t, 200) for t in ts]
    B.helm_batch_destroy(batch)
    for i in sorted({0, count // 2, count - 1}):
        plan = B.helm_plan_create(2, n, h, float(ks[i]), prec=B.HELM_PREC_MIXED)
        u = torch.zeros_like(g)
        st, it, hist = B.helm_solve(plan, f, g, u, 1e-8, 200)
        B.helm_plan_destroy(plan)
        assert (st, it) == hists[i][:2] and np.array_equal(hist, hists[i][2])
        assert torch.equal(u, us[i])


def test_diverging_and_nonfinite_outcomes():
    import torch
    from paper_2308_11469_gb300 import binding as B
    n, k = 63, 5.0                               # above k_max
    h, f, g = _problem(n, k, 3)
    got = []
    for mode in (B.HELM_COARSE_CTA, B.HELM_COARSE_AUTO):
        plan = B.helm_plan_create(2, n, h, k, prec=B.HELM_PREC_MIXED)
        B.helm_plan_set_coarse_mode(plan, mode)
        u = torch.zeros_like(g)
        got.append(B.helm_solve(plan, f, g, u, 1e-9, 200)[:2])
        bad = f.clone()
        bad[5, 7] = complex(float("nan"), 0.0)
        u.zero_()
        got.append(B.helm_solve(plan, bad, g, u, 1e-9, 200)[:2])
        B.helm_plan_destroy(plan)
    assert got[0] == got[2] and got[0][0] == B.HELM_DIVERGED
    assert got[1] == got[3] and got[1][0] == B.HELM_ENONFINITE
