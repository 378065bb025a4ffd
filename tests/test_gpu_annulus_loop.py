"""The annulus solve's device loop: more steps than its history ring holds, other buffers, cycles
and shifts on one plan, solves that end at their start.  All comparisons are exact: the same
launches on the same values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _solve(plan, d, tol, steps):
    from paper_2308_11469_gb300 import binding as B
    dd = torch.from_numpy(d).cuda()
    u = torch.full_like(dd, float("nan"))
    st, it, hist = B.helm_annulus_solve(plan, dd, u, tol, steps)
    return int(st), it, np.array(hist), u.cpu().numpy()


def _data(N, seed=0):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((N + 1, N + 1)) + 1j * rng.standard_normal((N + 1, N + 1))


@pytest.mark.parametrize("prec", ["MIXED", "FP64"])
def test_more_steps_than_the_ring(prec):
    from paper_2308_11469_gb300 import binding as B
    plan = B.helm_annulus_create(16, 1.0, 0.15, 0.8, getattr(B, "HELM_PREC_" + prec))
    B.helm_annulus_set_shift(plan, 3e4)              # slow: falls through thousands of steps
    d = _data(16)
    st, it, h, u = _solve(plan, d, 0.0, 4500)
    assert st == B.HELM_MAXITER and it == 4500 and len(h) == 4501
    assert np.isfinite(h).all() and h[-1] < h[4095] < h[100] and np.isfinite(u).all()
    for m in (4094, 4095, 4096, 101):
        st, it, g, _ = _solve(plan, d, 0.0, m)
        assert st == B.HELM_MAXITER and it == m and np.array_equal(g, h[:m + 1])
    B.helm_annulus_destroy(plan)


@pytest.mark.parametrize("prec", ["MIXED", "FP64"])
def test_one_plan_several_solves(prec):
    from paper_2308_11469_gb300 import binding as B
    plan = B.helm_annulus_create(64, 1.0, 0.15, 0.8, getattr(B, "HELM_PREC_" + prec))
    for alpha, cycle, seed, tol in [(0.8 * 0.8, (2, 2, 1), 1, 1e-8), (0.8 * 0.8, (2, 2, 1), 2, 1e-8),
                                    (0.8 * 0.8, (1, 3, 2), 1, 1e-6), (1.5, (1, 3, 2), 1, 1e-6)]:
        other = B.helm_annulus_create(64, 1.0, 0.15, 0.8, getattr(B, "HELM_PREC_" + prec))
        for p in (plan, other):
            B.helm_annulus_set_cycle(p, *cycle)
            B.helm_annulus_set_shift(p, alpha)
        a, b = (_solve(p, _data(64, seed), tol, 60) for p in (plan, other))
        B.helm_annulus_destroy(other)
        assert a[:2] == b[:2] and np.array_equal(a[2], b[2]) and np.array_equal(a[3], b[3])
    B.helm_annulus_destroy(plan)


def test_solves_that_end_at_their_start():
    from paper_2308_11469_gb300 import binding as B
    plan = B.helm_annulus_create(64, 1.0, 0.15, 0.8, B.HELM_PREC_MIXED)
    z = np.zeros((65, 65), dtype=complex)
    st, it, h, u = _solve(plan, z, 1e-8, 20)
    assert (st, it, h.tolist()) == (B.HELM_CONVERGED, 0, [0.0]) and not u.any()
    d = _data(64)
    st, it, h, u = _solve(plan, d, 1e-8, 0)
    assert (st, it, h.tolist()) == (B.HELM_MAXITER, 0, [1.0])
    assert np.array_equal(u, np.where(u != 0, d, 0)) and u.any()      # the hole's data alone
    st, it, h, u = _solve(plan, d, 1e-3, 60)
    assert st == B.HELM_CONVERGED and 0 < it < 60 and h[-1] <= 1e-3 < h[-2]
    B.helm_annulus_destroy(plan)
