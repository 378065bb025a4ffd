"""Long one-launch solves of small 2D grids against the launch-by-launch path, bit for bit: more
steps than the launch keeps undecided relres values for (32), step limits on both sides of that
number, histories of solves that diverge."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _both(n, k, seed, tol, caps, sched):
    from paper_2308_11469_gb300 import binding as B
    rng = np.random.default_rng(seed)
    f = torch.from_numpy(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))).cuda()
    g = torch.from_numpy(rng.standard_normal((n + 2, n + 2)) + 1j * rng.standard_normal((n + 2, n + 2))).cuda()
    out = []
    for mode in (B.HELM_COARSE_CTA, B.HELM_COARSE_AUTO):
        plan = B.helm_plan_create(2, n, 1.0 / (n + 1), k, prec=B.HELM_PREC_MIXED)
        B.helm_plan_set_cycle(plan, *sched)
        B.helm_plan_set_coarse_mode(plan, mode)
        for cap in caps:
            u = torch.zeros_like(g)
            out.append(B.helm_solve_ex(plan, f, g, u, tol, cap) + (u,))
        B.helm_plan_destroy(plan)
    half = len(caps)
    for a, b in zip(out[:half], out[half:]):
        assert a[:2] == b[:2]
        assert np.array_equal(a[2], b[2]) and np.array_equal(a[3], b[3])
        assert torch.equal(a[4], b[4])
    return out[:half]


@pytest.mark.parametrize("n", [31, 63])
@pytest.mark.parametrize("k", [4.05, 4.15])
@pytest.mark.parametrize("sched", [(0, 1, 1), (2, 2, 1)])
def test_more_steps_than_are_kept(n, k, sched):
    from paper_2308_11469_gb300 import binding as B
    full = _both(n, k, n, 1e-9, (200, 31, 32, 33, 34, 65), sched)
    assert full[0][0] == B.HELM_CONVERGED and full[0][1] > 65
    assert all(r[0] == B.HELM_MAXITER for r in full[1:])


@pytest.mark.parametrize("n", [31, 63])
def test_diverging_histories(n):
    from paper_2308_11469_gb300 import binding as B
    r = _both(n, 5.0, 3, 1e-9, (200,), (2, 2, 1))
    assert r[0][0] == B.HELM_DIVERGED


@pytest.mark.parametrize("n", [31, 63])
def test_at_the_floor(n):
    # tol = 0: relres falls for some thirty steps, then stands and wavers at its rounding floor
    _both(n, 3.0, 5, 0.0, (100,), (0, 1, 1))
