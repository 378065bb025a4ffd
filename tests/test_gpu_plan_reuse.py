"""One plan used for cycles of several schedules, solves and spectral radii in turn gives what a
fresh plan gives for each call (bit for bit), whatever ran before it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("D,n,prec", [(2, 63, 1), (2, 127, 0), (2, 511, 1), (3, 31, 1), (3, 15, 0)])
def test_mixed_use_of_one_plan(D, n, prec):
    from paper_2308_11469_gb300 import binding as B
    rng = np.random.default_rng(n)
    h, k = 1.0 / (n + 1), 2.0
    dt = torch.complex64 if prec else torch.complex128
    cplx = lambda shape: torch.from_numpy(rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).cuda()
    rhs, e0 = cplx((n,) * D).to(dt), cplx((n,) * D).to(dt)
    f, g = cplx((n,) * D), cplx((n + 2,) * D)

    def cycle(plan, nu):
        e = e0.clone()
        B.poisson_vcycle(plan, rhs, e, *nu)
        return e

    def solve(plan, cap):
        u = torch.zeros_like(g)
        st, it, hist, einf = B.helm_solve_ex(plan, f, g, u, 1e-8, cap)
        return torch.cat([torch.view_as_real(u).reshape(-1).cpu(), torch.from_numpy(hist), torch.from_numpy(einf),
                          torch.tensor([st, it], dtype=torch.float64)])

    def radius(plan):
        return torch.tensor(B.helm_spectral_radius(plan, 20, 1e-6, 2), dtype=torch.float64)

    def shift(plan):
        B.helm_plan_set_cavity(plan, k * k + 1.0, 0.5)
        return torch.zeros(1)

    calls = [lambda p: cycle(p, (2, 2)), lambda p: cycle(p, (0, 1)), lambda p: solve(p, 60), lambda p: cycle(p, (0, 1)),
             lambda p: solve(p, 3), lambda p: solve(p, 2), radius, lambda p: cycle(p, (2, 2)), shift,
             lambda p: cycle(p, (1, 1)), lambda p: solve(p, 1100), lambda p: cycle(p, (1, 1))]
    one = B.helm_plan_create(D, n, h, k, prec=prec)
    shifted = False
    for i, c in enumerate(calls):
        got = c(one)
        shifted = shifted or c is shift
        fresh = B.helm_plan_create(D, n, h, k, prec=prec)
        if shifted and c is not shift:
            shift(fresh)
        want = c(fresh)
        B.helm_plan_destroy(fresh)
        assert torch.equal(got, want), i
    B.helm_plan_destroy(one)
