"""The 3D per-step residual on the instance's fixed-point scale: relres against the residual of
the returned iterate in extended precision, with and without damping, for data that keep the
scale, that leave it (an iterate growing more than fourfold in a step: the tile is redone on
per-plane scales), spacings that are no power of two (per-plane scales throughout) and ragged
grids.  One unit of either scale is below 2^-56 of the iterate's largest value; a residual sums
12 of them over h^2, and rounding to the inner precision adds 2^-24 of itself."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
LD = np.longdouble


def _residual(u, f, h, k, p):
    out = []
    for a, b, c, s in ((u.real, u.imag, f.real, 1), (u.imag, u.real, f.imag, -1)):
        a, b, c = a.astype(LD), b.astype(LD), c.astype(LD)
        m = a[1:-1, 1:-1, 1:-1]
        lap = (a[2:, 1:-1, 1:-1] + a[:-2, 1:-1, 1:-1] + a[1:-1, 2:, 1:-1] + a[1:-1, :-2, 1:-1]
               + a[1:-1, 1:-1, 2:] + a[1:-1, 1:-1, :-2] - 6 * m) / (LD(h) * LD(h))
        out.append(c - lap - LD(k) * LD(k) * m + s * LD(p) * b[1:-1, 1:-1, 1:-1])
    return out


@pytest.mark.parametrize("n", [7, 31, 63])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("h_scale,k,p", [(1.0, 2.0, 0.0), (1.0, 3.0, 1.5), (0.7, 2.0, 0.0), (1.0, 9.0, 0.0)])
def test_relres_is_the_iterates(n, prec, h_scale, k, p):
    # k = 9 is far above k_max: the iterate grows sevenfold a step
    from paper_2308_11469_gb300 import binding as B
    h = h_scale / (n + 1)
    rng = np.random.default_rng(n)
    f = rng.standard_normal((n,) * 3) + 1j * rng.standard_normal((n,) * 3)
    g = rng.standard_normal((n + 2,) * 3) + 1j * rng.standard_normal((n + 2,) * 3)
    plan = B.helm_plan_create(3, n, h, k, prec=prec)
    B.helm_plan_set_cycle(plan, 0, 2, 1)
    if p:
        B.helm_plan_set_cavity(plan, k * k, p)
    fd, gd = torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda()
    base = None
    for steps in (0, 1, 2, 3, 6):
        u = torch.zeros_like(gd)
        st, it, hist = B.helm_solve(plan, fd, gd, u, 0.0, steps)
        un = u.cpu().numpy()
        r = _residual(un, f, h, k, p)
        norm = float(np.sqrt(sum((x * x).sum() for x in r)))
        base = norm / hist[0] if base is None else base        # ||b||
        want = norm / base
        unit = 2.0 ** -56 * 8 * np.abs(un).max() * 12 / (h * h) * np.sqrt(2.0 * n ** 3) / base
        if p == 0.0:
            # (with damping and a wall ||b|| is still that of the wall's share alone)
            assert it == steps
        assert abs(hist[-1] - want) <= unit + want * (2.0 ** -22 if prec else 2.0 ** -48), (steps, hist[-1], want)
    B.helm_plan_destroy(plan)
