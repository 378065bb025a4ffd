"""The 3D residual at its floor: how exact an iterate the outer iteration settles on, where the
history cannot show it (a residual that is off by a few units everywhere is driven to zero as
well).

An iterate is stored to half an ulp, and a correction below half an ulp leaves it alone: at a
fixed point the error is at most 2^-53 of the values for each, over 1 - (contraction of a step).
Both cases contract by less than 1/2 a step, and the runs are long enough to reach the floor.
The discrete operator is the library's: 1 / h^2 and k^2 rounded to FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")
U53 = 2.0 ** -53


def _settle(n, h, k, prec, f, g, calls, steps):
    """The iterate after calls x steps outer steps (each call goes on from the last one's)."""
    from paper_2308_11469_gb300 import binding as B
    plan = B.helm_plan_create(3, n, h, k, prec=prec)
    B.helm_plan_set_cycle(plan, 0, 2, 1)
    fd, gd = (torch.from_numpy(np.ascontiguousarray(a, dtype=complex)).cuda() for a in (f, g))
    u = torch.zeros_like(gd)
    for _ in range(calls):
        B.helm_solve(plan, fd, gd, u, 0.0, steps)
    B.helm_plan_destroy(plan)
    return u.cpu().numpy()


@pytest.mark.parametrize("n", [63, 127])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("side", [1.0, 0.7])
def test_smooth_source(n, prec, side):
    # f = sin sin sin is an eigenvector of the discrete Laplacian: u = f / (k^2 - lambda).  An
    # error of one sign over the grid is the one that the inverse amplifies most (N^2 / 30)
    h, k = side / (n + 1), 2.0 / side
    s = np.sin(PI * np.arange(1, n + 1).astype(LD) / (n + 1))
    lam = 3 * 4 * LD(1.0 / (h * h)) * np.sin(PI / (2 * LD(n + 1))) ** 2
    f = s[:, None, None] * s[None, :, None] * s[None, None, :]
    u = _settle(n, h, k, prec, (f * (1 + 2j)).astype(complex), np.zeros((n + 2,) * 3), 2, 19)
    want = f / (LD(k * k) - lam)
    got = u[1:-1, 1:-1, 1:-1]
    err = ((got.real.astype(LD) - want) ** 2 + (got.imag.astype(LD) - 2 * want) ** 2).sum()
    # two roundings over 1 - 1/2, relative to each component's own size
    assert float(np.sqrt(err / (5 * (want ** 2).sum()))) <= 4 * U53


@pytest.mark.parametrize("n", [63, 127])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("side", [1.0, 0.7])
@pytest.mark.parametrize("data", ["wall", "steep", "gauss"])
def test_field_that_decays_across_the_box(n, prec, side, data):
    # oscillating data on the face z = 0 (the iterate falls by seven orders of magnitude across the
    # box, or, steep, by four across a tile's planes) or a narrow source: h^2 times the residual of
    # every plane is at the rounding of that plane's own values: half an ulp of a node and its six
    # neighbours (12 of them in all), the same for a correction too small to be added, rounded up
    # to 32.  (steep: planes down to 2^-16 of the largest; in lower ones the corrections that follow
    # the roundings of the planes near the wall, 2^-53 k^2 h^2 of those, are above their own)
    h, k = side / (n + 1), 1.0 / side
    t = np.arange(n + 2) / (n + 1)
    f = np.zeros((n,) * 3, dtype=complex)
    g = np.zeros((n + 2,) * 3, dtype=complex)
    if data == "gauss":
        x = t[1:-1]
        b = [np.exp(-((x - c) ** 2) / (2 * 0.02 ** 2)) for c in (0.3, 0.55, 0.2)]
        f = b[0][:, None, None] * b[1][None, :, None] * b[2][None, None, :] * (1 - 0.5j)
    else:
        m = 4 if data == "wall" else (n + 1) // 8
        g[0] = np.sin(m * np.pi * t)[:, None] * np.sin(m * np.pi * t)[None, :] * (1 - 0.5j)
    u = _settle(n, h, k, prec, f, g, 6, 18)
    h2 = 1 / LD(1.0 / (h * h))
    for part, src in ((u.real, f.real), (u.imag, f.imag)):
        a = part.astype(LD)
        m = a[1:-1, 1:-1, 1:-1]
        r = (a[2:, 1:-1, 1:-1] + a[:-2, 1:-1, 1:-1] + a[1:-1, 2:, 1:-1] + a[1:-1, :-2, 1:-1]
             + a[1:-1, 1:-1, 2:] + a[1:-1, 1:-1, :-2] - 6 * m) + h2 * (LD(k * k) * m - src)
        plane = np.abs(a).max(axis=(1, 2))
        near = np.maximum(np.maximum(plane[:-2], plane[1:-1]), plane[2:])
        worst = (np.abs(r).max(axis=(1, 2)) / near).astype(float)
        if data == "steep":
            worst = worst[near >= 2.0 ** -16 * near.max()]
        assert worst.max() <= 32 * U53, (int(worst.argmax()) + 1, worst.max() / U53)


@pytest.mark.parametrize("prec", [0, 1])
def test_one_launch_for_both_kinds_of_spacing(prec):
    # a batch whose solves share a launch, with and without a power of two for h^2: each gets the
    # bits of its solve alone
    from paper_2308_11469_gb300 import binding as B
    n = 63
    rng = np.random.default_rng(5)
    f = torch.from_numpy(rng.standard_normal((n,) * 3) + 1j * rng.standard_normal((n,) * 3)).cuda()
    g = torch.from_numpy(rng.standard_normal((n + 2,) * 3) + 1j * rng.standard_normal((n + 2,) * 3)).cuda()
    hs = [1.0 / (n + 1), 0.7 / (n + 1), 0.7 / (n + 1)]
    batch = B.helm_batch_create(0)
    B.helm_batch_set_cycle(batch, 0, 2, 1)
    B.helm_batch_set_lanes(batch, 1)
    us = [torch.zeros_like(g) for _ in hs]
    ts = B.helm_batch_submit_many(batch, [(3, n, h, 2.0, f, g, u) for h, u in zip(hs, us)], prec, 1e-9, 60)
    B.helm_batch_step(batch, 0)
    got = [B.helm_batch_poll(batch, t, 60) for t in ts]
    B.helm_batch_destroy(batch)
    for h, u, r in zip(hs, us, got):
        plan = B.helm_plan_create(3, n, h, 2.0, prec=prec)
        B.helm_plan_set_cycle(plan, 0, 2, 1)
        v = torch.zeros_like(g)
        st, it, hist = B.helm_solve(plan, f, g, v, 1e-9, 60)
        B.helm_plan_destroy(plan)
        assert (st, it) == r[:2] and np.array_equal(hist, r[2]) and torch.equal(u, v)
