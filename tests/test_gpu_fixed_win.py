"""FP64 2D cycles in 64-bit fixed-point windows against the same cycle in extended precision:
the error is FP64's own.  The last update of a node and the correction under it make at most
ten roundings of half an ulp of values no larger than the result's largest: 10 * 2^-53 = 1.1e-15
of the result's norm.  Rough and smooth right-hand sides, an iterate far larger than the
correction, a spacing that is no power of two, values near both ends of the exponent range
(where the FP64 code takes over), a right-hand side that is zero over most of the grid, NaN."""
import numpy as np
import pytest

from oracle import multigrid as mg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


def _cycle(E, r, h, nu1, nu2):
    n = r.shape[0]
    if n == 15:                                  # the level solved exactly (sine basis)
        i = np.arange(1, n + 1).astype(LD)
        S = np.sin(PI * np.outer(i, i) / LD(n + 1)) * np.sqrt(LD(2) / LD(n + 1))
        lam = 4 / (h * h) * np.sin(PI * i / (2 * LD(n + 1))) ** 2
        E[1:-1, 1:-1] = S @ (-(S @ r @ S) / (lam[:, None] + lam[None, :])) @ S
        return
    for _ in range(nu1):
        for c in (0, 1):
            mg.rbgs_half_sweep(E, r, h, c)
    lap = (E[2:, 1:-1] + E[:-2, 1:-1] + E[1:-1, 2:] + E[1:-1, :-2] - 4 * E[1:-1, 1:-1]) / (h * h)
    rc = mg.restrict_fw(r - lap)
    Ec = np.zeros((rc.shape[0] + 2,) * 2, dtype=r.dtype)
    _cycle(Ec, rc, 2 * h, nu1, nu2)
    mg.prolong_add(E, Ec)
    for _ in range(nu2):
        for c in (0, 1):
            mg.rbgs_half_sweep(E, r, h, c)


def _run(n, h, r, e0, nu):
    from paper_2308_11469_gb300 import binding as B
    plan = B.helm_plan_create(2, n, h, 1.0, prec=B.HELM_PREC_FP64)
    e = torch.from_numpy(e0.copy()).cuda()
    B.poisson_vcycle(plan, torch.from_numpy(r).cuda(), e, *nu)
    B.helm_plan_destroy(plan)
    return e.cpu().numpy()


def _error(n, h, r, e0, nu):
    got, num, den = _run(n, h, r, e0, nu), LD(0), LD(0)
    for part in ("real", "imag"):
        E = np.zeros((n + 2, n + 2), dtype=LD)
        E[1:-1, 1:-1] = getattr(e0, part)
        _cycle(E, getattr(r, part).astype(LD), LD(h), *nu)
        num += ((getattr(got, part).astype(LD) - E[1:-1, 1:-1]) ** 2).sum()
        den += (E ** 2).sum()
    return float(np.sqrt(num / den))


def _rough(n, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))


@pytest.mark.parametrize("n", [31, 63, 127, 255, 511, 1023])
@pytest.mark.parametrize("nu", [(0, 1), (2, 2), (4, 0), (1, 3)])
@pytest.mark.parametrize("kind", ["rough", "smooth", "patch"])
def test_error_is_fp64s_own(n, nu, kind):
    h = (1.0 if kind != "smooth" else 0.7) / (n + 1)
    t = np.arange(1, n + 1) / (n + 1)
    if kind == "rough":
        r = _rough(n, n)
    elif kind == "smooth":
        r = np.sin(np.pi * t)[:, None] * np.sin(2 * np.pi * t)[None, :] \
            + 1j * np.exp(-((t[:, None] - .4) ** 2 + (t[None, :] - .6) ** 2) / (2 * .02 ** 2))
    else:
        r = np.zeros((n, n), dtype=complex)
        r[n // 2:n // 2 + 3, n // 3:n // 3 + 5] = 1.0 - 2.0j
    assert _error(n, h, r, np.zeros((n, n), dtype=complex), nu) <= 1.1e-15


@pytest.mark.parametrize("scale", [1e-303, 1e-280, 1e280, 1e303])
def test_exponent_range(scale):
    n = 127
    r = _rough(n, 5)
    a = _run(n, 1.0 / (n + 1), r, np.zeros((n, n), dtype=complex), (2, 2))
    b = _run(n, 1.0 / (n + 1), r * scale, np.zeros((n, n), dtype=complex), (2, 2))
    assert np.linalg.norm(b / scale - a) <= 3e-15 * np.linalg.norm(a)


def test_iterate_larger_than_the_result_and_nan():
    # the iterate (0.01) is 10 times the result and its residual, 8 / h^2 times it, all of what
    # the cycle works on: the roundings of that residual, 2^-53 * 0.01 (N / 20 of it after the
    # solve), are 51 / 10 of the result's own
    n = 1023
    r, e0 = _rough(n, 1), 0.01 * _rough(n, 2)
    assert _error(n, 1.0 / (n + 1), r, e0, (2, 2)) <= 10 * 2.0 ** -53 * 512
    r[7, 9] = complex("nan")
    assert np.isnan(_run(n, 1.0 / (n + 1), r, e0, (2, 2))).any()


@pytest.mark.parametrize("n", [1, 3, 7, 15, 31, 63])
@pytest.mark.parametrize("nu", [(0, 2), (2, 2), (2, 0)])
@pytest.mark.parametrize("kind", ["rough", "smooth", "patch"])
def test_3d_error_is_fp64s_own(n, nu, kind):
    # (a node's last update and correction: 7 + 8 terms, 14 roundings of half an ulp)
    from paper_2308_11469_gb300 import binding as B
    h = (0.7 if kind == "smooth" else 1.0) / (n + 1)
    rng = np.random.default_rng(n)
    if kind == "rough":
        r = rng.standard_normal((n,) * 3) + 1j * rng.standard_normal((n,) * 3)
    elif kind == "smooth":
        s = np.sin(np.pi * np.arange(1, n + 1) / (n + 1))
        r = (1 - 2j) * s[:, None, None] * s[None, :, None] * s[None, None, :]
    else:
        r = np.zeros((n,) * 3, dtype=complex)
        r[n // 2, n // 2, n // 3:n // 3 + 2] = 1.0 - 2.0j
    plan = B.helm_plan_create(3, n, h, 1.0, prec=B.HELM_PREC_FP64)
    e = torch.zeros((n,) * 3, dtype=torch.complex128, device="cuda")
    B.poisson_vcycle(plan, torch.from_numpy(r).cuda(), e, *nu)
    B.helm_plan_destroy(plan)
    got, num, den = e.cpu().numpy(), LD(0), LD(0)
    for part in ("real", "imag"):
        E = np.zeros((n + 2,) * 3, dtype=LD)
        mg.vcycle(E, getattr(r, part).astype(LD), LD(h), *nu)
        num += ((getattr(got, part).astype(LD) - E[1:-1, 1:-1, 1:-1]) ** 2).sum()
        den += (E ** 2).sum()
    assert float(np.sqrt(num / den)) <= 14 * 2.0 ** -53
