"""The FP64 annulus cycle's fixed-point windows against the plain numpy cycle: mesh widths that
are no powers of two, windows of zeros beside an impulse (a corner, an edge node, a tile
corner), sweep counts on both sides of the fixed-point limits.

Tolerance: as for the cycle's residuals, 2^-53 * 0.4 N^2 of the iterate for each step."""
import functools

import numpy as np
import pytest

from oracle import annulus as an
from .test_gpu_annulus_tiles import Level, _cycle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@functools.lru_cache(maxsize=None)
def _levels(N, side):
    out = []
    while N >= 8:
        L = Level(N, 0.15)
        L.h, L.g = side / N, an.geometry(N, side, 0.15 * side)
        assert (L.g.typ == an.geometry(N, 1.0, 0.15).typ).all()
        out.append(L)
        N //= 2
    return out


@pytest.mark.parametrize("N,side", [(128, 1.0), (128, 3.0), (256, 0.7)])
@pytest.mark.parametrize("data", ["rough", "corner", "edge", "tile"])
@pytest.mark.parametrize("cycle", [(2, 2, 1), (1, 4, 2), (3, 5, 1)])
def test_iterates_match_the_numpy_cycle(N, side, data, cycle):
    from paper_2308_11469_gb300 import binding as B
    k, steps = 0.8 / side, 2
    levels = _levels(N, side)
    L = levels[0]
    d = np.zeros((N + 1, N + 1), dtype=complex)
    if data == "rough":
        rng = np.random.default_rng(N)
        d = rng.standard_normal(d.shape) + 1j * rng.standard_normal(d.shape)
    else:
        d[{"corner": (0, N), "edge": (N, 33), "tile": (32, 63)}[data]] = 1.0 - 0.5j
    U = np.where(L.hole, d, 0)
    for _ in range(steps):
        lap = (L.nbrs(U) - 4.0 * U) / L.h ** 2 + k * k * U
        r = np.where(L.pde, d - lap, d - ((U - L.inward(U)) / L.h - 1j * k * U))
        r = np.where(L.hole, 0, r)
        e = np.zeros_like(U)
        for _ in range(cycle[2]):
            _cycle(levels, 0, e, r, cycle[0], cycle[1])
        U = U + e
    plan = B.helm_annulus_create(N, side, 0.15 * side, k, B.HELM_PREC_FP64)
    B.helm_annulus_set_cycle(plan, *cycle)
    dd = torch.from_numpy(np.ascontiguousarray(d)).cuda()
    u = torch.empty_like(dd)
    _, it, _ = B.helm_annulus_solve(plan, dd, u, 0.0, steps)
    B.helm_annulus_destroy(plan)
    assert it == steps
    err = np.linalg.norm(u.cpu().numpy() - U) / np.linalg.norm(U)
    assert err <= steps * 2.0 ** -53 * 0.4 * N * N, err


def test_iterates_beyond_the_scale():
    """Hole data of 2^1000 (mesh widths that keep the residuals finite): windows and the
    residual's tiles hold values that have no fixed-point scale and are evaluated in FP64."""
    from paper_2308_11469_gb300 import binding as B
    N, side = 128, 2.0 ** 497
    levels = _levels(N, side)
    L = levels[0]
    x = np.arange(N + 1) / N
    d = np.where(L.hole, 2.0 ** 1000 * (1.0 + 0.5 * x[:, None] + 0.25j * x[None, :]), 0)
    r = np.where(L.pde, -((L.nbrs(d) - 4.0 * d) / L.h ** 2), 0)
    e = np.zeros_like(d)
    _cycle(levels, 0, e, r, 2, 2)
    plan = B.helm_annulus_create(N, side, 0.15 * side, 0.0, B.HELM_PREC_FP64)
    dd = torch.from_numpy(d).cuda()
    u = torch.empty_like(dd)
    _, it, hist = B.helm_annulus_solve(plan, dd, u, 0.0, 1)
    B.helm_annulus_destroy(plan)
    assert it == 1 and np.isfinite(hist).all()
    U = (d + e) * 2.0 ** -1000
    err = np.linalg.norm(u.cpu().numpy() * 2.0 ** -1000 - U) / np.linalg.norm(U)
    assert err <= 2.0 ** -53 * 0.4 * N * N, err
