"""The annulus cycle's kernels (tiles of 16 and 32 nodes, the one-CTA tail) against the same
cycle written in plain numpy on full grids: the first FP64 residual norms of the outer
iteration, for sweep counts from 0 to 8 (window widths), several cycles a step (a nonzero
starting iterate) and holes whose ring meets tile corners.

Tolerance: the two evaluate the same FP64 operations up to their order; a rounding of the
correction (2^-53) reaches the residual through 8 / h^2 against the correction's own
lambda ~ 20, i.e. 2^-53 * 0.4 N^2 = 1.2e-11 at N = 512 before any averaging over nodes."""
import functools

import numpy as np
import pytest

from oracle import annulus as an

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
BAND, BAND_SWEEPS = 4, 4


class Level:
    def __init__(self, N, hole):
        self.N, self.h = N, 1.0 / N
        self.g = an.geometry(N, 1.0, hole)
        t = self.g.typ
        self.pde, self.edge, self.hole = t == an.PDE, t == an.EDGE, t == an.HOLE
        i = np.arange(N + 1)
        self.odd = (i[:, None] + i[None, :]) % 2
        box = np.flatnonzero(self.hole.any(axis=1))
        b0, b1 = max(1, box[0] - BAND), min(N - 1, box[-1] + BAND)
        ring = np.zeros_like(self.pde)
        ring[b0:b1 + 1, b0:b1 + 1] = True
        self.ring = ring & self.pde

    def inward(self, e):
        N, m = self.N, np.zeros_like(e)
        c = np.zeros(e.shape)
        for sl, src in (((0, slice(None)), (1, slice(None))), ((N, slice(None)), (N - 1, slice(None))),
                        ((slice(None), 0), (slice(None), 1)), ((slice(None), N), (slice(None), N - 1))):
            m[sl] += e[src]
            c[sl] += 1
        return np.where(self.edge, m / np.maximum(c, 1), 0)

    def nbrs(self, e):
        s = np.zeros_like(e)
        s[1:-1, 1:-1] = (e[:-2, 1:-1] + e[2:, 1:-1]) + (e[1:-1, :-2] + e[1:-1, 2:])
        return s

    def sweep(self, e, r, mask=None):
        for colour in (0, 1):
            new = np.where(self.pde, (self.nbrs(e) - self.h ** 2 * r) / 4.0, self.inward(e) + self.h * r)
            at = (self.odd == colour) & ~self.hole
            if mask is not None:
                at &= mask
            e[at] = new[at]

    def residual(self, e, r):
        res = np.where(self.pde, r - (self.nbrs(e) - 4.0 * e) / self.h ** 2, r - (e - self.inward(e)) / self.h)
        return np.where(self.hole, 0, res)


def _cycle(levels, l, e, r, nu1, nu2):
    L = levels[l]
    if l + 1 == len(levels):
        A = an.operator(L.g).toarray()
        e[:] = 0
        e[~L.hole] = np.linalg.solve(A, r[~L.hole])
        return
    C = levels[l + 1]
    for _ in range(nu1):
        L.sweep(e, r)
    res = L.residual(e, r)
    w = np.zeros_like(res)
    for a in (-1, 0, 1):
        for b in (-1, 0, 1):
            w[1:-1, 1:-1] += (2 - abs(a)) * (2 - abs(b)) / 16.0 * res[1 + a:L.N + a, 1 + b:L.N + b]
    rc = np.where(C.pde, w[::2, ::2], np.where(C.edge, res[::2, ::2], 0))
    ec = np.zeros((C.N + 1, C.N + 1), dtype=e.dtype)
    _cycle(levels, l + 1, ec, rc, nu1, nu2)
    P = np.zeros_like(e)
    P[::2, ::2] = ec
    P[1::2, ::2] = (ec[:-1] + ec[1:]) / 2
    P[:, 1::2] = (P[:, :-1:2] + P[:, 2::2]) / 2
    e += np.where(L.hole, 0, P)
    for _ in range(BAND_SWEEPS):
        L.sweep(e, r, L.ring)
    for _ in range(nu2):
        L.sweep(e, r)


@functools.lru_cache(maxsize=None)
def _levels(N, hole):
    out = []
    while N >= 8:
        out.append(Level(N, hole))
        N //= 2
    return out


@pytest.mark.parametrize("N,hole", [(16, 0.15), (32, 0.3), (64, 0.15), (128, 0.2), (512, 0.15)])
@pytest.mark.parametrize("cycle", [(2, 2, 1), (0, 3, 2), (3, 0, 1), (1, 2, 2), (8, 8, 1)])
def test_first_residuals_match_the_numpy_cycle(N, hole, cycle):
    from paper_2308_11469_gb300 import binding as B
    k, steps = 0.8, 3
    levels = _levels(N, hole)
    L = levels[0]
    rng = np.random.default_rng(N)
    data = rng.standard_normal((N + 1, N + 1)) + 1j * rng.standard_normal((N + 1, N + 1))
    U = np.where(L.hole, data, 0)
    want = []
    for s in range(steps + 1):
        lap = (L.nbrs(U) - 4.0 * U) / L.h ** 2 + k * k * U
        r = np.where(L.pde, data - lap, data - ((U - L.inward(U)) / L.h - 1j * k * U))
        r = np.where(L.hole, 0, r)
        want.append(np.linalg.norm(r))
        e = np.zeros_like(U)
        for _ in range(cycle[2]):
            _cycle(levels, 0, e, r, cycle[0], cycle[1])
        U = U + e
    plan = B.helm_annulus_create(N, 1.0, hole, k, B.HELM_PREC_FP64)
    B.helm_annulus_set_cycle(plan, *cycle)
    d = torch.from_numpy(np.ascontiguousarray(data)).cuda()
    u = torch.empty_like(d)
    st, it, hist = B.helm_annulus_solve(plan, d, u, 0.0, steps)
    B.helm_annulus_destroy(plan)
    assert it == steps
    np.testing.assert_allclose(hist, np.array(want) / want[0], rtol=1.2e-11 * max(1.0, (N / 512) ** 2))
