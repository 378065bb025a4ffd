"""One cycle of an FP64 annulus solve against the same cycle in extended precision.  The
hole data are zero, so the iterate after a step is the cycle's result itself.  The last update of
a node and the correction under it make at most ten roundings of 2^-53 (half an ulp) of values no
larger than the result's largest; what reaches the result from the levels below is that of an
FP64 cycle (numpy's, on the same data; the order of its sums is another: twice it).

Rough and smooth data, sources on the outer edge alone, and data of the signs that make the
windows' sums as large as they get (every term of every sweep adds: PDE rows -1, EDGE rows h, so
that h^2 rhs and h rhs are equal), at the sweep limits of the fixed-point windows and beside them.
(A second cycle starts from the stored iterate, whose own roundings it amplifies by N^2: its error
is that of the start.)"""
import functools

import numpy as np
import pytest

from oracle import annulus as an
from .test_gpu_annulus_tiles import BAND_SWEEPS, Level

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
LD = np.longdouble


@functools.lru_cache(maxsize=None)
def _levels(N, side):
    out = []
    while N >= 8:
        L = Level(N, 0.15)
        L.h = side / N
        L.g = an.geometry(N, side, 0.15 * side)
        out.append(L)
        N //= 2
    return out


def _solve(A, b):
    """Gaussian elimination with partial pivots, in A's precision."""
    A, b, n = A.copy(), b.copy(), len(A)
    for c in range(n):
        p = c + int(np.argmax(np.abs(A[c:, c])))
        A[[c, p]], b[[c, p]] = A[[p, c]], b[[p, c]]
        f = A[c + 1:, c] / A[c, c]
        A[c + 1:] -= f[:, None] * A[c]
        b[c + 1:] -= f * b[c]
    for c in range(n - 1, -1, -1):
        b[c] = (b[c] - A[c, c + 1:] @ b[c + 1:]) / A[c, c]
    return b


def _cycle(levels, l, e, r, nu1, nu2):
    L, t = levels[l], e.dtype.type
    h = t(L.h)
    if l + 1 == len(levels):
        e[:] = 0
        e[~L.hole] = _solve(an.operator(L.g).toarray().real.astype(t), r[~L.hole])
        return

    def sweep(mask=None):
        for colour in (0, 1):
            new = np.where(L.pde, (L.nbrs(e) - h * h * r) / 4, L.inward(e) + h * r)
            at = (L.odd == colour) & ~L.hole
            e[at if mask is None else at & mask] = new[at if mask is None else at & mask]
    C = levels[l + 1]
    for _ in range(nu1):
        sweep()
    res = np.where(L.pde, r - (L.nbrs(e) - 4 * e) / (h * h), r - (e - L.inward(e)) / h)
    res = np.where(L.hole, t(0), res)
    w = np.zeros_like(res)
    for a in (-1, 0, 1):
        for b in (-1, 0, 1):
            w[1:-1, 1:-1] += t((2 - abs(a)) * (2 - abs(b))) / 16 * res[1 + a:L.N + a, 1 + b:L.N + b]
    ec = np.zeros((C.N + 1, C.N + 1), dtype=e.dtype)
    _cycle(levels, l + 1, ec, np.where(C.pde, w[::2, ::2], np.where(C.edge, res[::2, ::2], t(0))), nu1, nu2)
    P = np.zeros_like(e)
    P[::2, ::2] = ec
    P[1::2, ::2] = (ec[:-1] + ec[1:]) / 2
    P[:, 1::2] = (P[:, :-1:2] + P[:, 2::2]) / 2
    e += np.where(L.hole, t(0), P)
    for _ in range(BAND_SWEEPS):
        sweep(L.ring)
    for _ in range(nu2):
        sweep()


@pytest.mark.parametrize("N,side", [(64, 1.0), (128, 1.0), (128, 0.7), (256, 1.0)])
@pytest.mark.parametrize("data", ["rough", "smooth", "edge", "largest"])
@pytest.mark.parametrize("cycle", [(2, 2), (2, 4), (0, 1), (1, 4), (3, 2)])
def test_error_is_fp64s_own(N, side, data, cycle):
    from paper_2308_11469_gb300 import binding as B
    levels = _levels(N, side)
    L = levels[0]
    x = np.arange(N + 1) / N
    if data == "rough":
        d = np.random.default_rng(N).standard_normal((N + 1, N + 1))
    elif data == "smooth":
        d = np.sin(2 * np.pi * x)[:, None] * np.cos(3 * x)[None, :]
    elif data == "edge":
        d = np.where(L.edge, 1.0, 0.0)
    else:
        d = np.where(L.edge, L.h, -1.0)
    d = np.where(L.hole, 0.0, d)
    plan = B.helm_annulus_create(N, side, 0.15 * side, 0.0, B.HELM_PREC_FP64)
    B.helm_annulus_set_cycle(plan, *cycle, 1)
    dd = torch.from_numpy(d * (1.0 - 0.5j)).cuda()
    u = torch.empty_like(dd)
    _, it, _ = B.helm_annulus_solve(plan, dd, u, 0.0, 1)
    B.helm_annulus_destroy(plan)
    assert it == 1
    got = u.cpu().numpy()
    e, E = np.zeros_like(d), np.zeros(d.shape, dtype=LD)
    _cycle(levels, 0, e, d, *cycle)
    _cycle(levels, 0, E, d.astype(LD), *cycle)
    norm = float(np.sqrt((E * E).sum()))
    own = float(np.sqrt(((e - E) ** 2).sum())) / norm
    for part, s in ((got.real, 1.0), (got.imag, -0.5)):
        err = float(np.sqrt(((part.astype(LD) / s - E) ** 2).sum())) / norm
        assert err <= 2.0 * own + 10 * 2.0 ** -53, (err * 2.0 ** 53, own * 2.0 ** 53)
