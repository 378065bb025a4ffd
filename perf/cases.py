"""Timed cases of the library's public entry points over the range that they are used in.

Every case is a call that a program of this framework makes: a cavity solve through a plan
(``helm_solve``), a single multigrid cycle as a preconditioner (``poisson_vcycle``), a batch
run to completion, a burst of requests through the server, or the annular scattering problem.
Grids of this library are n = 2^m - 1 nodes per axis (cavity) or 2^m intervals (annulus), so
the odd sizes are all there are.  Sizes, tolerances, schedules and wave numbers are those of
the benchmark's legs, of the served stream and of the GPU tests: V(0,1) in 2D and V(0,2) in 3D
are what the autotuner settles on, V(2,2) is the default of a plan that is not tuned.

``prepare`` makes what such a program holds before the call (device arrays and the plan, batch
or server); ``run`` is one pass; ``exact`` restates the answer in torch, in 64 bits: the
discrete solution by sine transforms (cavity) or by block elimination (annulus), the cycle by
its textbook components.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2308_11469_gb300 import binding as B
from paper_2308_11469_gb300 import serve

MIXED, FP64 = "mixed", "fp64"
PREC = {MIXED: B.HELM_PREC_MIXED, FP64: B.HELM_PREC_FP64}


def _dev():
    return torch.device("cuda", torch.cuda.current_device())


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest call: one default cycle as a preconditioner on the 63^2 grid
        {"name": "vcycle 2D 63 mixed", "kind": "vcycle", "D": 2, "n": 63, "prec": MIXED, "nu1": 2, "nu2": 2},
        # the 63^2 plane-wave cavity of the benchmark, a plan as created (not tuned), both precisions
        {"name": "solve 2D 63 mixed", "kind": "solve", "D": 2, "n": 63, "prec": MIXED, "nu1": 2, "nu2": 2,
         "k": 2.0, "p": 0.0, "wall": True, "tol": 1e-10},
        {"name": "solve 2D 63 fp64", "kind": "solve", "D": 2, "n": 63, "prec": FP64, "nu1": 2, "nu2": 2,
         "k": 2.0, "p": 0.0, "wall": True, "tol": 1e-10},
        # a mid-sized damped cavity (p > 0) with wall data on the default schedule
        {"name": "solve 2D 511 mixed damped", "kind": "solve", "D": 2, "n": 511, "prec": MIXED, "nu1": 2, "nu2": 2,
         "k": 3.0, "p": 2.0, "wall": True, "tol": 1e-8},
        # the headline: four 1023^2 Gaussian cavities, k = 1..4, one batch in two lanes
        {"name": "batch 2D 1023 x4 mixed", "kind": "sweep", "n": 1023, "count": 4, "kmax": 4.0},
        # its plain FP64 form, one solve alone
        {"name": "solve 2D 1023 fp64", "kind": "solve", "D": 2, "n": 1023, "prec": FP64, "nu1": 0, "nu2": 1,
         "k": 2.0, "p": 0.0, "wall": False, "tol": 1e-8},
        # the 255^3 cube with wall data, and a mid-sized cube in FP64
        {"name": "solve 3D 255 mixed", "kind": "solve", "D": 3, "n": 255, "prec": MIXED, "nu1": 0, "nu2": 2,
         "k": 4.0, "p": 0.0, "wall": True, "tol": 1e-8},
        {"name": "solve 3D 127 fp64", "kind": "solve", "D": 3, "n": 127, "prec": FP64, "nu1": 0, "nu2": 2,
         "k": 3.0, "p": 0.0, "wall": True, "tol": 1e-8},
        # 512 uneven 2D cavities, one batch to completion
        {"name": "batch 2D x512 mixed", "kind": "batch", "count": 512, "mix": 4},
        # a burst of mixed 2D / 3D requests through the continuous-batching server
        {"name": "serve x16 mixed", "kind": "serve", "count": 16, "mix": 5},
        # the annular scattering problem: the benchmark's grid mixed, a smaller one in FP64
        {"name": "annulus 1024 mixed", "kind": "annulus", "N": 1024, "prec": MIXED, "hole": 0.15, "k": 0.8,
         "tol": 1e-8},
        {"name": "annulus 256 fp64", "kind": "annulus", "N": 256, "prec": FP64, "hole": 0.15, "k": 0.8,
         "tol": 1e-8},
    ]


def _kmax(D, n):
    return math.sqrt(D * 4.0) * (n + 1) * math.sin(math.pi / (2.0 * (n + 1)))


def draw(rng: random.Random):
    kind = rng.choice(["vcycle", "solve", "solve", "solve", "sweep", "batch", "serve", "annulus", "annulus"])
    if kind == "vcycle":
        D = rng.choice([2, 3])
        nu1, nu2 = rng.choice([(2, 2), (1, 1), (0, 1), (0, 2), (2, 1)])
        return {"kind": kind, "D": D, "n": 2 ** (rng.randint(5, 11) if D == 2 else rng.randint(4, 8)) - 1,
                "prec": rng.choice([MIXED, FP64]), "nu1": nu1, "nu2": nu2}
    if kind == "solve":
        D, prec = rng.choice([2, 2, 3]), rng.choice([MIXED, MIXED, FP64])
        hi = {(2, MIXED): 11, (2, FP64): 10, (3, MIXED): 8, (3, FP64): 7}[D, prec]
        n = 2 ** rng.randint(5 if D == 2 else 4, hi) - 1
        nu1, nu2 = rng.choice([(2, 2), (0, 1) if D == 2 else (0, 2)])
        return {"kind": kind, "D": D, "n": n, "prec": prec, "nu1": nu1, "nu2": nu2,
                "k": round(rng.uniform(0.5, 0.74 * _kmax(D, n)), 4), "p": rng.choice([0.0, 0.0, 2.0]),
                "wall": rng.choice([True, False]), "tol": rng.choice([1e-8, 1e-8, 1e-10]) if n <= 511 else 1e-8}
    if kind == "sweep":
        return {"kind": kind, "n": 2 ** rng.randint(7, 10) - 1, "count": rng.randint(2, 6),
                "kmax": round(rng.uniform(2.0, 4.0), 4)}
    if kind == "batch":
        return {"kind": kind, "count": int(2 ** rng.uniform(4, 9)), "mix": rng.randint(6, 10 ** 6)}
    if kind == "serve":
        most = work(next(c for c in listed() if c["kind"] == kind))
        while True:                            # a mix may hold more large cubes than the listed one
            case = {"kind": kind, "count": rng.randint(4, 16), "mix": rng.randint(6, 10 ** 6)}
            if all(v <= most[m] for m, v in work(case).items()):
                return case
    prec = rng.choice([MIXED, FP64])
    return {"kind": kind, "N": 2 ** rng.randint(5, 10 if prec == MIXED else 9), "prec": prec,
            "hole": 0.15, "k": round(rng.uniform(0.3, 0.85), 4), "tol": 1e-8}   # the hole of the method's own example


# ------------------------------------------------------------------ inputs

def _axis(n, h, dev):
    return torch.arange(n + 2, dtype=torch.float64, device=dev) * h


def _plane_wave(D, n, h, kappa, d, dev):
    """exp(i kappa d.x) on the padded grid."""
    t = _axis(n, h, dev)
    ph = [torch.polar(torch.ones_like(t), kappa * float(d[a]) * t) for a in range(D)]
    if D == 2:
        return (ph[1][:, None] * ph[0][None, :]).contiguous()
    return (ph[2][:, None, None] * ph[1][None, :, None] * ph[0][None, None, :]).contiguous()


def _gaussians(D, n, h, rng, dev, width=0.02):
    """Eight Gaussians with seeded centres and complex amplitudes, on the interior."""
    c = rng.uniform(0.2, 0.8, size=(8, D))
    a = rng.standard_normal(8) + 1j * rng.standard_normal(8)
    t = _axis(n, h, dev)[1:-1]
    one = torch.exp(-((t[None, None, :] - torch.from_numpy(c).to(dev)[:, :, None]) ** 2) / (2.0 * width * width))
    one = one.to(torch.complex128)
    amp = torch.from_numpy(a).to(dev)
    if D == 2:
        return torch.einsum("g,gy,gx->yx", amp, one[:, 1], one[:, 0]).contiguous()
    return torch.einsum("g,gz,gy,gx->zyx", amp, one[:, 2], one[:, 1], one[:, 0]).contiguous()


def _cavity(D, n, k, wall, rng, dev):
    """(f, g): a plane wave on the wall (with a sine source in 3D), or Gaussian sources."""
    h = 1.0 / (n + 1)
    if not wall:
        return _gaussians(D, n, h, rng, dev), torch.zeros((n + 2,) * D, dtype=torch.complex128, device=dev)
    d = rng.standard_normal(D)
    d /= np.linalg.norm(d)
    g = _plane_wave(D, n, h, k, d, dev)
    if D == 2:
        return torch.zeros((n, n), dtype=torch.complex128, device=dev), g
    t = math.pi * _axis(n, h, dev)[1:-1]
    f = torch.sin(t)[:, None, None] * torch.sin(2 * t)[None, :, None] * torch.sin(t)[None, None, :]
    return f.to(torch.complex128).contiguous(), g


def _batch_mix(case):
    """[(D, n, k, wall)] of a batch: sizes and wave numbers of the benchmark's uneven batch."""
    rng = np.random.default_rng(case["mix"])
    ns = rng.choice([63, 127, 255, 511], size=case["count"], p=[0.4, 0.3, 0.2, 0.1])
    us = rng.uniform(0.0, 1.0, size=case["count"])
    return [(2, int(n), 0.5 + float(u) * (0.9 * _kmax(2, int(n)) - 0.5), False) for n, u in zip(ns, us)]


def _serve_mix(case):
    """[(D, n, k, wall)] of a burst: the served stream's sizes (70 % 2D), k and kinds of data."""
    rng = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["count"]):
        D = 2 if rng.uniform() < 0.7 else 3
        n = int(rng.choice([127, 255, 511, 1023, 2047] if D == 2 else [63, 127, 255]))
        out.append((D, n, 0.5 + float(rng.uniform()) * (0.9 * _kmax(D, n) - 0.5), bool(rng.uniform() < 0.5)))
    return out


def _sweep_mix(case):
    return [(2, case["n"], case["kmax"] * (i + 1) / case["count"], False) for i in range(case["count"])]


_MIX = {"batch": _batch_mix, "serve": _serve_mix, "sweep": _sweep_mix}


def _data(case, seed, dev):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "vcycle":
        dt = torch.complex64 if case["prec"] == MIXED else torch.complex128
        gen = torch.Generator(device=dev).manual_seed(seed)
        re, im = (torch.randn((case["n"],) * case["D"], generator=gen, device=dev, dtype=torch.float64)
                  for _ in range(2))
        return torch.complex(re, im).to(dt).contiguous()
    if kind == "solve":
        return _cavity(case["D"], case["n"], case["k"], case["wall"], rng, dev)
    if kind == "annulus":
        N, c, k = case["N"], case["hole"], case["k"]
        th = float(rng.uniform(0.0, 2.0 * math.pi))
        x = -0.5 + torch.arange(N + 1, dtype=torch.float64, device=dev) / N
        hole = x.abs() <= c + 1e-9
        ph = torch.polar(torch.ones_like(x), -k * math.cos(th) * x)[:, None] * \
            torch.polar(torch.ones_like(x), -k * math.sin(th) * x)[None, :]
        return torch.where(hole[:, None] & hole[None, :], -ph, torch.zeros_like(ph)).contiguous()
    return [(D, n, k) + _cavity(D, n, k, wall, rng, dev) for D, n, k, wall in _MIX[kind](case)]


# ------------------------------------------------------------------ what a program holds, and one pass

def prepare(case, seed):
    dev, kind = _dev(), case["kind"]
    s = {"case": case}
    data = _data(case, seed, dev)
    if kind == "vcycle":
        n, D = case["n"], case["D"]
        s["plan"] = B.helm_plan_create(D, n, 1.0 / (n + 1), 1.0, prec=PREC[case["prec"]])
        s["rhs"], s["e"] = data, torch.zeros_like(data)
    elif kind == "solve":
        n, D = case["n"], case["D"]
        s["plan"] = B.helm_plan_create(D, n, 1.0 / (n + 1), case["k"], prec=PREC[case["prec"]])
        B.helm_plan_set_cycle(s["plan"], case["nu1"], case["nu2"], 1)
        if case["p"]:
            B.helm_plan_set_cavity(s["plan"], case["k"] ** 2, case["p"])
        s["f"], s["g"] = data
        s["u"] = torch.zeros_like(s["g"])
    elif kind == "annulus":
        s["plan"] = B.helm_annulus_create(case["N"], 1.0, case["hole"], case["k"], PREC[case["prec"]])
        s["data"], s["u"] = data, torch.zeros_like(data)
    else:
        s["U"] = torch.zeros(sum(g.numel() for *_, g in data), dtype=torch.complex128, device=dev)
        s["jobs"], off = [], 0
        for D, n, k, f, g in data:
            s["jobs"].append((D, n, 1.0 / (n + 1), k, f, g, s["U"][off:off + g.numel()].view(g.shape)))
            off += g.numel()
        if kind == "serve":
            s["server"] = serve.Server(120 << 30, chunk=4, class_schedules={2: (0, 1, 1), 3: (0, 2, 1)})
        else:
            s["batch"] = B.helm_batch_create(0)
            B.helm_batch_set_cycle(s["batch"], 0, 1, 1)
            if kind == "sweep":                    # longest solve first, alone in its lane
                B.helm_batch_set_lanes(s["batch"], 2)
                s["jobs"].reverse()
    return s


def _whole(hist):
    """The history in an array whose length does not depend on the data (the rest zero)."""
    out = np.zeros(256)
    out[:hist.size] = hist
    return out


def run(s):
    kind = s["case"]["kind"]
    if kind == "vcycle":
        s["e"].zero_()
        B.poisson_vcycle(s["plan"], s["rhs"], s["e"], s["case"]["nu1"], s["case"]["nu2"])
        return {"e": s["e"]}
    if kind == "solve":
        s["u"].zero_()
        st, it, hist = B.helm_solve(s["plan"], s["f"], s["g"], s["u"], s["case"]["tol"], 255)
        return {"u": s["u"], "status": st, "iters": it, "relres": _whole(hist)}
    if kind == "annulus":
        st, it, hist = B.helm_annulus_solve(s["plan"], s["data"], s["u"], s["case"]["tol"], 255)
        return {"u": s["u"], "status": st, "iters": it, "relres": _whole(hist)}
    s["U"].zero_()
    if kind == "serve":
        srv = s["server"]
        done = srv.run([serve.Job(i, *j, 0.0) for i, j in enumerate(s["jobs"])], realtime=False)
        res = [(j.status, j.iters) for j in sorted(done, key=lambda j: j.rid)]
        done.clear()
    else:
        tickets = B.helm_batch_submit_many(s["batch"], s["jobs"], B.HELM_PREC_MIXED, 1e-8, 3000)
        B.helm_batch_step(s["batch"], 0)
        res = [(st, it) for _, st, it in B.helm_batch_poll_many(s["batch"], tickets)]
    return {"u": s["U"], "status": np.array([r[0] for r in res]), "iters": np.array([r[1] for r in res])}


# ------------------------------------------------------------------ what a pass cannot do without

def _solve_work(D, n, k, p, tol, nu):
    """Source, the wall's nodes and the solution once; the outer steps that exact inner solves
    take, each a residual (16 flops a node) and a cycle of nu sweeps and two transfers."""
    rho = math.hypot(k * k, p) / _kmax(D, n) ** 2
    steps = max(1.0, math.log(tol) / math.log(rho))
    pts = n ** D
    cycle = (nu * 2 * (2 * D + 2) + 2 * (2 * 2 ** D)) * 2 ** D / (2 ** D - 1)
    return 16.0 * pts + 16.0 * ((n + 2) ** D - pts) + 16.0 * (n + 2) ** D, steps * pts * (16.0 + cycle)


def work(case):
    kind = case["kind"]
    if kind == "vcycle":
        pts, el = case["n"] ** case["D"], 8.0 if case["prec"] == MIXED else 16.0
        D, nu = case["D"], case["nu1"] + case["nu2"]
        return {"bytes": 2 * el * pts,
                "flops": pts * (nu * 2 * (2 * D + 2) + 2 * (2 * 2 ** D)) * 2 ** D / (2 ** D - 1)}
    if kind == "solve":
        b, f = _solve_work(case["D"], case["n"], case["k"], case["p"], case["tol"], case["nu1"] + case["nu2"])
    elif kind == "annulus":
        pts = (case["N"] + 1) ** 2
        b, f = 32.0 * pts, 50.0 * pts * (16.0 + (4 * 2 * 6 + 16) * 4 / 3)
    else:
        rows = [_solve_work(D, n, k, 0.0, 1e-8, 1 if D == 2 else 2) for D, n, k, _ in _MIX[kind](case)]
        b, f = sum(r[0] for r in rows), sum(r[1] for r in rows)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the same in 64 bits

def _sine(n, dev):
    """The orthonormal sine basis of the 1-D Dirichlet Laplacian (symmetric)."""
    i = torch.arange(1, n + 1, dtype=torch.float64, device=dev)
    # the argument reduced exactly before the sine: i j mod 2 (n + 1)
    m = torch.remainder(i[:, None] * i[None, :], 2.0 * (n + 1))
    return math.sqrt(2.0 / (n + 1)) * torch.sin(math.pi / (n + 1) * m)


def _along(S, a):
    """S applied along every axis of the complex array a."""
    for d in range(a.dim()):
        a = torch.movedim(a, d, -1)
        a = torch.complex(a.real @ S, a.imag @ S)
        a = torch.movedim(a, -1, d)
    return a


def _helmholtz(f, g, k, p):
    """Padded u with (Delta_h + k^2 + i p) u = f inside and u = g on the wall."""
    D, n = f.dim(), f.shape[0]
    h = 1.0 / (n + 1)
    inner = (slice(1, -1),) * D
    u = g.clone()
    u[inner] = 0
    b = f.clone()
    for a in range(D):                     # wall neighbours to the right-hand side
        for side, edge in ((0, 0), (-1, n - 1)):
            src = list(inner)
            src[a] = side
            dst = [slice(None)] * D
            dst[a] = edge
            b[tuple(dst)] -= u[tuple(src)] / (h * h)
    S = _sine(n, f.device)
    lam = 4.0 / (h * h) * torch.sin(math.pi / (2.0 * (n + 1)) *
                                    torch.arange(1, n + 1, dtype=torch.float64, device=f.device)) ** 2
    tot = torch.zeros((n,) * D, dtype=torch.float64, device=f.device)
    for a in range(D):
        tot = tot + lam.view([n if d == a else 1 for d in range(D)])
    u[inner] = _along(S, _along(S, b) / (k * k + 1j * p - tot))
    return u


def _shifted(E, a, s):
    idx = [slice(1, -1)] * E.dim()
    idx[a] = slice(1 + s, E.shape[a] - 1 + s)
    return E[tuple(idx)]


def _cycle(E, r, h, nu1, nu2, exact_n):
    """One V(nu1, nu2) cycle on the padded iterate E, in place; level exact_n solved directly."""
    D, n = r.dim(), r.shape[0]
    inner = (slice(1, -1),) * D
    if n == exact_n:
        lam = 4.0 / (h * h) * torch.sin(math.pi / (2.0 * (n + 1)) *
                                        torch.arange(1, n + 1, dtype=torch.float64, device=r.device)) ** 2
        tot = sum(lam.view([n if d == a else 1 for d in range(D)]) for a in range(D))
        S = _sine(n, r.device)
        E[inner] = _along(S, -_along(S, r) / tot)
        return
    if n == 1:
        E[inner] = -(h * h) * r / (2.0 * D)
        return
    i = torch.arange(1, n + 1, device=r.device)
    par = sum(i.view([n if d == a else 1 for d in range(D)]) for a in range(D)) % 2

    def sweep():
        for colour in (0, 1):
            nb = sum(_shifted(E, a, s) for a in range(D) for s in (1, -1))
            E[inner] = torch.where(par == colour, (nb - (h * h) * r) / (2.0 * D), E[inner])
    for _ in range(nu1):
        sweep()
    lap = (sum(_shifted(E, a, s) for a in range(D) for s in (1, -1)) - 2 * D * E[inner]) / (h * h)
    P = torch.zeros_like(E)
    P[inner] = r - lap
    for a in range(D):                     # [1 2 1] / 4 along the axis, at the even nodes
        lo, mid, hi = ([slice(None)] * D for _ in range(3))
        lo[a], mid[a], hi[a] = slice(1, n - 1, 2), slice(2, n, 2), slice(3, n + 1, 2)
        P = (P[tuple(lo)] + 2.0 * P[tuple(mid)] + P[tuple(hi)]) / 4.0
        pad = [0, 0] * D
        pad[2 * (D - 1 - a)] = pad[2 * (D - 1 - a) + 1] = 1
        P = torch.complex(torch.nn.functional.pad(P.real, pad), torch.nn.functional.pad(P.imag, pad))
    Ec = torch.zeros_like(P)
    _cycle(Ec, P[inner].contiguous(), 2.0 * h, nu1, nu2, exact_n)
    for a in range(D):                     # linear interpolation along the axis
        shape = list(Ec.shape)
        m = shape[a]
        shape[a] = 2 * m - 1
        R = torch.zeros(shape, dtype=Ec.dtype, device=Ec.device)
        ev, od, q0, q1 = ([slice(None)] * D for _ in range(4))
        ev[a], od[a], q0[a], q1[a] = slice(0, None, 2), slice(1, None, 2), slice(0, -1), slice(1, None)
        R[tuple(ev)] = Ec
        R[tuple(od)] = 0.5 * (Ec[tuple(q0)] + Ec[tuple(q1)])
        Ec = R
    E[inner] += Ec[inner]
    for _ in range(nu2):
        sweep()


def _annulus(data, c, k):
    """u of the annular problem by block elimination over the grid's rows (x = const)."""
    N, dev = data.shape[0] - 1, data.device
    h = 1.0 / N
    x = -0.5 + h * torch.arange(N + 1, dtype=torch.float64, device=dev)
    hx = x.abs() <= c + 1e-9
    z = torch.zeros(N + 1, dtype=torch.complex128, device=dev)
    one = torch.ones_like(z)
    X, Y = [], []                          # S_i^-1 C_i and S_i^-1 b_i of the eliminated rows
    for i in range(N + 1):
        hole = hx & bool(hx[i])
        # PDE rows; the first and last node of the row are edge nodes
        dia, up, dn = (-4.0 / (h * h) + k * k) * one, one / (h * h), one / (h * h)
        lo, hi = one / (h * h), one / (h * h)                     # towards i - 1, i + 1
        ends = (0, N)
        if i in ends:
            dia, up, dn = (1.0 / h - 1j * k) * one, 0 * one, 0 * one
            lo, hi = (0 * one, -one / h) if i == 0 else (-one / h, 0 * one)
        for j in ends:
            w = 0.5 if i in ends else 1.0
            dia[j] = 1.0 / h - 1j * k
            up[j], dn[j] = (-w / h, 0) if j == 0 else (0, -w / h)
            lo[j], hi[j] = w * lo[j] if i in ends else 0, w * hi[j] if i in ends else 0
        dia = torch.where(hole, one, dia)
        up, dn, lo, hi = (torch.where(hole, z, v) for v in (up, dn, lo, hi))
        S = torch.diag(dia) + torch.diag(up[:-1], 1) + torch.diag(dn[1:], -1)
        b = data[i].clone()
        if i:
            S = S - lo[:, None] * X[-1]
            b = b - lo * Y[-1]
        inv = torch.linalg.inv(S)
        X.append(inv * hi[None, :])
        Y.append(inv @ b)
    u = torch.empty_like(data)
    u[N] = Y[N]
    for i in range(N - 1, -1, -1):
        u[i] = Y[i] - X[i] @ u[i + 1]
    return u


def exact(case, seed):
    dev, kind = _dev(), case["kind"]
    data = _data(case, seed, dev)
    if kind == "vcycle":
        D, n = case["D"], case["n"]
        top = {(2, MIXED): 31, (3, MIXED): 15, (2, FP64): 15}.get((D, case["prec"]), 0)
        E = torch.zeros((n + 2,) * D, dtype=torch.complex128, device=dev)
        _cycle(E, data.to(torch.complex128), 1.0 / (n + 1), case["nu1"], case["nu2"], top)
        return {"e": E[(slice(1, -1),) * D].contiguous()}
    if kind == "solve":
        return {"u": _helmholtz(*data, case["k"], case["p"]), "status": None, "iters": None, "relres": None}
    if kind == "annulus":
        if case["N"] > 512:                # over 20 s
            return None
        return {"u": _annulus(data, case["hole"], case["k"]), "status": None, "iters": None, "relres": None}
    U = [_helmholtz(f, g, k, 0.0).reshape(-1) for _, _, k, f, g in data]
    return {"u": torch.cat(U), "status": None, "iters": None}
