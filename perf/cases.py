"""Performance cases of the compact GKS library: what its users run, through
its public entry points (``binding.Solver`` and ``binding.Batch``).

Kinds of case:
  step    set a state, advance it by CFL time steps, read it back
          (``set_state``, ``step_cfl``, ``get_state``): 1D, 2D and 3D, FP64
          and mixed precision, Euler and Navier-Stokes, every scheme;
  batch   the same for many independent 2D grids (``Batch.run``);
  faces   the interface states and the interface fluxes of a state
          (``reconstruct``, ``flux``).

A pass starts from the same state each time, so it can be repeated; the copies
in and out are those a program makes that reads its results every few steps.
Mixed precision computes fluxes and gradients in FP32, so a program that
chose it takes its fields as FP32.  The flows amplify rounding-level
differences (shocks, GENO's switches), tenfold in about eight steps: passes
are short, and the shocks weak enough (Mach below 1.6) that no average comes
near vacuum.

``exact`` is the same scheme in plain torch, FP64 throughout, written from its
formulas (moment conditions solved numerically, velocity integrals term by
term) without the library's code.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_2507_20461_gb300 import binding as B

GAMMA = 1.4
DEVICE = "cuda:0"

# Floating-point operations of one cell-update (one time step of one cell):
# tests/golden/flop_counts.json; 1D compact: two stages of one face flux and
# three variables' reconstruction.
STEP_FLOPS = {1: 2700.0, 2: 24773.0, 3: 146440.0}
NC_FLOPS = {5: 3262.0, 6: 5686.0}


def _case(kind, n, precision=1, *, name=None, ic="modes", bc="periodic", limiter=0, order=0, mu=0.0, steps=1, fused=False,
          grids=1):
    nx, ny, nz = tuple(n) + (1,) * (3 - len(n))
    c = dict(kind=kind, dim=len(n), nx=nx, ny=ny, nz=nz, precision=precision, ic=ic, bc=bc, limiter=limiter, order=order,
             mu=mu, steps=steps, fused=fused, grids=grids)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the paper's 1D Riemann problems (400 cells): launches and latency are everything
        _case("step", (400,), 0, name="riemann_1d_400_fp64", ic="jumps", bc="transmissive", steps=20),
        # long 1D non-compact runs (6th order, HLLC, RK4), a million cells, odd count
        _case("step", (1000003,), 0, name="noncompact6_1d_1m_fp64", bc="transmissive", order=6, steps=1),
        # a small 2D grid: coarse-grid studies, tests, parameter scans
        _case("step", (64, 64), 1, name="small_2d_64_mixed", steps=4),
        # the four-quadrant Riemann problem at its stated size, plain FP64
        _case("step", (512, 512), 0, name="quadrants_2d_512_fp64", ic="jumps", bc="transmissive", steps=2),
        # the headline workload: 2048^2 periodic, density modes and shocks, mixed precision
        _case("step", (2048, 2048), 1, name="modes_2d_2048_mixed", steps=2),
        # one fused kernel per stage, ragged grid between slip walls, WENO-Z weights
        _case("step", (1003, 777), 1, name="fused_2d_walls_wenoz_mixed", bc="reflective", limiter=2, steps=2, fused=True),
        # viscous flow in a box: no-slip on three sides, a symmetry line on top
        _case("step", (390, 195), 0, name="viscous_box_2d_fp64", ic="modes", bc="box", mu=0.002, steps=2),
        # many uneven 2D grids at once, sides log-uniform (ensemble runs), mixed precision
        _case("batch", (96, 1024), 1, name="batch_12_grids_mixed", ic="jumps", bc="transmissive", steps=2, grids=12),
        # the same in FP64, smaller
        _case("batch", (64, 256), 0, name="batch_6_grids_fp64", ic="jumps", bc="transmissive", steps=2, grids=6),
        # the 3D workload: 256^3 periodic
        _case("step", (256, 256, 256), 1, name="modes_3d_256_mixed", steps=1),
        # 3D Navier-Stokes between walls, ragged
        _case("step", (99, 64, 50), 1, name="viscous_3d_ragged_mixed", bc="noslip", mu=0.002, steps=2),
        # interface states and fluxes of a 2D FP64 state, ragged (analysis, coupling to other codes)
        _case("faces", (301, 214), 0, name="faces_2d_301x214_fp64"),
    ]


def _logu(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["1d", "nc", "2d", "2d", "2d64", "3d", "3d64", "batch", "faces"])
    lim = rng.choice([0, 0, 0, 1, 2])
    bc = rng.choice(["periodic", "transmissive", "reflective", "noslip"])
    mu = rng.choice([0.0, 0.0, 0.002])
    if kind == "1d":
        precision = rng.choice([0, 0, 1])
        return _case("step", (_logu(rng, 100, 200000 if precision == 0 else 2000),), precision, ic="jumps", bc=bc,
                     limiter=rng.choice([0, 0, 1, 2, 3]) if precision == 0 else lim, steps=rng.randint(2, 12 if precision == 0 else 3))
    if kind == "nc":
        return _case("step", (_logu(rng, 200, 2000000),), 0, bc=rng.choice(["periodic", "transmissive", "reflective"]),
                     order=rng.choice([5, 6]), limiter=rng.choice([0, 0, 1]), steps=rng.randint(1, 3))
    if kind == "2d":
        nx = _logu(rng, 48, 1600)
        return _case("step", (nx, max(40, int(nx * rng.uniform(0.4, 1.3)))), 1, bc=bc, limiter=lim, mu=mu,
                     steps=rng.randint(1, 2), fused=rng.random() < 0.4)
    if kind == "2d64":
        nx = _logu(rng, 40, 512)
        return _case("step", (nx, max(32, int(nx * rng.uniform(0.4, 1.0)))), 0, ic=rng.choice(["modes", "jumps"]), bc=bc,
                     limiter=lim, mu=mu, steps=rng.randint(1, 3))
    if kind == "3d":
        nx = _logu(rng, 32, 192)
        return _case("step", (nx, max(20, int(nx * rng.uniform(0.5, 1.0))), max(20, int(nx * rng.uniform(0.5, 1.0)))), 1, bc=bc,
                     limiter=lim, mu=mu, steps=rng.randint(1, 2))
    if kind == "3d64":
        nx = _logu(rng, 12, 56)
        return _case("step", (nx, max(8, int(nx * rng.uniform(0.5, 1.0))), max(8, int(nx * rng.uniform(0.5, 1.0)))), 0, bc=bc,
                     limiter=lim, mu=mu, steps=1)
    if kind == "batch":
        precision = rng.choice([0, 1, 1])
        lo = rng.randint(33, 100)
        return _case("batch", (lo, lo + _logu(rng, 40, 200 if precision == 0 else 900)), precision, ic="jumps",
                     bc=rng.choice(["periodic", "transmissive", "reflective"]), limiter=lim, steps=rng.randint(1, 2),
                     grids=rng.randint(3, 12))
    if rng.random() < 0.7:
        n = (_logu(rng, 33, 600), _logu(rng, 33, 300))
    else:
        n = tuple(rng.randint(16, 40) for _ in range(3))
    return _case("faces", n, 0, bc=bc, limiter=lim, mu=mu)


# ---------------------------------------------------------------- inputs

BC = {"periodic": 0, "transmissive": 1, "reflective": 2, "noslip": 3}


def _sides(case):
    if case["bc"] == "box":
        return [3, 3, 3, 2, 3, 3]
    return [BC[case["bc"]]] * 6


def _rand(seed):
    return np.random.default_rng(int(seed) & 0xFFFFFFFF)


def _cons(rho, vel, p):
    return torch.stack([rho, *(rho * u for u in vel), p / (GAMMA - 1) + 0.5 * rho * sum(u * u for u in vel)])


def _coords(n, d, device):
    """cell-centre coordinates in [0, 1] per axis, the coordinate of axis d on the faces instead"""
    out = []
    for a, k in enumerate(n):
        x = torch.arange(k + (a == d), dtype=torch.float64, device=device)
        x = (x if a == d else x + 0.5) / k
        out.append(x.reshape((-1,) + (1,) * a))
    return out


def _modes(n, seed, device, d=None):
    """Conservative variables at the cell centres (or on the faces of axis d): density and velocity modes
    around rho = 1, p = 1, with planar slabs of shocked gas (Rankine-Hugoniot, Mach 1.15-1.6)."""
    m, rng = len(n), _rand(seed)
    X = _coords(n, d, device)
    rho, vel = 1.0 + 0 * sum(X), [0.1 * (-1) ** a + 0 * sum(X) for a in range(m)]
    for i in range(8):
        k = rng.integers(-5, 6, m)
        k[i % m] = k[i % m] or 1
        arg = 2 * math.pi * sum(int(k[a]) * X[a] for a in range(m))
        rho = rho + 0.03 * torch.cos(arg + rng.uniform(0, 6.28))
        vel[i % m] = vel[i % m] + 0.04 * torch.cos(arg + rng.uniform(0, 6.28))
    p = 1.0 + 0 * rho
    r0 = rho
    for i in range(4):
        nrm = [0] * m
        nrm[i % m] = 1
        if m > 1 and i >= 2:
            nrm[(i + 1) % m] = int(rng.choice([-1, 1]))
        size = math.sqrt(sum(k * k for k in nrm))
        mach, off = rng.uniform(1.15, 1.6), rng.uniform(0, 1)
        behind = torch.remainder(sum(k * x for k, x in zip(nrm, X)) - off, 1.0) > 1.0 - 0.07 * size
        r = (GAMMA + 1) * mach**2 / ((GAMMA - 1) * mach**2 + 2)
        du = mach * torch.sqrt(GAMMA / r0) * (1 - 1 / r)
        rho = torch.where(behind, r0 * r, rho)
        p = torch.where(behind, 1 + 2 * GAMMA / (GAMMA + 1) * (mach**2 - 1) + 0 * p, p)
        vel = [torch.where(behind, du * k / size, u) for k, u in zip(nrm, vel)]
    return _cons(rho, vel, p)


def _jumps(n, seed, device):
    """A Riemann problem: 2^m constant states meeting at the middle (periodic boundaries repeat it), zero gradients."""
    m, rng = len(n), _rand(seed)
    X = _coords(n, None, device)
    q = sum((X[a] >= 0.5).long() << a for a in range(m))
    st = torch.tensor([[rng.uniform(0.5, 1.5)] + [rng.uniform(-0.4, 0.4) for _ in range(m)] + [rng.uniform(0.5, 1.5)]
                       for _ in range(2**m)], dtype=torch.float64, device=device)
    W = _cons(st[q, 0], [st[q, 1 + a] for a in range(m)], st[q, m + 1])
    return W, torch.zeros((m,) + tuple(W.shape), dtype=torch.float64, device=device)


def _state(n, ic, seed, device):
    """Averages W[v][k][j][i], gradients G[d][v][k][j][i] and the cell size of a box whose first side is 1."""
    n, h = tuple(n), 1.0 / n[0]
    if ic == "jumps":
        W, G = _jumps(n, seed, device)
    else:
        W = _modes(n, seed, device)
        G = torch.empty((len(n),) + tuple(W.shape), dtype=torch.float64, device=device)
        for d in range(len(n)):
            G[d] = _modes(n, seed, device, d).diff(dim=W.ndim - 1 - d) / h
    return W.contiguous(), G, h


def _size(case):
    return (case["nx"], case["ny"], case["nz"])[: case["dim"]]


def _batch_sizes(case, seed):
    """sides log-uniform in [nx, ny], the same for every seed but for their order (plans differ, work does not)"""
    lo, hi, k = case["nx"], case["ny"], 2 * case["grids"]
    s = [int(round(lo * (hi / lo) ** ((i + 0.5) / k))) for i in range(k)]
    _rand(7).shuffle(s)
    return list(zip(s[::2], s[1::2]))


def prepare(case, seed):
    if case["kind"] == "batch":
        sizes = _batch_sizes(case, seed)
        b = B.Batch([n[0] for n in sizes], [n[1] for n in sizes], [1.0 / n[0] for n in sizes], gamma=GAMMA, bc=BC[case["bc"]],
                    precision=case["precision"], limiter=case["limiter"])
        states = [_state(n, case["ic"], seed * 64 + g, DEVICE)[:2] for g, n in enumerate(sizes)]
        return dict(case=case, batch=b, states=states, out=[(torch.empty_like(W), torch.empty_like(G)) for W, G in states])
    n = _size(case)
    W, G, h = _state(n, case["ic"], seed, DEVICE)
    s = B.Solver(n, hi=[k * h for k in n], gamma=GAMMA, bc=_sides(case), precision=case["precision"], limiter=case["limiter"],
                 order=case["order"] or None, stage_kernels=int(case["fused"]), mu=case["mu"])
    st = dict(case=case, solver=s, W=W, G=G)
    if case["kind"] == "faces":
        nf, ng, nv, m = s.nfaces, s.ngauss, s.nv, s.dim
        st["states"] = torch.empty((2, nv, m + 1, ng, nf), dtype=torch.float64, device=DEVICE)
        st["flux"] = torch.empty((3, nv, ng, nf), dtype=torch.float64, device=DEVICE)
    else:
        st["Wo"], st["Go"] = torch.empty_like(W), torch.empty_like(G)
    return st


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b = state["batch"]
        for g, (W, G) in enumerate(state["states"]):
            b.set_state(g, W, G)
        b.run(0.4, case["steps"])
        for g, (W, G) in enumerate(state["out"]):
            b.get_state(g, W, G)
        W, G = (torch.cat([o[i].reshape(-1) for o in state["out"]]) for i in (0, 1))
    elif case["kind"] == "faces":
        s = state["solver"]
        s.set_state(state["W"], state["G"])
        s.reconstruct(state["states"])
        s.flux(0.1 / case["nx"], state["flux"])
        return {"values": state["states"][:, :, 0], "slopes": state["states"][:, :, 1:], "F": state["flux"][0],
                "dFdt": state["flux"][1], "W": state["flux"][2]}
    else:
        s = state["solver"]
        s.set_state(state["W"], state["G"])
        s.step_cfl(0.4, case["steps"])
        W, G = state["Wo"], state["Go"]
        s.get_state(W, G)
    return {"W": W.float(), "G": G.float()} if case["precision"] else {"W": W, "G": G}


def work(case):
    m = case["dim"]
    sizes = _batch_sizes(case, 0) if case["kind"] == "batch" else [_size(case)]
    cells = sum(math.prod(n) for n in sizes)
    if case["kind"] == "batch":
        m = 2
    state = 8.0 * (m + 2) * (m + 1) * cells
    if case["kind"] == "faces":
        nf, ng = sum(math.prod(n) // k * (k + 1) for n in sizes for k in n), 2 ** (m - 1)
        # one stage's reconstruction and fluxes: half a step
        return {"bytes": state + 8.0 * nf * ng * (m + 2) * (2 * (m + 1) + 3), "flops": 0.5 * STEP_FLOPS[m] * cells}
    per = NC_FLOPS[case["order"]] if case["order"] in NC_FLOPS else STEP_FLOPS[m]
    return {"bytes": 2 * state, "flops": per * cells * case["steps"]}


# ---------------------------------------------------------------- the scheme in plain FP64 torch


def _pad(A, axis, k, bc_lo, bc_hi, a, m, lead):
    """k ghost layers along tensor axis `axis` (space axis a); A is averages (lead = 1) or gradients (lead = 2)."""
    n = A.shape[axis]
    if bc_lo == 0:
        return torch.cat([A.narrow(axis, n - k, k), A, A.narrow(axis, 0, k)], axis)

    def ghost(part, t):
        s = torch.ones(m + 2, dtype=A.dtype, device=A.device)
        if t >= 2:
            s[1 + a] = -1
        if t == 3:
            s[1 : m + 1] = -1
        g = part.flip(axis) * s.reshape((-1,) + (1,) * (A.ndim - lead))
        if lead == 2:
            g[a] *= -1
        return g

    return torch.cat([ghost(A.narrow(axis, 0, k), bc_lo), A, ghost(A.narrow(axis, n - k, k), bc_hi)], axis)


def _padded(W, G, bcs, k, m):
    for a in range(m):
        W = _pad(W, W.ndim - 1 - a, k, bcs[2 * a], bcs[2 * a + 1], a, m, 1)
        G = _pad(G, G.ndim - 1 - a, k, bcs[2 * a], bcs[2 * a + 1], a, m, 2)
    return W, G


def _mean1(p, c):
    """average of x^p over the unit cell centred at c"""
    return ((c + 0.5) ** (p + 1) - (c - 0.5) ** (p + 1)) / (p + 1)


def _mean(e, c):
    return math.prod(_mean1(p, x) for p, x in zip(e, c))


def _diff(e, a):
    """(factor, exponents) of the derivative of a monomial along axis a"""
    return (e[a], tuple(p - (i == a) for i, p in enumerate(e))) if e[a] else (0, e)


def _cubic(m):
    """Least-squares cubic: its monomials, the map from the cross data (neighbour difference and cell-unit
    gradient per neighbour, then the own gradient), and the indicators' quadratic forms."""
    mono = [e for e in itertools.product(range(4), repeat=m) if 1 <= sum(e) <= 3 and e != (1, 1, 1)]
    zero, rows = (0,) * m, []
    for q in range(2 * m):
        c = tuple((1 if q & 1 else -1) * (i == q // 2) for i in range(m))
        rows.append([_mean(e, c) - _mean(e, zero) for e in mono])
        rows += [[f * _mean(x, c) for f, x in (_diff(e, a) for e in mono)] for a in range(m)]
    rows += [[f * _mean(x, zero) for f, x in (_diff(e, a) for e in mono)] for a in range(m)]
    QH, Qt = np.zeros((len(mono),) * 2), np.zeros((len(mono),) * 2)
    for l in itertools.product(range(4), repeat=m):
        if not 1 <= sum(l) <= 3:
            continue
        der = []
        for e in mono:
            f, x = 1.0, e
            for a in range(m):
                for _ in range(l[a]):
                    g, x = _diff(x, a)
                    f *= g
            der.append((f, x))
        T = np.array([[f * g * _mean(tuple(i + j for i, j in zip(x, y)), zero) if f and g else 0.0 for g, y in der] for f, x in der])
        QH += T
        Qt += T if sum(l) == 3 else 0
    return mono, np.linalg.pinv(np.array(rows)), QH, Qt


def _chi(ISt, ISH, ISL, r, C=20.0, eps=1e-15):
    aH, aL = 1 + (ISt / (ISH + eps)) ** r, 1 + (ISt / (ISL + eps)) ** r
    return torch.tanh(C * 2 * aH / (aH + aL)) / math.tanh(C)


def _weights(lim, d, IS, tau, eps=1e-15, d0=0.85, ct=1e-6):
    """(chi, per-sub-stencil weights) of the WENO-Z / TENO combination; candidate 0 the high-order polynomial"""
    if lim == 2:
        w = [k * (1 + tau / (i + eps)) for k, i in zip(d, IS)]
    else:
        low = torch.stack(IS).amin(0)
        g = [((low + eps) / (i + eps)) ** 7 for i in IS]
        tot = sum(g)
        w = [torch.where(x <= ct * tot, 0.0 * x, k + 0.0 * x) for k, x in zip(d, g)]
    tot = sum(w)
    chi = w[0] / tot / d0
    return chi, [x / tot - chi * k for x, k in zip(w[1:], d[1:])]


def _blend(d, m, lim, cub):
    """Blended cubic [NC, cells...] of one variable from its cross data d [ND, cells...]"""
    mono, fit, QH, Qt = cub
    t = lambda x: torch.as_tensor(x, dtype=d.dtype, device=d.device)  # noqa: E731
    shape, d = d.shape[1:], d.reshape(d.shape[0], -1)
    c = t(fit) @ d
    if lim == 1:
        return c.reshape((-1,) + shape)
    ISH, ISt = (c * (t(QH) @ c)).sum(0), (c * (t(Qt) @ c)).sum(0)
    g = []
    for q in range(2 * m):
        s, o = (1.0 if q & 1 else -1.0), q * (1 + m)
        g.append(torch.stack([0.5 * (s * d[o] + d[o + 1 + a]) if a == q // 2 else d[o + 1 + a] for a in range(m)]))
    IS = [(x * x).sum(0) for x in g]
    if lim == 0:
        al = torch.stack(IS)
        chi = _chi(ISt, ISH, (al.sum(0) - al.amin(0) - al.amax(0)) / (2 * m - 2), 3)
        w = [1 / (i + 1e-15) ** 2 for i in IS]
        tot = sum(w)
        w = [(1 - chi) * x / tot for x in w]
    else:
        chi, w = _weights(lim, [0.85] + [0.15 / (2 * m)] * (2 * m), [ISH] + IS, ISt)
    c = chi * c
    for a in range(m):
        c[mono.index(tuple(int(i == a) for i in range(m)))] += sum(x * y[a] for x, y in zip(w, g))
    return c.reshape((-1,) + shape)


def _blended(W, G, h, bcs, lim, m, cub):
    """Blended cubics [NC, nv, cells + ghost ring] and the averages there"""
    Wp, Gp = _padded(W, G * h, bcs, 2, m)

    def at(A, o):
        for a in range(m):
            ax = A.ndim - 1 - a
            A = A.narrow(ax, 1 + o[a], A.shape[ax] - 2)
        return A

    zero, out = (0,) * m, []
    for v in range(m + 2):
        d = []
        for q in range(2 * m):
            o = tuple((1 if q & 1 else -1) * (i == q // 2) for i in range(m))
            d.append(at(Wp[v], o) - at(Wp[v], zero))
            d += [at(Gp[a, v], o) for a in range(m)]
        d += [at(Gp[a, v], zero) for a in range(m)]
        out.append(_blend(torch.stack(d), m, lim, cub))
    return torch.stack(out, 1), at(Wp, zero)


def _admit(val, der, cell, m):
    p = lambda w: w[m + 1] - 0.5 * sum(w[1 + a] ** 2 for a in range(m)) / w[0]  # noqa: E731
    ok = (val[0] > 0.3 * cell[0]) & (p(val) > 0.3 * p(cell))
    return torch.where(ok, val, cell), torch.where(ok, der, 0.0 * der)


def _quad(mono):
    """<u^i v^j w^k xi^(2l)> of a Maxwellian given its moment lists"""
    return lambda e, M: math.prod([M[a][p] for a, p in enumerate(e) if p], start=torch.ones((), dtype=torch.float64, device=M[0][1].device))


def _max_moments(U, th, K, m, half=0):
    def rec(m0, m1, u, top):
        out = [m0, m1]
        for k in range(top - 1):
            out.append(u * out[-1] + (k + 1) * th * out[-2])
        return out

    one = torch.ones_like(th)
    if half:
        lam = 0.5 / th
        m0 = 0.5 * torch.erfc(-half * torch.sqrt(lam) * U[0])
        m1 = U[0] * m0 + half * 0.5 * torch.exp(-lam * U[0] ** 2) / torch.sqrt(math.pi * lam)
        mu = rec(m0, m1, U[0], 6)
    else:
        mu = rec(one, U[0], U[0], 6)
    return [mu] + [rec(one, U[a], U[a], 5) for a in range(1, m)] + [[one, K * th, K * (K + 2) * th**2]]


def _unit(m, a, p=1):
    return tuple(p * (i == a) for i in range(m + 1))


def _plus(x, y):
    return tuple(i + j for i, j in zip(x, y))


def _psi(m):
    zero = (0,) * (m + 1)
    return [{zero: 1.0}] + [{_unit(m, a): 1.0} for a in range(m)] + [{**{_unit(m, a, 2): 0.5 for a in range(m)}, _unit(m, m): 0.5}]


def _psi_mean(poly, M, m, k):
    """[<psi_b u^k poly>]_b"""
    memo = {}

    def mom(e):
        if e not in memo:
            r = M[0][e[0]]
            for a in range(1, m + 1):
                if e[a]:
                    r = r * M[a][e[a]]
            memo[e] = r
        return memo[e]

    out = []
    for psi in _psi(m):
        r = 0.0
        for e, c in poly.items():
            x = sum(f * mom(_plus(_plus(e, g), _unit(m, 0, k))) for g, f in psi.items())
            r = r + c * x
        out.append(r)
    return torch.stack(out)


def _prim(W, m):
    U = [W[1 + a] / W[0] for a in range(m)]
    p = (GAMMA - 1) * (W[m + 1] - 0.5 * sum(W[1 + a] * U[a] for a in range(m)))
    return W[0], U, p, p / W[0]


def _micro(U, th, r, N, m):
    """Coefficients of a on psi with <a psi> = r"""
    s = [r[1 + a] - U[a] * r[0] for a in range(m)]
    sE = r[m + 1] - 0.5 * sum(u * u for u in U) * r[0] - sum(u * x for u, x in zip(U, s))
    aE = (2 * sE - N * th * r[0]) / (N * th * th)
    al = [x / th for x in s]
    a0 = r[0] - 0.5 * aE * N * th - sum(x * u for x, u in zip(al, U)) + 0.5 * aE * sum(u * u for u in U)
    return [a0] + [x - aE * u for x, u in zip(al, U)] + [aE]


def _slope_poly(s, m):
    """sum_e u_e (s_e . psi)"""
    poly = {}
    for e, c in enumerate(s):
        for b, psi in enumerate(_psi(m)):
            for g, f in psi.items():
                k = _plus(g, _unit(m, e))
                poly[k] = poly.get(k, 0.0) + f * c[b]
    return poly


def _gks(Wl, Wr, dl, dr, dt, mu, m):
    """F, dF/dt, W(dt/2) in the face frame; dl, dr [m, nv, faces]"""
    N = 2 / (GAMMA - 1)
    K = N - m
    one = {(0,) * (m + 1): 1.0}

    def dot_psi(c):
        poly = {}
        for b, psi in enumerate(_psi(m)):
            for g, f in psi.items():
                poly[g] = poly.get(g, 0.0) + f * c[b]
        return poly

    def slopes(rho, U, th, d):
        return [_micro(U, th, d[e] / rho, N, m) for e in range(m)]

    W0 = Fk = WT = FT = WA = FA = 0.0
    press = []
    for W, d, half in ((Wl, dl, 1), (Wr, dr, -1)):
        rho, U, p, th = _prim(W, m)
        press.append(p)
        M, full = _max_moments(U, th, K, m, half), _max_moments(U, th, K, m)
        T = _slope_poly(slopes(rho, U, th, d), m)
        W0 = W0 + rho * _psi_mean(one, M, m, 0)
        Fk = Fk + rho * _psi_mean(one, M, m, 1)
        WT = WT + rho * _psi_mean(T, M, m, 0)
        FT = FT + rho * _psi_mean(T, M, m, 1)
        if mu:
            A = dot_psi(_micro(U, th, -_psi_mean(T, full, m, 0), N, m))
            WA = WA + rho * _psi_mean(A, M, m, 0)
            FA = FA + rho * _psi_mean(A, M, m, 1)
    rho, U, p0, th = _prim(W0, m)
    M = _max_moments(U, th, K, m)
    T = _slope_poly(slopes(rho, U, th, 0.5 * (dl + dr)), m)
    Tm = _psi_mean(T, M, m, 0)
    A = dot_psi(_micro(U, th, -Tm, N, m))
    F0, FT0, FA0 = (rho * _psi_mean(x, M, m, 1) for x in (one, T, A))
    W0t = -rho * Tm
    pl, pr = press
    tau = mu / p0 if mu else 0.0
    tn = 0.05 * dt + (pl - pr).abs() / (pl + pr) * dt + tau

    def flux(x):
        e = torch.exp(-x / tn)
        ie, ite = tn * (1 - e), tn * tn - tn * (x + tn) * e
        return ((x - ie) * F0 + (ite + tau * (ie - x)) * FT0 + (0.5 * x * x + tau * (ie - x)) * FA0 + ie * Fk - (ite + tau * ie) * FT
                - tau * ie * FA)

    h = 0.5 * dt
    Fh, F1, e = flux(h), flux(dt), torch.exp(-h / tn)
    Wh = W0 + (h * (1 - e)) * W0t - (h + tau) * e * WT - tau * e * WA
    return (4 * Fh - F1) / dt, 4 * (F1 - 2 * Fh) / dt**2, Wh


def _gauss(m):
    r = 1 / (2 * math.sqrt(3))
    return [(s,) for s in (-r, r)] if m == 2 else [(s, t) for t in (-r, r) for s in (-r, r)]


def _faces(W, G, h, dt, case, cub, want):
    """Multi-D faces, per direction: want = "flux": (F, dF/dt, W(dt/2)) [3, nv, ng, faces...]; "states":
    [2, nv, m + 1, ng, faces...]"""
    m, bcs = case["dim"], _sides(case)
    mono = cub[0]
    b, w = _blended(W, G, h, bcs, case["limiter"], m, cub)
    out = []
    for d in range(m):
        tang = [a for a in range(m) if a != d]
        perm = [0, 1 + d] + [1 + a for a in tang] + [m + 1]
        per_g = []
        for g in _gauss(m):
            st = []
            for side in (0, 1):
                x = [0.0] * m
                x[d] = 0.5 - side
                for a, s in zip(tang, g):
                    x[a] = s
                ev = [[math.prod(q**p for q, p in zip(x, e)) - _mean(e, (0,) * m) for e in mono]]
                for a in range(m):
                    ev.append([f * math.prod(q**p for q, p in zip(x, y)) if f else 0.0 for f, y in (_diff(e, a) for e in mono)])

                def cut(A):
                    for a in range(m):
                        ax = A.ndim - 1 - a
                        k = A.shape[ax]
                        A = A.narrow(ax, side, k - 1) if a == d else A.narrow(ax, 1, k - 2)
                    return A

                bb, cell = cut(b), cut(w)
                v = (torch.tensor(ev, dtype=W.dtype, device=W.device) @ bb.reshape(len(mono), -1)).reshape((1 + m,) + tuple(bb.shape[1:]))
                st.append(_admit(cell + v[0], v[1:] / h, cell, m))
                del bb, v
            (vl, dl), (vr, dr) = st
            if want == "states":
                per_g.append(torch.stack([torch.cat([v[None], s]).transpose(0, 1) for v, s in st]))
                continue
            axes = [d] + tang
            q = torch.stack(_gks(vl[perm], vr[perm], dl[axes][:, perm], dr[axes][:, perm], dt, case["mu"], m))
            q = q[:, [perm.index(v) for v in range(m + 2)]]
            ax = q.ndim - 1 - d
            for t, i in ((bcs[2 * d], 0), (bcs[2 * d + 1], q.shape[ax] - 1)):
                if t >= 2:
                    q.select(ax, i)[:2, [0, m + 1]] = 0.0
            per_g.append(q)
        out.append(torch.stack(per_g, 3 if want == "states" else 2))
    return out


def _polys_from(conditions, deg):
    """Polynomial coefficients (x^1..x^deg, zero-average basis about cell 0) as a map of the data: conditions
    are ("avg" | "der", cell)."""
    rows = [[_mean1(p, c) - _mean1(p, 0) if k == "avg" else p * _mean1(p - 1, c) for p in range(1, deg + 1)] for k, c in conditions]
    return np.linalg.solve(np.array(rows), np.eye(deg))


def _eval1(c, x, n):
    val = sum(c[p - 1] * (x**p - _mean1(p, 0)) for p in range(1, n + 1))
    return val, sum(p * c[p - 1] * x ** (p - 1) for p in range(1, n + 1))


def _lin(Mx, data):
    return [sum(float(k) * x for k, x in zip(row, data)) for row in Mx]


def _js(c):
    """sum_l int (d^l p)^2 over the cell of sum_p c_p x^p (p = 1..)"""
    n, r = len(c), 0.0
    for l in range(1, n + 1):
        k = [(math.perm(p, l), p - l) for p in range(1, n + 1)]
        r = r + sum(f * g * _mean1(i + j, 0) * c[a] * c[b] for a, (f, i) in enumerate(k) for b, (g, j) in enumerate(k) if i >= 0 and j >= 0)
    return r


def _side_1d(w, d, lim):
    """Value and slope (cell units, relative to cell 1) at the right face of cell 1 of w[0..3] = cells -1, 0, 1, 2"""
    u = [x - w[1] for x in w]
    c7 = _lin(_polys_from([("avg", -1), ("avg", 1), ("avg", 2)] + [("der", k) for k in (-1, 0, 1, 2)], 7), [u[0], u[2], u[3]] + d)
    qv, qd = _eval1(c7, 0.5, 7)
    if lim == 1:
        return qv, qd
    subs = [_lin(_polys_from(k, 2), x) for k, x in (([("avg", -1), ("der", -1)], [u[0], d[0]]), ([("avg", -1), ("avg", 1)], [u[0], u[2]]),
                                                    ([("avg", 1), ("avg", 2)], [u[2], u[3]]))]
    IS, pv = [_js(c) for c in subs], [_eval1(c, 0.5, 2) for c in subs]
    al = torch.stack(IS)
    ISt = (0.5 * (IS[1] + IS[2]) - IS[0]).abs()
    if lim == 0:
        chi = _chi(ISt, al.amax(0), al.amin(0), 2)
        k = [c / (i + 1e-15) ** 2 for c, i in zip((1.0, 8.0, 1.0), IS)]
        tot = sum(k)
        k = [(1 - chi) * x / tot for x in k]
    else:
        chi, k = _weights(lim, [0.85, 0.015, 0.12, 0.015], [al.amax(0)] + IS, ISt)
    return tuple(chi * q + sum(x * y[i] for x, y in zip(k, pv)) for i, q in enumerate((qv, qd)))


def _faces_1d(W, G, h, dt, case, want):
    bcs, n = _sides(case), W.shape[1]
    Wp, Gp = _padded(W, G * h, bcs, 2, 1)
    w, d = [Wp[:, i : i + n + 1] for i in range(4)], [Gp[0, :, i : i + n + 1] for i in range(4)]
    lv, ls = _side_1d(w, d, case["limiter"])
    rv, rs = _side_1d(w[::-1], [-x for x in d[::-1]], case["limiter"])
    st = [_admit(w[1] + lv, ls[None] / h, w[1], 1), _admit(w[2] + rv, -rs[None] / h, w[2], 1)]
    if want == "states":
        return [torch.stack([torch.stack([v, s[0]], 1) for v, s in st])[:, :, :, None]]
    q = torch.stack(_gks(st[0][0], st[1][0], st[0][1], st[1][1], dt, case["mu"], 1))
    for t, i in ((bcs[0], 0), (bcs[1], n)):
        if t >= 2:
            q[:2, [0, 2], i] = 0.0
    return [q[:, :, None]]


def _update(W, G, h, dt, case, cub):
    """L(F), L(dF/dt) and the averaged gradients of W(dt/2) of one stage"""
    m = case["dim"]
    f = _faces_1d(W, G, h, dt, case, "flux") if m == 1 else _faces(W, G, h, dt, case, cub, "flux")
    D = [q.mean(2).diff(dim=q.ndim - 2 - d) / h for d, q in enumerate(f)]
    return -sum(x[0] for x in D), -sum(x[1] for x in D), torch.stack([x[2] for x in D])


def _dt(W, h, case, cfl=0.4):
    m = case["dim"]
    rho, U, p, _ = _prim(W, m)
    dt = cfl * h / float((torch.stack(U).abs().amax(0) + torch.sqrt(GAMMA * p / rho)).max())
    if case["mu"]:
        dt = min(dt, cfl * h * h / (2 * max(1, m - 1) * case["mu"] / float(rho.min())))
    return dt


def _nc_left(u, order, lim):
    """Left value relative to the cell, u the averages at offsets -2.. relative to it"""
    sets = [[-2, -1], [-1, 1], [1, 2]] if order == 5 else [[-2, -1], [-1, 1], [-1, 1, 2], [1, 2, 3]]
    high = [-2, -1, 1, 2] if order == 5 else [-2, -1, 1, 2, 3]
    poly = lambda s: _lin(_polys_from([("avg", k) for k in s], len(s)), [u[k + 2] for k in s])  # noqa: E731
    qH = _eval1(poly(high), 0.5, len(high))[0]
    if lim == 1:
        return qH
    c = [poly(s) for s in sets]
    IS, p = torch.stack([_js(x) for x in c]), [_eval1(x, 0.5, len(x))[0] for x in c]
    chi = _chi((0.5 * (IS[0] + IS[-1]) - IS[1]).abs(), IS.amax(0), IS.amin(0), 2)
    k = [(8.0 if i == 1 else 1.0) / (x + 1e-15) ** 2 for i, x in enumerate(IS)]
    return chi * qH + (1 - chi) * sum(a * b for a, b in zip(k, p)) / sum(k)


def _hllc(L, R):
    pr = lambda w: (w[0], w[1] / w[0], (GAMMA - 1) * (w[2] - 0.5 * w[1] ** 2 / w[0]))  # noqa: E731
    fl = lambda w, r, u, p: torch.stack([w[1], w[1] * u + p, u * (w[2] + p)])  # noqa: E731
    (rl, ul, pl), (rr, ur, pq) = pr(L), pr(R)
    cl, cr = torch.sqrt(GAMMA * pl / rl), torch.sqrt(GAMMA * pq / rr)
    SL, SR = torch.minimum(ul - cl, ur - cr), torch.maximum(ul + cl, ur + cr)
    Ss = (pq - pl + rl * ul * (SL - ul) - rr * ur * (SR - ur)) / (rl * (SL - ul) - rr * (SR - ur))

    def star(w, r, u, p, S):
        k = r * (S - u) / (S - Ss)
        us = torch.stack([k, k * Ss, k * (w[2] / r + (Ss - u) * (Ss + p / (r * (S - u))))])
        return fl(w, r, u, p) + S * (us - w)

    lo, hi = star(L, rl, ul, pl, SL), star(R, rr, ur, pq, SR)
    return torch.where(SL >= 0, fl(L, rl, ul, pl), torch.where(Ss >= 0, lo, torch.where(SR >= 0, hi, fl(R, rr, ur, pq))))


def _nc_L(W, h, case):
    n, bcs, order = W.shape[1], _sides(case), case["order"]
    Wp = _pad(W, 1, 3, bcs[0], bcs[1], 0, 1, 1)
    st = []
    for side in (0, 1):
        w = [Wp[:, (5 - i if side else i) :][:, : n + 1] for i in range(6)]
        v = w[2] + _nc_left([x - w[2] for x in w], order, case["limiter"])
        st.append(_admit(v, v[None], w[2], 1)[0])
    F = _hllc(*st)
    for t, i in ((bcs[0], 0), (bcs[1], n)):
        if t >= 2:
            F[[0, 2], i] = 0.0
    return -F.diff(dim=1) / h


def _advance(W, G, h, case):
    m = case["dim"]
    cub = _cubic(m) if m > 1 else None
    for _ in range(case["steps"]):
        dt = _dt(W, h, case)
        if case["order"] in NC_FLOPS:
            k1 = _nc_L(W, h, case)
            k2 = _nc_L(W + 0.5 * dt * k1, h, case)
            k3 = _nc_L(W + 0.5 * dt * k2, h, case)
            k4 = _nc_L(W + dt * k3, h, case)
            W = W + dt / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
            continue
        LF, LT, Gs = _update(W, G, h, dt, case, cub)
        _, LTs, Gn = _update(W + 0.5 * dt * LF + dt * dt / 8 * LT, Gs, h, dt, case, cub)
        W, G = W + dt * LF + dt * dt / 6 * (LT + 2 * LTs), Gn
    return W, G


def exact(case, seed, device=None):
    device = device or DEVICE
    if case["kind"] == "batch":
        got = []
        for g, n in enumerate(_batch_sizes(case, seed)):
            W, G, h = _state(n, case["ic"], seed * 64 + g, device)
            got.append(_advance(W, G, h, dict(case, nx=n[0], ny=n[1])))
        return {k: torch.cat([x[i].reshape(-1) for x in got]) for i, k in enumerate("WG")}
    W, G, h = _state(_size(case), case["ic"], seed, device)
    if case["kind"] == "faces":
        m, out = case["dim"], {}
        cub = _cubic(m)
        flat = lambda f, lead: torch.cat([q.reshape(tuple(q.shape[:lead]) + (-1,)) for q in f], -1)  # noqa: E731
        S = flat(_faces(W, G, h, None, case, cub, "states"), 4)
        q = flat(_faces(W, G, h, torch.tensor(0.1 / case["nx"], dtype=W.dtype, device=device), case, cub, "flux"), 3)
        out["values"], out["slopes"] = S[:, :, 0], S[:, :, 1:]
        out["F"], out["dFdt"], out["W"] = q
        return out
    W, G = _advance(W, G, h, case)
    return {"W": W, "G": G}
