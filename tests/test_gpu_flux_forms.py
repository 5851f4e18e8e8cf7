"""gks_flux in each of its forms (a lane per Gauss point on small grids, a thread
per face past the line; Euler and Navier-Stokes), FP64 against the oracle and mixed
precision against FP64, and the mixed-precision 2D step with either value of
stage_kernels against the FP64 step, on cuda:0.

Bars: FP64 flux as on small grids (test_gpu_parity.py: 1e-12, dF/dt 1e-10 of F / dt as
well); mixed 2e-5 and 2e-4, the flux at one point (test_gks_point_host.py); a mixed
step mean |rho - rho_fp64| <= 1e-5, the mixed-precision bar.  Smooth states, where
rounding is not amplified.  No mass or energy crosses a wall, exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_2507_20461_gb300 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _state(n, seed):
    m, rng = len(n), np.random.default_rng(seed)
    h = 1.0 / max(n)
    X = np.meshgrid(*[(np.arange(k) + 0.5) / k for k in reversed(n)], indexing="ij")
    rho = 1.0 + 0.2 * sum(np.sin(2 * np.pi * x + rng.uniform(0, 6)) for x in X)
    vel = [0.3 * np.cos(2 * np.pi * X[-1 - a] + rng.uniform(0, 6)) for a in range(m)]
    p = 1.0 + 0.1 * sum(np.cos(2 * np.pi * x + rng.uniform(0, 6)) for x in X)
    W = np.array([rho, *(rho * v for v in vel), p / 0.4 + 0.5 * rho * sum(v * v for v in vel)])
    G = np.zeros((m,) + W.shape)
    for a in range(m):
        if n[a] > 2:
            G[a] = np.gradient(W, h, axis=1 + (m - 1 - a))
    return W, G, h


def _solver(n, h, sides, precision, **kw):
    return B.Solver(n, hi=[k * h for k in n], bc=list(sides) + [0] * (6 - len(sides)), precision=precision, **kw)


def _faces(n):
    return [int(np.prod([k + (a == d) for a, k in enumerate(n)])) for d in range(len(n))]


def _flux(n, sides, mu, precision, W, G, h, dt):
    """through gks_flux, in the form that the number of 64-thread blocks of faces selects"""
    s = _solver(n, h, sides, precision, mu=mu)
    s.set_state(torch.from_numpy(W).to(DEV), torch.from_numpy(G).to(DEV))
    m = len(n)
    out = torch.full((3 * (m + 2) * (2 * m - 2) * sum(_faces(n)),), np.nan, dtype=torch.float64, device=DEV)
    s.flux(dt, out)
    s.close()
    return out.cpu().numpy().reshape(3, m + 2, 2 * m - 2, -1)


def _check(n, sides, got, ref, dt, tF, tT, tW):
    F = np.abs(ref[0]).max()
    assert np.abs(got[0] - ref[0]).max() <= tF * F
    assert np.abs(got[1] - ref[1]).max() <= tT * (np.abs(ref[1]).max() + F / dt)
    assert np.abs(got[2] - ref[2]).max() <= tW * np.abs(ref[2]).max()
    off, m = 0, len(n)
    for d, nf in enumerate(_faces(n)):
        ext = tuple(k + (a == d) for a, k in enumerate(n))
        f = got[:2, [0, m + 1], :, off : off + nf].reshape((2, 2, -1) + tuple(reversed(ext)))
        for side, at in ((0, 0), (1, -1)):
            if sides[2 * d + side] >= 2:
                assert np.all(np.take(f, at, axis=f.ndim - 1 - d) == 0.0)
        off += nf


def _past_the_line(n, blocks_per_sm):
    return sum(_faces(n)) / 64 > blocks_per_sm * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("mu", [0.0, 0.002])
@pytest.mark.parametrize("n,sides,past", [((37, 29), (2, 3, 1, 2), False), ((11, 9, 7), (3, 2, 0, 0, 1, 3), False),
                                          ((151, 110), (1, 1, 3, 2), True), ((25, 24, 23), (2, 1, 3, 3, 0, 0), True)])
def test_fp64_flux_matches_oracle(n, sides, past, mu):
    assert _past_the_line(n, 3) == past
    W, G, h = _state(n, sum(n))
    cfg = O.make_cfg(len(n), n, h, bc=tuple(sides) + (0,) * (6 - len(sides)), mu=mu)
    dt = 0.2 * h / O.max_wavespeed(cfg, W)
    _check(n, sides, _flux(n, sides, mu, 0, W, G, h, dt), O.flux(cfg, dt, W, G), dt, 1e-12, 1e-10, 1e-12)


@pytest.mark.parametrize("mu", [0.0, 0.002])
@pytest.mark.parametrize("n,sides,past", [((37, 29), (2, 3, 1, 2), False), ((11, 9, 7), (3, 2, 0, 0, 1, 3), False),
                                          ((281, 262), (1, 1, 3, 2), True), ((38, 37, 36), (2, 1, 3, 3, 0, 0), True)])
def test_mixed_flux_matches_fp64_flux(n, sides, past, mu):
    assert _past_the_line(n, 12) == past
    W, G, h = _state(n, sum(n))
    dt = 0.1 * h
    _check(n, sides, _flux(n, sides, mu, 1, W, G, h, dt), _flux(n, sides, mu, 0, W, G, h, dt), dt, 2e-5, 2e-4, 2e-5)


def _run(n, W, G, h, sides, precision, steps, **kw):
    s = _solver(n, h, sides, precision, **kw)
    Wd, Gd = torch.from_numpy(W).to(DEV), torch.from_numpy(G).to(DEV)
    s.set_state(Wd, Gd)
    for _ in range(steps):
        s.step(0.1 * h)
    s.get_state(Wd, Gd)
    assert s.status() == 0
    s.close()
    return Wd.cpu().numpy()


@pytest.mark.parametrize("n", [(32, 8), (37, 29), (64, 64), (100, 17), (5, 3), (1, 9), (33, 1), (130, 70)])
@pytest.mark.parametrize("sides,limiter,mu", [((0, 0, 0, 0), 0, 0.0), ((1, 1, 1, 1), 0, 0.0), ((2, 2, 2, 2), 2, 0.0),
                                              ((3, 3, 3, 3), 1, 0.0), ((3, 2, 0, 0), 0, 0.0), ((1, 1, 3, 2), 0, 2e-4)])
@pytest.mark.parametrize("stage_kernels", [0, 1])
def test_mixed_step_matches_fp64_step(n, sides, limiter, mu, stage_kernels):
    W, G, h = _state(n, 3 * sum(n))
    a = _run(n, W, G, h, sides, 1, 4, limiter=limiter, mu=mu, stage_kernels=stage_kernels)
    b = _run(n, W, G, h, sides, 0, 4, limiter=limiter, mu=mu)
    assert np.abs(b[0] - W[0]).mean() > 1e-3  # the steps moved the state
    assert np.abs(a[0] - b[0]).mean() <= 1e-5
