"""A step of a state and of the same state with averages, gradients and
viscosity times 2^k: the equations and the linear weights (limiter 1) have no
absolute scale, so the result is the step's times 2^k as long as the state is in
the format's range; with a density and pressure jump, where the admissibility
fallback is in play.  On grids where the flux takes a lane per Gauss point and
where it takes a thread per face, and in 1D in the short and the long form.

Bars: scaling by a power of two commutes with every rounding, so only a decision
taken by another formula at the scaled state moves, by a rounding: FP64 1e-12 of
the largest value (gradients 1e-11 of it over h), mixed 1e-6 and 1e-4."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2507_20461_gb300 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _state(n, jump):
    m, rng = len(n), np.random.default_rng(sum(n))
    X = np.meshgrid(*[(np.arange(k) + 0.5) / k for k in reversed(n)], indexing="ij")
    ph = rng.uniform(0, 6, size=(m + 2, m))
    rho = 1.0 + 0.2 * sum(np.sin(2 * np.pi * x + a) for x, a in zip(X, ph[0]))
    vel = [0.3 * np.cos(2 * np.pi * X[-1 - i] + ph[1 + i, 0]) for i in range(m)]
    p = 1.0 + 0.1 * sum(np.cos(2 * np.pi * x + a) for x, a in zip(X, ph[m + 1]))
    if jump:
        low = sum(X) > 0.5 * m
        rho, p = np.where(low, 0.3 * rho, rho), np.where(low, 0.3 * p, p)
    W = np.array([rho, *(rho * u for u in vel), p / 0.4 + 0.5 * rho * sum(u * u for u in vel)])
    G = np.stack([np.gradient(W, axis=W.ndim - 1 - a) for a in range(m)])
    return np.ascontiguousarray(W), np.ascontiguousarray(G)


def _step(n, W, G, precision, mu, **kw):
    s = B.Solver(n, hi=[float(k) for k in n], bc=B.BC_TRANSMISSIVE, precision=precision, limiter=1, mu=mu, **kw)
    Wd, Gd = torch.from_numpy(W).to(DEV), torch.from_numpy(G).to(DEV)
    s.set_state(Wd, Gd)
    s.step(0.1)
    s.get_state(Wd, Gd)
    assert s.status() == 0
    s.close()
    return Wd.cpu().numpy(), Gd.cpu().numpy()


CASES = [(1, k, n, {}) for k in (-90, -75, 40) for n in ((40, 24), (300, 260), (12, 9, 10), (40, 41, 42))]
CASES += [(0, k, n, {}) for k in (-400, -360, 345) for n in ((40, 24), (260, 200), (12, 9, 10), (30, 31, 32), (50,), (9001,))]
CASES += [(0, -520, n, {}) for n in ((40, 24), (260, 200), (12, 9, 10), (50,), (9001,))]
CASES += [(0, k, n, {"order": 6}) for k in (-400, 345) for n in ((50,), (9001,))]


@pytest.mark.parametrize("precision,k,n,kw", CASES)
@pytest.mark.parametrize("mu,jump", [(0.0, False), (0.0, True), (0.01, False)])
def test_step_scales_with_the_state(precision, k, n, kw, mu, jump):
    if kw and mu:
        pytest.skip("the non-compact schemes are inviscid")
    W, G = _state(n, jump)
    W1, G1 = _step(n, W, G, precision, mu, **kw)
    Wk, Gk = _step(n, np.ldexp(W, k), np.ldexp(G, k), precision, float(np.ldexp(mu, k)), **kw)
    top = np.abs(W1).max()
    tw, tg = (1e-6, 1e-4) if precision else (1e-12, 1e-11)
    assert np.abs(np.ldexp(Wk, -k) - W1).max() <= tw * top
    assert np.abs(np.ldexp(Gk, -k) - G1).max() <= tg * top
