"""The 1D stage kernels at the sizes where they change form: the FP64 short
form (eight lanes per face, blocks of 15 cells) and the long form (a warp's 31
cells) against the oracle's step, at one cell, at the edges of a block and a
group, and around the line between the forms (three blocks per SM), where
the two forms run on either side of it.

Bar: the FP64 step's (relative L1 1e-12 per variable and step); the sizes past the
line use a smooth state, where rounding is not amplified."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
from paper_2507_20461_gb300 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _state(n, seed):
    rng = np.random.default_rng(seed)
    x = (np.arange(n) + 0.5) / n
    rho = 1.0 + 0.2 * np.sin(2 * np.pi * x + rng.uniform(0, 6))
    u = 0.3 * np.cos(2 * np.pi * x + rng.uniform(0, 6))
    p = 1.0 + 0.1 * np.sin(4 * np.pi * x)
    W = np.array([rho, rho * u, p / 0.4 + 0.5 * rho * u * u])
    G = np.zeros((1, 3, n)) if n < 3 else np.gradient(W, 1.0 / n, axis=1)[None]
    return np.ascontiguousarray(W), np.ascontiguousarray(G)


def _line():
    """the largest n of the short form on this GPU"""
    return 15 * 3 * torch.cuda.get_device_properties(0).multi_processor_count


SIZES = [1, 2, 14, 15, 16, 31, 32, 63, 400, "line", "line+1", 9001]


@pytest.mark.parametrize("order,bc,mu,limiter", [(8, 1, 0.0, 0), (8, 0, 0.0, 3), (8, 3, 0.01, 2), (5, 2, 0.0, 0), (6, 0, 0.0, 0), (6, 1, 0.0, 1)])
@pytest.mark.parametrize("size", SIZES)
def test_steps_match_oracle(order, bc, mu, limiter, size):
    n = _line() + (1 if size == "line+1" else 0) if isinstance(size, str) else size
    if mu * n > 4.0:
        pytest.skip("mean free path above the cell size: the viscous scheme is unstable there (gradients grow 1e5-fold in 3 steps)")
    W, G = _state(n, 11 * order + bc)
    h = 1.0 / n
    cfg = O.make_cfg(1, (n,), h, bc=bc, limiter=limiter, mu=mu)
    s = B.Solver((n,), bc=bc, precision=0, order=order, limiter=limiter, mu=mu)
    Wd, Gd = torch.from_numpy(W.copy()).to(DEV), torch.from_numpy(G.copy()).to(DEV)
    s.set_state(Wd, Gd)
    steps = 3
    s.step_cfl(0.3, steps)
    s.get_state(Wd, Gd)
    s.close()
    for _ in range(steps):
        if order == 8:
            assert O.step(cfg, O.cfl_dt(cfg, W, 0.3), W, G) == 0
        else:
            assert O.nc_step(cfg, order, 0.3 * h / O.max_wavespeed(cfg, W), W) == 0
    got = Wd.cpu().numpy()
    for v in range(3):
        assert np.abs(got[v] - W[v]).sum() <= 1e-12 * steps * max(np.abs(W[v]).sum(), np.abs(W[0]).sum())
    if order == 8:
        gt = Gd.cpu().numpy()
        assert np.abs(gt - G).max() <= 1e-11 * steps * np.abs(W).max() / h


@pytest.mark.parametrize("order", [8, 6])
def test_forms_agree_across_given_and_cfl_steps(order):
    """a given time step and the CFL clock take the same step"""
    n = 401
    W, G = _state(n, 5)
    out = []
    for cfl in (True, False):
        s = B.Solver((n,), bc=1, precision=0, order=order)
        Wd, Gd = torch.from_numpy(W.copy()).to(DEV), torch.from_numpy(G.copy()).to(DEV)
        s.set_state(Wd, Gd)
        if cfl:
            s.step_cfl(0.3, 2)
        else:
            for _ in range(2):
                s.step(0.3 / n / s.max_wavespeed())
        s.get_state(Wd, Gd)
        s.close()
        out.append(Wd.cpu().numpy())
    np.testing.assert_allclose(out[0], out[1], rtol=0, atol=1e-13 * np.abs(out[0]).max())
