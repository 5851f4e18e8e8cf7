"""The multi-D step where its launches change form (small grids spread a cell's
variables and a face's Gauss points over threads), the wave speed left by a
step's last stage, the FP32 admissibility test's range, and states in and out
of buffers that the one-kernel transfer does and does not take.

The forms run the same formulas, so a periodic grid and the same grid
replicated past the line agree to rounding; smooth states, where rounding is
not amplified.  Bars: FP64 1e-12 of the largest value (the step's bar), mixed
1e-6 (averages; gradients 1e-4 of it over h), as the fused and unfused stages
are held to."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2507_20461_gb300 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _smooth(n, seed):
    """averages and gradients of a periodic state on n cells of side 1"""
    m, rng = len(n), np.random.default_rng(seed)
    X = [((np.arange(k) + 0.5) / k).reshape((-1,) + (1,) * a) for a, k in enumerate(n)]
    zero = 0 * sum(X)
    ph = [2 * np.pi * X[i % m] + rng.uniform(0, 6) for i in range(m + 2)]
    rho = 1 + 0.2 * np.sin(ph[0]) + zero
    vel = [0.3 * np.cos(ph[1 + i]) + zero for i in range(m)]
    W = np.stack([rho, *(rho * u for u in vel), (1 + 0.1 * np.sin(ph[m + 1])) / 0.4 + 0.5 * rho * sum(u * u for u in vel)])
    G = np.stack([(np.roll(W, -1, W.ndim - 1 - a) - np.roll(W, 1, W.ndim - 1 - a)) / 2 for a in range(m)])
    return np.ascontiguousarray(W), np.ascontiguousarray(G)


def _run(W, G, precision, run, **kw):
    n = tuple(reversed(W.shape[1:]))
    s = B.Solver(n, hi=[float(k) for k in n], precision=precision, **kw)
    Wd, Gd = torch.from_numpy(W).to(DEV), torch.from_numpy(G).to(DEV)
    s.set_state(Wd, Gd)
    run(s)
    Wo, Go = torch.empty_like(Wd), torch.empty_like(Gd)
    s.get_state(Wo, Go)
    s.close()
    return Wo.cpu().numpy(), Go.cpu().numpy()


@pytest.mark.parametrize("n,reps", [((5, 3), (90, 150)), ((63, 65), (6, 7)), ((33, 1), (9, 280)), ((7, 5, 6), (7, 9, 8))])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("mu,limiter", [(0.0, 0), (0.01, 2)])
def test_small_grid_is_the_replicated_one(n, reps, precision, mu, limiter):
    W, G = _smooth(n, 3)
    big = (1,) + tuple(reversed(reps))
    def run(s):
        for _ in range(3):
            s.step(0.1)
    Ws, Gs = _run(W, G, precision, run, mu=mu, limiter=limiter)
    Wb, Gb = _run(np.tile(W, big), np.tile(G, (1,) + big), precision, run, mu=mu, limiter=limiter)
    top = np.abs(Ws).max()
    tw, tg = (1e-6, 1e-4) if precision else (1e-12, 1e-11)
    assert np.abs(Wb - np.tile(Ws, big)).max() <= tw * top
    assert np.abs(Gb - np.tile(Gs, (1,) + big)).max() <= tg * top


@pytest.mark.parametrize("n", [(40, 24), (260, 300), (12, 9, 10), (40, 41, 42)])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("mu", [0.0, 0.05])
def test_cfl_steps_in_one_call_and_one_by_one(n, precision, mu):
    """The wave speed that a step leaves is the one a pass over its state finds, up to its rounding."""
    W, G = _smooth(n, 5)
    def one_by_one(s):
        for _ in range(4):
            s.step_cfl(0.4, 1)
    a = _run(W, G, precision, lambda s: s.step_cfl(0.4, 4), mu=mu)
    b = _run(W, G, precision, one_by_one, mu=mu)
    top = np.abs(a[0]).max()
    tw, tg = (1e-6, 1e-4) if precision else (1e-12, 1e-11)
    assert np.abs(a[0] - b[0]).max() <= tw * top and np.abs(a[1] - b[1]).max() <= tg * top


@pytest.mark.parametrize("n", [(40, 24), (300, 260), (12, 9, 10)])
@pytest.mark.parametrize("exponent", [-44, 40])
def test_mixed_step_scales_with_density(n, exponent):
    """rho, momentum and energy times 2^k: the step's result times 2^k (linear weights, which have no absolute scale)."""
    W, G = _smooth(n, 9)
    k = 2.0**exponent
    run = lambda s: s.step(0.1)  # noqa: E731
    W1, G1 = _run(W, G, 1, run, limiter=1)
    Wk, Gk = _run(W * k, G * k, 1, run, limiter=1)
    top = np.abs(W1).max()
    assert np.abs(Wk / k - W1).max() <= 1e-6 * top
    assert np.abs(Gk / k - G1).max() <= 1e-4 * top


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [(31, 17), (9, 8, 7), (50,)])
def test_state_through_every_kind_of_buffer(n, precision):
    """Device tensors, offset views of one, and host arrays give the same states in and out."""
    W, G = _smooth(n, 7)
    nw, ng = W.size, G.size
    s = B.Solver(n, hi=[float(k) for k in n], precision=precision)
    out = []
    for kind in ("device", "offset", "host"):
        if kind == "host":
            Wi, Gi = W.copy(), G.copy()
            Wo, Go = np.empty_like(W), np.empty_like(G)
        else:
            off = 0 if kind == "device" else 1
            buf = torch.empty(2 * (nw + ng + 1), dtype=torch.float64, device=DEV)
            parts = [buf[off + i : off + j] for i, j in ((0, nw), (nw, nw + ng), (nw + ng, 2 * nw + ng), (2 * nw + ng, 2 * (nw + ng)))]
            Wi, Gi, Wo, Go = (p.view(x.shape) for p, x in zip(parts, (W, G, W, G)))
            Wi.copy_(torch.from_numpy(W))
            Gi.copy_(torch.from_numpy(G))
        s.set_state(Wi, Gi)
        s.get_state(Wo, Go)
        host = [x if kind == "host" else x.cpu().numpy() for x in (Wo, Go)]
        assert np.array_equal(host[0], W) and np.array_equal(host[1], G), kind
        s.step_cfl(0.4, 2)
        for _ in range(2):  # reading twice reads the same
            s.get_state(Wo, Go)
            out.append([np.array(x if kind == "host" else x.cpu().numpy()) for x in (Wo, Go)])
    s.close()
    for w, g in out[1:]:
        assert np.array_equal(w, out[0][0]) and np.array_equal(g, out[0][1])
