"""The multi-D step assembled on the CPU from the item functions that the step's
kernels run (the reconstruction into the grouped layout, step_face_item,
step_update_item; csrc/step_flux.cuh) through the test-only CUDA stand-in,
against the oracle's step: every boundary type and mixed sides, the weight
variants, Euler and Navier-Stokes, sizes from one cell across to past a group of
32 cells and faces, FP64 and mixed precision.

Bars: FP64 the step's (relative L1 1e-12 per variable, gradients 1e-11).  Mixed: the
FP32 flux is good to 2e-5 of its size at a point (test_gks_point_host.py) and a
step adds the differences of two faces a direction times dt / h < 0.3 in each of
two stages, so 2e-5 of the largest value; gradients are differences of interface
states over h, 1e-4 of it over h."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2507_20461_gb300", "csrc")

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("sp") / "step_path_check")
    r = subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(HERE, "hostshim"), "-I", CSRC,
                        os.path.join(HERE, "step_path_check.cpp"), "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


def _state(n, seed):
    m, rng = len(n), np.random.default_rng(seed)
    X = np.meshgrid(*[(np.arange(k) + 0.5) / k for k in reversed(n)], indexing="ij")
    rho = 1.0 + 0.2 * sum(np.sin(2 * np.pi * x + rng.uniform(0, 6)) for x in X)
    vel = [0.3 * np.cos(2 * np.pi * X[-1 - a] + rng.uniform(0, 6)) for a in range(m)]
    p = 1.0 + 0.1 * sum(np.cos(2 * np.pi * x + rng.uniform(0, 6)) for x in X)
    W = np.array([rho, *(rho * v for v in vel), p / 0.4 + 0.5 * rho * sum(v * v for v in vel)])
    h = 1.0 / max(n)
    G = np.zeros((m,) + W.shape)
    for a in range(m):
        if n[a] > 2:
            G[a] = np.gradient(W, h, axis=1 + (m - 1 - a))
    return W, G, h


CASES = [  # n, sides, limiter, mu
    ((12, 10), (0, 0, 0, 0), 0, 0.0),
    ((33, 7), (1, 1, 1, 1), 0, 0.0),
    ((1, 9), (2, 2, 0, 0), 2, 0.0),
    ((40, 1), (0, 0, 3, 3), 1, 0.0),
    ((31, 34), (3, 2, 2, 3), 0, 0.0),
    ((16, 16), (3, 3, 3, 2), 0, 0.01),
    ((9, 11), (0, 0, 0, 0), 3, 0.0),
    ((6, 5, 4), (0, 0, 0, 0, 0, 0), 0, 0.0),
    ((4, 6, 5), (1, 1, 2, 2, 3, 3), 2, 0.0),
    ((3, 1, 7), (0, 0, 3, 1, 2, 1), 0, 0.01),
    ((7, 5, 3), (2, 3, 0, 0, 1, 1), 1, 0.0),
]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,sides,lim,mu", CASES)
def test_step_of_the_kernels_items_matches_oracle(exe, oracle, n, sides, lim, mu, prec):
    if prec and lim == 3:
        pytest.skip("TENO's cut is a switch: FP32 rounding may flip it")
    m = len(n)
    W, G, h = _state(n, 13 * sum(n) + lim)
    cfg = oracle.make_cfg(m, n, h, bc=tuple(sides) + (0,) * (6 - len(sides)), limiter=lim, mu=mu)
    dt = 0.3 * h / oracle.max_wavespeed(cfg, W)
    text = "\n".join([repr(float(dt)), " ".join(repr(float(v)) for v in W.ravel()), " ".join(repr(float(v)) for v in G.ravel())]) + "\n"
    n3 = list(n) + [1] * (3 - m)
    r = subprocess.run([exe, str(m), *map(str, n3), repr(h), str(lim), repr(mu), str(prec), *map(str, tuple(sides) + (0,) * (6 - len(sides)))],
                       input=text, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    lines = r.stdout.strip().splitlines()
    Wg = np.array([float(t) for t in lines[0].split()]).reshape(W.shape)
    Gg = np.array([float(t) for t in lines[1].split()]).reshape(G.shape)
    assert int(lines[2]) == 0
    Wo, Go = W.copy(), G.copy()
    assert oracle.step(cfg, dt, Wo, Go) == 0
    top = np.abs(Wo).max()
    if prec:
        assert np.abs(Wg - Wo).max() <= 2e-5 * top
        assert np.abs(Gg - Go).max() <= 1e-4 * top / h
        return
    for v in range(m + 2):
        assert np.abs(Wg[v] - Wo[v]).sum() <= 1e-12 * max(np.abs(Wo[v]).sum(), np.abs(Wo[0]).sum())
    assert np.abs(Gg - Go).max() <= 1e-11 * top / h
