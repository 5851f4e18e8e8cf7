"""The face flux of a state and of the same state with averages, gradients and
viscosity times 2^k, on the CPU through the test-only CUDA stand-in: the
equations and the linear weights (limiter 1) have no absolute scale, so the
result is the flux times 2^k as long as the state itself is in range.  With a
density and pressure jump, so that the admissibility fallback is in play.

Bars: scaling by a power of two commutes with every rounding, so only what
leaves the format's range differs: FP64 1e-13 and FP32 1e-6 of the quantity's
largest value (a decision taken by another formula at the scaled state moves
by a rounding; the FP32 shadow's low part loses bits below 2^-126), dF/dt of
F / dt as well."""
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
    out = str(tmp_path_factory.mktemp("sc") / "state_scale_check")
    r = subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(HERE, "hostshim"), "-I", CSRC,
                        os.path.join(HERE, "state_scale_check.cpp"), "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


def _state(n, jump):
    m, rng = len(n), np.random.default_rng(5 * sum(n) + len(n))
    X = np.meshgrid(*[(np.arange(k) + 0.5) / k for k in reversed(n)], indexing="ij")
    rho = 1.0 + 0.2 * sum(np.sin(2 * np.pi * x + rng.uniform(0, 6)) for x in X)
    vel = [0.4 * np.cos(2 * np.pi * X[-1 - a] + rng.uniform(0, 6)) for a in range(m)]
    p = 1.0 + 0.1 * sum(np.cos(2 * np.pi * x + rng.uniform(0, 6)) for x in X)
    h = 1.0 / n[0]
    if jump:
        low = sum(X) > 0.5 * m
        rho, p = np.where(low, 0.06 * rho, rho), np.where(low, 0.05 * p, p)
    W = np.array([rho, *(rho * v for v in vel), p / 0.4 + 0.5 * rho * sum(v * v for v in vel)])
    G = np.stack([np.gradient(W, h, axis=1 + (m - 1 - a)) for a in range(m)])
    return W, G + rng.normal(scale=0.3, size=G.shape) * np.abs(W), h


def _check(exe, n, mu, prec, k, jump, bar):
    W, G, h = _state(n, jump)
    dt = 0.2 * h
    text = " ".join(repr(float(v)) for v in W.ravel()) + "\n" + " ".join(repr(float(v)) for v in G.ravel()) + "\n"
    n3 = list(n) + [1] * (3 - len(n))
    r = subprocess.run([exe, str(len(n)), *map(str, n3), repr(h), "1", repr(mu), repr(dt), str(prec), str(k), *"002211"],
                       input=text, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    F, Ft, Wh, st = [[float(x) for x in ln.split()] for ln in r.stdout.strip().splitlines()]
    assert st == [0.0, 0.0]
    assert F[0] <= bar * F[1]
    assert Ft[0] <= 10 * bar * (Ft[1] + F[1] / dt)
    assert Wh[0] <= bar * Wh[1]


GRIDS = [(12, 10), (6, 5, 4)]


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("mu,jump", [(0.0, False), (0.0, True), (0.01, False)])
@pytest.mark.parametrize("k", [-90, -75, -44, 40, 60])
def test_fp32_flux_scales_with_the_state(exe, n, mu, jump, k):
    _check(exe, n, mu, 1, k, jump, 1e-6)


@pytest.mark.parametrize("n", GRIDS + [(31,)])
@pytest.mark.parametrize("mu,jump", [(0.0, False), (0.0, True), (0.01, False)])
@pytest.mark.parametrize("k", [-400, -360, -300, 300, 345])
def test_fp64_flux_scales_with_the_state(exe, n, mu, jump, k):
    _check(exe, n, mu, 0, k, jump, 1e-13)


@pytest.mark.parametrize("n", GRIDS + [(31,)])
@pytest.mark.parametrize("mu,jump", [(0.0, False), (0.0, True), (0.01, False)])
@pytest.mark.parametrize("k", [-900, -520, -515, 515, 520, 900])
def test_fp64_flux_scales_past_the_root_of_the_range(exe, n, mu, jump, k):
    """pressures whose products leave the format: the relaxation time is a quotient of them"""
    _check(exe, n, mu, 0, k, jump, 1e-13)


def test_fp64_admissibility_matches_its_definition(tmp_path):
    exe = str(tmp_path / "admissible_check")
    r = subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(HERE, "hostshim"), "-I", CSRC,
                        os.path.join(HERE, "admissible_check.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    count, accepted, wrong = map(int, subprocess.run([exe], capture_output=True, text=True, timeout=60).stdout.split())
    assert count > 250000 and 0.1 * count < accepted < 0.9 * count and wrong == 0
