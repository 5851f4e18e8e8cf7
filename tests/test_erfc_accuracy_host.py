"""The error of the FP64 erfc / exp pair of the half-space moments (csrc/gks_device.cuh,
RT<double>::erfc_exp, host build) in units of the result's last place, against
mpmath, over its table's range.  Bar: 1/2 for the last sum, 1/64 for the constant
term (taken where the function is all but a double), and the roundings of the
other terms, which are at most 0.1 of the value (|x - x_k| <= 1/64, logarithmic
derivative below 6.3): two of half a unit each, a unit of the term weighing up
to twice one of the value: 0.92."""
import math
import os
import random
import shutil
import subprocess

import pytest

mp = pytest.importorskip("mpmath")

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2507_20461_gb300", "csrc")
pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <initializer_list>
#include "gks_device.cuh"
int main() { double a, h, e; while (std::scanf("%lf", &a) == 1) { gks::RT<double>::erfc_exp(a, h, e); std::printf("%.17g %.17g\n", h, e); } }
"""


def _ulps(v, true):
    return float(abs(mp.mpf(v) - true) / mp.mpf(2) ** (math.frexp(float(true))[1] - 53))


def test_table_is_good_to_a_unit(tmp_path):
    (tmp_path / "t.cpp").write_text(SRC)
    exe = str(tmp_path / "t")
    r = subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(HERE, "hostshim"), "-I", CSRC, str(tmp_path / "t.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    rng = random.Random(5)
    pts = [rng.uniform(0, 3) for _ in range(3000)] + [rng.uniform(0, 0.7) for _ in range(3000)]
    out = subprocess.run([exe], input="\n".join(map(repr, pts)), capture_output=True, text=True).stdout.split()
    mp.mp.dps = 40
    for p, h, e in zip(pts, out[::2], out[1::2]):
        assert _ulps(float(h), mp.erfc(mp.mpf(p))) <= 0.92, p
        assert _ulps(float(e), mp.exp(-(mp.mpf(p) ** 2))) <= 0.92, p
