"""The FP64 erfc / exp pair of the half-space moments (csrc/gks_device.cuh,
RT<double>::erfc_exp, host build) against mpmath: on the interval edges and
centres of its table, around the line to the library functions, signs, zero,
and values past it.  Bar: truncation below 2^-55, then one rounding of the
argument (exact), of each of the 8 Horner steps scaled by |d| <= 1/64 and of the
reflection 2 - h: 2 ulp of erfc's scale 1 for negative arguments, 2 ulp
relative for positive ones; past the table the library's error grows with
the argument's square (x^2 rounded before the exponential): 2 + x^2 ulp."""
import os
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


def test_erfc_exp_pair(tmp_path):
    (tmp_path / "t.cpp").write_text(SRC)
    exe = str(tmp_path / "t")
    r = subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(HERE, "hostshim"), "-I", CSRC, str(tmp_path / "t.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    pts = [k / 64 + d for k in range(0, 194) for d in (0.0, 1e-9, 0.0031, 0.0077)] + [2.9999999999999996, 3.0, 3.5, 5.0, 8.0, 1e-300]
    pts += [-p for p in pts]
    out = subprocess.run([exe], input="\n".join(repr(p) for p in pts), capture_output=True, text=True).stdout.split()
    mp.mp.dps = 40
    ulp = mp.mpf(2) ** -52
    for p, h, e in zip(pts, out[::2], out[1::2]):
        x = mp.mpf(p)
        wide = 2 + (x * x if abs(p) >= 3 else 0)
        assert abs(mp.mpf(h) - mp.erfc(x)) <= wide * ulp * (mp.erfc(x) if p > 0 else 1), p
        assert abs(mp.mpf(e) / mp.exp(-x * x) - 1) <= wide * ulp, p
