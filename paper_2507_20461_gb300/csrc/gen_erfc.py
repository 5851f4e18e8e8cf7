"""Generate erfc_table.cuh: the approximations of erfc and exp(-x^2) behind the
half-space moments of the FP64 gas-kinetic flux.

On each interval |x - k/32| <= 1/64, k = 0 .. 96, the degree-8 Chebyshev
interpolants of erfc(x) and exp(-x^2), as polynomials in x - x_k (their
truncation is below 2^-55 of the value there; checked here).  The x_k are
accurate table points (Gal's method): the first double k/32 + j 2^-40, j = 0, 1,
.., at which both functions lie within 1/64 of a unit in the last place of a
double, so that the constant terms carry no rounding and a result little more
than its last operation's.  All arithmetic in mpmath at 50 digits from the
functions' definitions.

Run: python gen_erfc.py (writes erfc_table.cuh beside it)."""
import math
import os

import mpmath as mp

mp.mp.dps = 50
HERE = os.path.dirname(os.path.abspath(__file__))
DEG, STEP, ROWS = 8, 32, 97
FUNCTIONS = (mp.erfc, lambda x: mp.exp(-x * x))


def off_grid(v):
    """distance of v from the nearest double, in units of its last place"""
    f = float(v)
    return abs(v - mp.mpf(f)) / (mp.mpf(2) ** (math.frexp(f)[1] - 53))


def node(k):
    j = 0
    while True:
        x = mp.mpf(k) / STEP + mp.mpf(j) / 2**40
        if all(off_grid(f(x)) <= mp.mpf(1) / 64 for f in FUNCTIONS):
            return x
        j += 1


def interpolant(f, c, r, deg):
    """monomial coefficients in x - c of the Chebyshev interpolant of f on |x - c| <= r"""
    n = deg + 1
    nodes = [mp.cos(mp.pi * (2 * i + 1) / (2 * n)) for i in range(n)]
    A = mp.matrix(n, n)
    b = mp.matrix(n, 1)
    for i, z in enumerate(nodes):
        for j in range(n):
            A[i, j] = z**j
        b[i] = f(c + r * z)
    a = mp.lu_solve(A, b)
    return [a[j] / mp.mpf(r) ** j for j in range(n)]


def horner(a, d):
    s = mp.mpf(0)
    for c in reversed(a):
        s = s * d + c
    return s


def table():
    rows, worst = [], mp.mpf(0)
    r = mp.mpf(1) / (2 * STEP)
    for k in range(ROWS):
        c = node(k)
        row = []
        for f in FUNCTIONS:
            a = interpolant(f, c, r, DEG)
            for i in range(-16, 17):
                d = r * i / 16
                worst = max(worst, abs(horner(a, d) / f(c + d) - 1))
            row.append([float(f(c))] + [float(v) for v in a[1:]])
        rows.append(row + [[float(c), 0.0]])
    assert worst < mp.mpf(2) ** -55, worst
    return rows, worst


def main():
    rows, worst = table()
    L = ["/* Generated by gen_erfc.py (Chebyshev interpolation, 50 digits).  Do not edit. */", "#pragma once", "",
         f"/* FP64: row k, polynomials in x - x_k on |x - k/{STEP}| <= 1/{2 * STEP}, x < 3: erfc(x) coefficients 0..{DEG},",
         f" * exp(-x^2) coefficients 0..{DEG}, x_k (k/{STEP} but for less than 2^-20) and 0; worst relative truncation {mp.nstr(worst, 2)}. */",
         f"#define ERFC_DEG {DEG}", f"#define ERFC_STEP {STEP}", f"#define ERFC_ROWS {ROWS}",
         f"static __device__ __align__(16) const double erfc_rows[ERFC_ROWS][2 * (ERFC_DEG + 1) + 2] = {{"]
    for row in rows:
        L.append("    {" + ", ".join(repr(v) for f in row for v in f) + "},")
    L += ["};", ""]
    with open(os.path.join(HERE, "erfc_table.cuh"), "w") as f:
        f.write("\n".join(L))
    print("truncation", mp.nstr(worst, 3))


if __name__ == "__main__":
    main()
