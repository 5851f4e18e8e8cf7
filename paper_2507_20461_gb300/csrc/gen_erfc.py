"""Generate erfc_table.cuh: the approximations of erfc and exp(-x^2) behind the
half-space moments of the FP64 gas-kinetic flux.

On each interval |x - k/32| <= 1/64, k = 0 .. 96, the degree-8 Chebyshev
interpolants of erfc(x) and exp(-x^2), as polynomials in x - k/32 (their
truncation is below 2^-55 of the value there; checked here).  All arithmetic in
mpmath at 50 digits; the method is plain Chebyshev interpolation of the
functions' definitions.

Run: python gen_erfc.py (writes erfc_table.cuh beside it)."""
import os

import mpmath as mp

mp.mp.dps = 50
HERE = os.path.dirname(os.path.abspath(__file__))
DEG, STEP, ROWS = 8, 32, 97


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
        c = mp.mpf(k) / STEP
        row = []
        for f in (mp.erfc, lambda x: mp.exp(-x * x)):
            a = interpolant(f, c, r, DEG)
            for i in range(-16, 17):
                d = r * i / 16
                worst = max(worst, abs(horner(a, d) / f(c + d) - 1))
            row.append([float(v) for v in a])
        rows.append(row)
    assert worst < mp.mpf(2) ** -55, worst
    return rows, worst


def main():
    rows, worst = table()
    L = ["/* Generated by gen_erfc.py (Chebyshev interpolation, 50 digits).  Do not edit. */", "#pragma once", "",
         f"/* FP64: row k, polynomials in x - k/{STEP} on |x - k/{STEP}| <= 1/{2 * STEP}, x < 3: erfc(x) coefficients 0..{DEG},",
         f" * then exp(-x^2) coefficients 0..{DEG}; worst relative truncation {mp.nstr(worst, 2)}. */",
         f"#define ERFC_DEG {DEG}", f"#define ERFC_STEP {STEP}", f"#define ERFC_ROWS {ROWS}",
         f"static __device__ __align__(16) const double erfc_rows[ERFC_ROWS][2 * (ERFC_DEG + 1)] = {{"]
    for row in rows:
        L.append("    {" + ", ".join(repr(v) for f in row for v in f) + "},")
    L += ["};", ""]
    with open(os.path.join(HERE, "erfc_table.cuh"), "w") as f:
        f.write("\n".join(L))
    print("truncation", mp.nstr(worst, 3))


if __name__ == "__main__":
    main()
