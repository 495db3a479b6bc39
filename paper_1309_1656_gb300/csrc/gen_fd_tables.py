"""Writes fd_tables.h: the coefficient tables the library uses to evaluate
complete Fermi-Dirac integrals F_k(x) = -Li_{k+1}(-e^x) (Sec. 2.2) in double
precision on the GPU, for k = -1/2, 1/2, 3/2 (D3Q19) and k = 1 (D2Q9).

  x <= -1      F_k(x) = sum_{n>=1} (-1)^(n+1) e^(nx) / n^(k+1)   (SERIES: n^-(k+1))
  |x| < 1      F_k(x) = sum_j eta(k+1-j) x^j / j!                 (TAYLOR)
  1 <= x < 49  Chebyshev series on 24 intervals of width 2        (CHEB)
  x >= 49      x^(k+1)/Gamma(k+2) sum_n 2 eta(2n) (k+1)k...(k+2-2n) x^-2n  (ASYM)

For -8 <= x < 1, where one evaluation serves the one-pass solve, POLY holds
polynomials in x - c on 36 intervals of width 1/4 (c the centre) for
(F_{h-2}, F_{h-1}, F_h), h = 1 and 3/2, interpolated at the Chebyshev points
(error below 1e-18 of F_k), and POLYF those of F_{h-3} in single precision.

Values come from mpmath at 40 digits (polylog and altzeta); the FDF_*
tables are single-precision truncations of the same expansions.  Run with
`python gen_fd_tables.py` from this directory; the output is committed so
building the library needs no mpmath.  k = 1 uses only SERIES and TAYLOR
(the library reflects F_1(x) = x^2/2 + pi^2/6 - F_1(-x) for x > 0).
"""
import os

import mpmath as mp

mp.mp.dps = 40
KS = [mp.mpf(-1) / 2, mp.mpf(1) / 2, mp.mpf(3) / 2, mp.mpf(1)]
NSER, NTAY, NINT, WIDTH, X0, NCHEB, NASYM = 40, 34, 24, 2, 1, 24, 9
NSERF, NTAYF, NCHEBF, NASYMF = 20, 17, 10, 4
PX0, PINT, PDEG, PDEGF = -8, 36, 10, 4


def F(k, x):
    return -mp.re(mp.polylog(k + 1, -mp.exp(x)))


def cheb_coeffs(k, a, b, n):
    # c_j = (2/n) sum_m f(x_m) cos(j theta_m), theta_m = pi (m + 1/2) / n
    nodes = [mp.pi * (m + mp.mpf(1) / 2) / n for m in range(n)]
    vals = [F(k, (a + b) / 2 + (b - a) / 2 * mp.cos(t)) for t in nodes]
    c = []
    for j in range(n):
        s = mp.fsum(v * mp.cos(j * t) for v, t in zip(vals, nodes))
        c.append(2 * s / n)
    c[0] /= 2
    return c


def poly_coeffs(k, c, r, deg):
    """Monomial coefficients in x - c of the interpolant of F_k of degree deg
    at the Chebyshev points of [c - r, c + r]."""
    n = deg + 1
    t = [r * mp.cos(mp.pi * (m + mp.mpf(1) / 2) / n) for m in range(n)]
    A = mp.matrix(n, n)
    for i in range(n):
        for j in range(n):
            A[i, j] = (t[i] / r) ** j
    v = mp.lu_solve(A, mp.matrix([F(k, c + x) for x in t]))
    return [v[j] / r ** j for j in range(n)]


def fmt(v):
    return "%.17e" % float(v)


def fmtf(v):
    return "%.9ef" % float(v)


def main():
    out = []
    out.append("// Generated by gen_fd_tables.py (mpmath, 40 digits). Do not edit.")
    out.append("// Coefficients for complete Fermi-Dirac integrals F_k, k = -1/2, 1/2, 3/2, 1.")
    out.append("#pragma once")
    out.append("#define FD_NSER %d\n#define FD_NTAY %d\n#define FD_NINT %d\n#define FD_WIDTH %d" % (NSER, NTAY, NINT, WIDTH))
    out.append("#define FD_X0 %d\n#define FD_NCHEB %d\n#define FD_NASYM %d" % (X0, NCHEB, NASYM))
    ser = [[1 / mp.power(n, k + 1) for n in range(1, NSER + 1)] for k in KS]
    tay = [[mp.altzeta(k + 1 - j) / mp.factorial(j) for j in range(NTAY)] for k in KS]
    out.append("__constant__ double FD_SERIES[4][FD_NSER] = {")
    out += ["  {" + ", ".join(fmt(v) for v in row) + "}," for row in ser]
    out.append("};")
    out.append("__constant__ double FD_TAYLOR[4][FD_NTAY] = {")
    out += ["  {" + ", ".join(fmt(v) for v in row) + "}," for row in tay]
    out.append("};")
    out.append("__constant__ double FD_CHEB[3][FD_NINT][FD_NCHEB] = {")
    cheb = []
    for k in KS[:3]:
        out.append("  {")
        cheb.append([])
        for i in range(NINT):
            a = X0 + WIDTH * i
            c = cheb_coeffs(k, mp.mpf(a), mp.mpf(a + WIDTH), NCHEB)
            cheb[-1].append(c)
            out.append("    {" + ", ".join(fmt(v) for v in c) + "},")
        out.append("  },")
    out.append("};")
    asym = []
    for k in KS[:3]:
        row = [1 / mp.gamma(k + 2)]
        for n in range(1, NASYM):
            prod = mp.mpf(1)
            for m in range(2 * n):
                prod *= (k + 1 - m)
            row.append(2 * mp.altzeta(2 * n) * prod)
        asym.append(row)
    out.append("// ASYM[k][0] = 1/Gamma(k+2), ASYM[k][n] = 2 eta(2n) (k+1)k...(k+2-2n)")
    out.append("__constant__ double FD_ASYM[3][FD_NASYM] = {")
    out += ["  {" + ", ".join(fmt(v) for v in row) + "}," for row in asym]
    out.append("};")
    # Single-precision copies for the float solve, truncated where the
    # dropped terms are below ~1e-9 relative: series 20 terms (x <= -1,
    # q^20 < 2e-9), Taylor 17 (|x| < 1, pi^-17 < 4e-9), Chebyshev 10
    # (tail < 1e-9 on every interval), Sommerfeld 4 (x >= 49).
    out.append("#define FDF_NSER %d\n#define FDF_NTAY %d\n#define FDF_NCHEB %d\n#define FDF_NASYM %d"
               % (NSERF, NTAYF, NCHEBF, NASYMF))
    out.append("__constant__ float FDF_SERIES[4][FDF_NSER] = {")
    out += ["  {" + ", ".join(fmtf(v) for v in row[:NSERF]) + "}," for row in ser]
    out.append("};")
    out.append("__constant__ float FDF_TAYLOR[4][FDF_NTAY] = {")
    out += ["  {" + ", ".join(fmtf(v) for v in row[:NTAYF]) + "}," for row in tay]
    out.append("};")
    out.append("__constant__ float FDF_CHEB[3][FD_NINT][FDF_NCHEB] = {")
    for c_k in cheb:
        out.append("  {")
        for c in c_k:
            out.append("    {" + ", ".join(fmtf(v) for v in c[:NCHEBF]) + "},")
        out.append("  },")
    out.append("};")
    out.append("__constant__ float FDF_ASYM[3][FDF_NASYM] = {")
    out += ["  {" + ", ".join(fmtf(v) for v in row[:NASYMF]) + "}," for row in asym]
    out.append("};")
    # polynomials on the intervals of the one-pass solve
    out.append("#define FD_PX0 %d\n#define FD_PINT %d\n#define FD_PDEG %d\n#define FD_PDEGF %d" % (PX0, PINT, PDEG, PDEGF))
    for name, typ, deg, cols, f in (("FD_POLY", "double", PDEG, 3, fmt), ("FDF_POLY", "float", PDEGF, 1, fmtf)):
        out.append("static __device__ const %s %s[2][FD_PINT][%s + 1][%d] = {" % (typ, name, "FD_PDEG" if cols == 3 else "FD_PDEGF", cols))
        for h in (mp.mpf(1), mp.mpf(3) / 2):
            out.append("  {")
            for i in range(PINT):
                c = mp.mpf(PX0) + (i + mp.mpf(1) / 2) / 4
                ks = [h - 2, h - 1, h] if cols == 3 else [h - 3]
                p = [poly_coeffs(k, c, mp.mpf(1) / 8, deg) for k in ks]
                out.append("    {" + ", ".join("{" + ", ".join(f(q[j]) for q in p) + "}" for j in range(deg + 1)) + "},")
            out.append("  },")
        out.append("};")
    here = os.path.dirname(os.path.abspath(__file__))
    with open(os.path.join(here, "fd_tables.h"), "w") as f:
        f.write("\n".join(out) + "\n")


if __name__ == "__main__":
    main()
