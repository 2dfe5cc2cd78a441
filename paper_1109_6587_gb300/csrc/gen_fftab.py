"""Writes ggem_fftab.cuh: the smooth parts of the GGEM local kernels in float
pairs, for the double-float element rule.

With lengths in units of 1/(sqrt(2) alpha), rho the scaled distance and
s = rho^2 = 2 alpha^2 r^2, the local Stokeslet and stresslet of Eq. (local) are
  G^l: A = 1/rho   - A_g(s),  B = 1/rho^3 - B_g(s)   (times sqrt(2) alpha),
  T^l: D = D_g(s) - 1/rho^5,  E = E_g(s)             (times 12 alpha^2),
where, with I_m(s) = int_0^1 t^m exp(-s t^2 / 2) dt and c = sqrt(2 / pi),
  A_g = c (I_0 + exp(-s/2)),  B_g = c I_2,  D_g = c I_4 / 3,  E_g = c exp(-s/2) / 6
(erf(rho / sqrt 2) = c rho I_0; the others by parts) are entire in s: no
exponential, no erfc and no division remain per pair beyond 1/rho.

Each is a polynomial of degree 9 in u = s - i on the intervals |s - i| <= 1/2,
i = 0 .. 72 (exp(-36) is below the last bit of a double): the Chebyshev
interpolant at the first-kind points, in monomials, by mpmath at 50 digits;
degrees 0..6 as float pairs, 7..9 as floats (their terms are below 2e-8).
Run: python gen_fftab.py > ggem_fftab.cuh

The FP64 sums take the same functions in doubles, of degree 10 (truncation below
2e-17 of each function's largest value), near the target.  Farther out 1/rho - A_g
and the like are differences of nearly equal numbers (the local kernels fall as
exp(-s/2)), so from s = 3.5 on they take the local kernels themselves, scaled,
  1 - rho A_g, 1 - rho^3 B_g, 1 - rho^5 D_g = erfc(x) - w, erfc(x) + w,
  erfc(x) + w (1 + 2 x^2 / 3),  x = rho / sqrt 2,  w = 2 x exp(-x^2) / sqrt(pi),
in the same degree and intervals (relative truncation below 1e-15 where they are
used: A and B from interval 6, D from interval 4).
Run: python gen_fftab.py fp64 > ggem_smooth64.cuh
"""
import sys

import mpmath as mp
import numpy as np

mp.mp.dps = 50
NINT, DEG, PAIRS, DEG64, FAR0 = 73, 9, 7, 10, 4


def smooth(m, s):
    return mp.hyp1f1(mp.mpf(m + 1) / 2, mp.mpf(m + 3) / 2, -s / 2) / (m + 1)


C = mp.sqrt(2 / mp.pi)
FUNCS = [lambda s: C * (smooth(0, s) + mp.exp(-s / 2)), lambda s: C * smooth(2, s),
         lambda s: C * smooth(4, s) / 3, lambda s: C * mp.exp(-s / 2) / 6]
FAR = [lambda s, k=k: 1 - mp.sqrt(s) ** (2 * k + 1) * FUNCS[k](s) for k in range(3)]


def interpolant(f, i, deg=DEG):
    """Monomial coefficients in u of f(i + u), |u| <= 1/2."""
    n = deg + 1
    v = [mp.cos(mp.pi * (k + mp.mpf(1) / 2) / n) for k in range(n)]
    y = [f(i + x / 2) for x in v]
    c = [2 * mp.fsum(y[k] * mp.cos(j * mp.pi * (k + mp.mpf(1) / 2) / n) for k in range(n)) / n
         for j in range(n)]
    c[0] /= 2
    T = [[mp.mpf(1)], [mp.mpf(0), mp.mpf(1)]]
    for j in range(2, n):
        t = [mp.mpf(0)] + [2 * a for a in T[-1]]
        for k, a in enumerate(T[-2]):
            t[k] -= a
        T.append(t)
    out = [mp.mpf(0)] * n
    for j in range(n):
        for k, a in enumerate(T[j]):
            out[k] += c[j] * a
    return [a * mp.mpf(2) ** k for k, a in enumerate(out)]      # v = 2 u


def hexf(x):
    m, e = float(np.float32(x)).hex().split("p")
    return m.rstrip("0").rstrip(".") + "p" + str(int(e)) + "f"


def main():
    print("// Generated by gen_fftab.py (mpmath, 50 digits): A_g, B_g, D_g, E_g on |s - i| <= 1/2,")
    print("// degree %d in u = s - i.  kFFPair[function][degree][interval] = (hi, lo) of degrees" % DEG)
    print("// 0..%d; kFFTail[function][interval] = degrees %d..%d as floats." % (PAIRS - 1, PAIRS, DEG))
    print("#pragma once")
    print("#define GGEM_FF_NINT %d" % NINT)
    print("#define GGEM_FF_PAIRS %d" % PAIRS)
    tab = [[interpolant(f, i) for i in range(NINT)] for f in FUNCS]
    print("__device__ const float2 kFFPair[4][%d][%d] = {" % (PAIRS, NINT))
    for t in tab:
        print("    {")
        for k in range(PAIRS):
            row = []
            for i in range(NINT):
                h = float(np.float32(float(t[i][k])))
                row.append("{%s,%s}" % (hexf(h), hexf(float(t[i][k] - mp.mpf(h)))))
            print("        {" + ",\n         ".join(",".join(row[j:j + 4]) for j in range(0, NINT, 4))
                  + "},")
        print("    },")
    print("};")
    print("__device__ const float4 kFFTail[4][%d] = {" % NINT)
    for t in tab:
        print("    {")
        for i in range(NINT):
            print("        {" + ",".join(hexf(float(t[i][k])) for k in range(PAIRS, DEG + 1))
                  + ",0.f},")
        print("    },")
    print("};")


def table64(name, rows):
    """rows[function][degree][interval]"""
    print("__device__ const double %s[%d][%d][%d] = {" % (name, len(rows), DEG64 + 1, NINT))
    for tab in rows:
        print("    {")
        for row in tab:
            print("        {" + ",\n         ".join(", ".join(row[j:j + 4])
                                                    for j in range(0, NINT, 4)) + "},")
        print("    },")
    print("};")


def main64():
    print("// Generated by gen_fftab.py fp64 (mpmath, 50 digits), degree %d in u = s - i on" % DEG64)
    print("// |s - i| <= 1/2, as [function][degree][interval]: kFar64 the scaled local kernels")
    print("// 1 - rho A_g, 1 - rho^3 B_g, 1 - rho^5 D_g (zero below interval %d, where they are" % FAR0)
    print("// not used), kSmooth64 A_g, B_g, D_g, E_g.")
    print("#pragma once")
    print("#define GGEM_SMOOTH64_NINT %d" % NINT)
    print("#define GGEM_SMOOTH64_DEG %d" % DEG64)

    def rows(f, i0):
        tab = [interpolant(f, i, DEG64) if i >= i0 else [mp.mpf(0)] * (DEG64 + 1)
               for i in range(NINT)]
        return [[float(tab[i][k]).hex() for i in range(NINT)] for k in range(DEG64 + 1)]
    table64("kFar64", [rows(f, FAR0) for f in FAR])
    table64("kSmooth64", [rows(f, 0) for f in FUNCS])


if __name__ == "__main__":
    main64() if sys.argv[1:] == ["fp64"] else main()
