"""Writes ``pair_tables.h``: the float-pair flux kernel's function tables.

1. Phi(s) = erfc(-s)/2 and phi(s) = exp(-s^2)/sqrt(pi) = Phi'(s) on [-6, 6]:
768 intervals of width 1/64 with centres c_k = -6 + (k + 1/2)/64. A row holds
the Chebyshev interpolant of degree 6 of Phi in z = s - c_k (mpmath, 50
digits): a_0, a_1, a_2 and 3 a_3 as pairs of floats (hi + lo, for the Horner
steps whose terms exceed 2^-24 of the result) and a_3 .. a_6 as floats. phi is
the derivative of the same polynomial, so one row serves both.

2. 2^(j/64), j < 64, as pairs of floats, and ln2/64 in three floats whose
first has 11 significant bits (its products with the reduction's integer, up
to 13 bits, are exact).

3. ln x by table, x = 2^e m: for m's top seven bits j, F_j = 1/(1 + (j +
1/2)/128) rounded to eight significant bits (so that m F_j - 1 is exact in a
float) and -ln F_j as a pair of floats; ln2 in three floats whose first has 12
significant bits.

Run: python gen_pair_tables.py  (writes pair_tables.h next to this file)
"""

import os

import mpmath as mp
import numpy as np

mp.mp.dps = 50

LO, HI, INV_W = -6, 6, 64
DEG = 6
EXP_BITS = 6


def split(x, parts=2):
    """x as a sum of floats, each the rounding of what is left."""
    out = []
    for _ in range(parts):
        f = float(np.float32(float(x)))
        out.append(f)
        x = x - mp.mpf(f)
    return out


def interpolant(f, lo, hi, centre):
    """Monomial coefficients in (s - centre) of the Chebyshev interpolant."""
    n = DEG + 1
    nodes = [(lo + hi) / 2 + (hi - lo) / 2 * mp.cos(mp.pi * (k + mp.mpf(1) / 2) / n) for k in range(n)]
    A = mp.matrix(n, n)
    for i, u in enumerate(nodes):
        for j in range(n):
            A[i, j] = (u - centre) ** j
    c = mp.lu_solve(A, mp.matrix([f(u) for u in nodes]))
    return [c[j] for j in range(n)]


def main(path=None):
    rows, worst, worst_d = [], mp.mpf(0), mp.mpf(0)
    for k in range((HI - LO) * INV_W):
        lo = mp.mpf(LO) + mp.mpf(k) / INV_W
        hi, c = lo + mp.mpf(1) / INV_W, lo + mp.mpf(1) / (2 * INV_W)
        a = interpolant(lambda s: mp.erfc(-s) / 2, lo, hi, c)
        for t in range(9):
            s = lo + (hi - lo) * t / 8
            z = s - c
            p = sum(a[i] * z ** i for i in range(DEG + 1))
            d = sum(i * a[i] * z ** (i - 1) for i in range(1, DEG + 1))
            worst = max(worst, abs(p - mp.erfc(-s) / 2))
            worst_d = max(worst_d, abs(d - mp.exp(-s * s) / mp.sqrt(mp.pi)))
        row = split(a[0]) + split(a[1]) + split(a[2]) + split(3 * a[3])
        rows.append(row + [float(np.float32(float(a[i]))) for i in range(3, 7)])
    assert worst < 1e-18 and worst_d < 3e-15, (worst, worst_d)
    n_exp = 1 << EXP_BITS
    ln2_n = mp.log(2) / n_exp
    e = int(mp.floor(mp.log(ln2_n, 2)))
    l1 = mp.floor(ln2_n / mp.mpf(2) ** (e - 10)) * mp.mpf(2) ** (e - 10)  # 11 significant bits
    l2, l3 = split(ln2_n - l1)
    if path is None:
        path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "pair_tables.h")
    with open(path, "w") as f:
        f.write("// Generated by gen_pair_tables.py -- do not edit.\n#pragma once\n\nnamespace lskum {\n\n")
        f.write("// {a0 hi, lo, a1 hi, lo, a2 hi, lo, 3 a3 hi, lo, a3, a4, a5, a6} of Phi(s) = erfc(-s)/2 in\n"
                f"// z = s - c_k; interpolation error {float(worst):.1e}, of the derivative "
                f"{float(worst_d):.1e}.\n")
        f.write(f"constexpr int kPhiPieces = {len(rows)};\nconstexpr float kPhiLo = {float(LO)!r}f;\n"
                f"constexpr float kPhiInvW = {float(INV_W)!r}f;\n")
        f.write("alignas(16) __device__ const float kPhiTab[kPhiPieces][12] = {\n")
        for r in rows:
            f.write("    {" + ", ".join(f"{v!r}f" for v in r) + "},\n")
        f.write("};\n\n")
        f.write(f"constexpr int kPairExpBits = {EXP_BITS};\n")
        f.write(f"constexpr float kPairLn2N1 = {float(l1)!r}f;\nconstexpr float kPairLn2N2 = {l2!r}f;\n"
                f"constexpr float kPairLn2N3 = {l3!r}f;\n")
        f.write(f"constexpr float kPairInvLn2N = {float(np.float32(float(1 / ln2_n)))!r}f;\n")
        f.write(f"alignas(8) __device__ const float kPairExp2[{n_exp}][2] = {{\n")
        for j in range(n_exp):
            h, l = split(mp.mpf(2) ** (mp.mpf(j) / n_exp))
            f.write(f"    {{{h!r}f, {l!r}f}},\n")
        f.write("};\n\n")
        ln2_hi = mp.floor(mp.log(2) * 2 ** 12) / 2 ** 12
        ln2_mid, ln2_lo = split(mp.log(2) - ln2_hi)
        f.write("// {F_j, -ln F_j hi, lo, 0}\n")
        f.write(f"constexpr float kPairLn2Hi = {float(ln2_hi)!r}f;\nconstexpr float kPairLn2Mid = {ln2_mid!r}f;\n"
                f"constexpr float kPairLn2Lo = {ln2_lo!r}f;\n")
        f.write("alignas(16) __device__ const float kPairLog[128][4] = {\n")
        for j in range(128):
            F = 1 / (1 + (mp.mpf(j) + mp.mpf(1) / 2) / 128)
            F = mp.nint(F * 2 ** 8) / 2 ** 8  # in (1/2, 1]: eight bits
            h, l = split(-mp.log(F))
            f.write(f"    {{{float(F)!r}f, {h!r}f, {l!r}f, 0.0f}},\n")
        f.write("};\n\n}  // namespace lskum\n")
    print(f"wrote {path}: {len(rows)} pieces, error {float(worst):.1e}, derivative {float(worst_d):.1e}")


if __name__ == "__main__":
    main()
