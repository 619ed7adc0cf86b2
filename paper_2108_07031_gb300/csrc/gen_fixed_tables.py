"""Writes ``fixed_tables.h``: the 64-bit fixed-point tables of the FP64 flux's
large steps.

1. 2^(j/256), j < 256, in units of 2^-63, and the coefficients (ln2/256)^m / m!
of 2^(h/256) - 1 for h in [0, 1): m = 1..3 in units of 2^-72, 4 in units of
2^-70, 5 in units of 2^-72 (the two last fit 32 bits).

2. erfcx(a) = e^(a^2) erfc(a) on [0, 6]: 384 intervals of width 1/64, each the
Chebyshev interpolant of degree 6 (mpmath, 50 digits) as b_0 - h (b_1 - h (b_2 -
...)) in h = 64 a - k: the derivatives of erfcx alternate in sign, so that every
b is positive. Units of 2^-63, b_5 and b_6 fit 32 bits.

Run: python gen_fixed_tables.py  (writes fixed_tables.h next to this file)
"""

import os

import mpmath as mp

mp.mp.dps = 50

PIECES, INV_W, DEG = 384, 64, 6


def erfcx(a):
    return mp.exp(a * a) * mp.erfc(a)


def interpolant(lo):
    """Coefficients in h = (a - lo) INV_W on [0, 1)."""
    n = DEG + 1
    nodes = [mp.mpf(1) / 2 + mp.cos(mp.pi * (k + mp.mpf(1) / 2) / n) / 2 for k in range(n)]
    A = mp.matrix(n, n)
    for i, h in enumerate(nodes):
        for j in range(n):
            A[i, j] = h ** j
    c = mp.lu_solve(A, mp.matrix([erfcx(lo + h / INV_W) for h in nodes]))
    return [c[j] for j in range(n)]


def units(x, bits):
    return int(mp.nint(x * mp.mpf(2) ** bits))


def main(path=None):
    rows, worst = [], mp.mpf(0)
    for k in range(PIECES):
        lo = mp.mpf(k) / INV_W
        c = interpolant(lo)
        for t in range(9):
            h = mp.mpf(t) / 8
            f = erfcx(lo + h / INV_W)
            worst = max(worst, abs(sum(c[m] * h ** m for m in range(DEG + 1)) / f - 1))
        b = [units(c[m] * (-1) ** m, 63) for m in range(DEG + 1)]
        assert min(b) > 0 and max(b[5:]) < 1 << 32 and b[0] <= 1 << 63
        rows.append(b)
    assert worst < 1e-17, worst
    e = mp.log(2) / 256
    a = [e ** m / mp.factorial(m) for m in range(1, 6)]
    if path is None:
        path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fixed_tables.h")
    with open(path, "w") as f:
        f.write("// Generated by gen_fixed_tables.py -- do not edit.\n#pragma once\n\n"
                "#include <cstdint>\n\nnamespace lskum {\n\n")
        for m in range(3):
            f.write(f"constexpr uint64_t kFixE{m + 1} = 0x{units(a[m], 72):016x}ULL;\n")
        f.write(f"constexpr uint32_t kFixE4 = 0x{units(a[3], 70):08x}u, kFixE5 = 0x{units(a[4], 72):08x}u;\n")
        f.write(f"constexpr uint64_t kFixLog2e = 0x{units(1 / mp.log(2), 63):016x}ULL;  // units of 2^-63\n")
        f.write(f"constexpr uint64_t kFixHalfIsqPi = 0x{units(1 / (2 * mp.sqrt(mp.pi)), 64):016x}ULL;"
                "  // 1/(2 sqrt(pi)), units of 2^-64\n")
        f.write(f"constexpr int kFixPieces = {PIECES};\n\n")
        f.write("struct FixPiece {\n    uint64_t b[5];\n    uint32_t b5, b6;\n};\n\n")
        f.write("__device__ const uint64_t kFixExp2[256] = {\n")
        for j in range(256):
            f.write(f"    0x{units(mp.mpf(2) ** (mp.mpf(j) / 256), 63):016x}ULL,\n")
        f.write("};\n\nalignas(16) __device__ const FixPiece kFixErfcx[kFixPieces] = {\n")
        for b in rows:
            f.write("    {{" + ", ".join(f"0x{v:x}ULL" for v in b[:5]) + f"}}, 0x{b[5]:x}u, 0x{b[6]:x}u}},\n")
        f.write("};\n\n}  // namespace lskum\n")


if __name__ == "__main__":
    main()
