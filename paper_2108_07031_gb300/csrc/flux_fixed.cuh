// Split-flux differences of the neighbour pairs whose step is too large for
// flux_pair.cuh, where G(q~_j) - G(q~_0) is the difference of two full
// evaluations: 1/sqrt(beta), exponentials, erfc and the moments in 64-bit fixed
// point, FP64 for the residual of 1/beta and the products of the rounded
// factors. An FP64 instruction costs 64 issue slots of the other pipes on this
// GPU, a 64 x 64 bit product about ten.
//
// With beta = -q4/2, i = 1/sqrt(beta), S = (q2, q3) i / 2, N = |S|^2, Phi(s) =
// erfc(-s)/2, T(s) = s Phi(s) + e^(-s^2) / (2 sqrt(pi)), P(s) = s T + Phi/2,
// C(s) = (3/2 + N/2) T + s Phi/4 and E = exp(q1 + N), the flux of the molecules
// with positive a-velocity is (m0 T, m1 P, m1 S_b T, m3 C) at s = S_a, m0 = E i^6,
// m1 = E i^7, m3 = E i^8; that of the negative ones (-, +, -, -) at s = -S_a.
//
// Compiled by a host compiler, the same code runs on the CPU (the tests do).
#pragma once

#include "pair_convert.cuh"

#ifndef __CUDACC__
#define __device__
#endif
#include "fixed_tables.h"

namespace lskum {

LSKUM_HD uint64_t mulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return uint64_t((unsigned __int128)a * b >> 64);
#endif
}
LSKUM_HD double dfma(double a, double b, double c) {
#ifdef __CUDA_ARCH__
    return __fma_rn(a, b, c);
#else
    return std::fma(a, b, c);
#endif
}

// |x| of the given bits in units of 2^-frac, truncated; |x| < 2^(64 - frac).
LSKUM_HD uint64_t to_fixed(uint64_t bits, int frac) {
    const uint64_t m = (bits & 0x000fffffffffffffULL) | 0x0010000000000000ULL;
    const int sh = int(bits >> 52 & 0x7ff) - 1075 + frac;
    return sh >= 0 ? m << sh : (sh > -64 ? m >> -sh : 0);
}

// v 2^e rounded to nearest, v > 0 (0 gives 0), the result normal.
LSKUM_HD double to_double(uint64_t v, int e) {
#ifdef __CUDA_ARCH__
    const int z = __clzll(int64_t(v));
#else
    const int z = v ? __builtin_clzll(v) : 64;
#endif
    if (v == 0) return 0.0;
    v <<= z;
    return dvalue((uint64_t(1085 + e - z) << 52) + (v >> 11) + (v >> 10 & 1));
}

// 2^(frac 2^-64) in units of 2^-63, truncated: by table for the leading 8 bits
// and the exponential series of degree 5 for the others; within 2^-59.
LSKUM_HD uint64_t exp2_fixed(uint64_t frac) {
    const uint64_t t = kFixExp2[frac >> 56], h = frac << 8;
    const uint64_t h32 = h >> 32;
    const uint64_t c4 = kFixE4 + (kFixE5 * h32 >> 34);                // 2^-70
    const uint64_t c3 = kFixE3 + (uint64_t(uint32_t(c4)) * h32 >> 30);  // 2^-72 from here on
    const uint64_t c2 = kFixE2 + (uint64_t(uint32_t(c3 >> 12)) * h32 >> 20);
    const uint64_t c1 = kFixE1 + mulhi(c2, h);
    return t + (mulhi(t, mulhi(c1, h)) >> 8);
}

LSKUM_HD int64_t smulhi(int64_t a, int64_t b) {
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return int64_t((__int128)a * b >> 64);
#endif
}

// v (1 + x 2^-64) for v < 2^63 and a small x of either sign.
LSKUM_HD uint64_t grow(uint64_t v, int64_t x) {
    const uint64_t c = mulhi(v, uint64_t(x < 0 ? -x : x));
    return x < 0 ? v - c : v + c;
}

constexpr int64_t kFixSEnd = (int64_t(6) << 60) - (int64_t(1) << 54);  // |S| < 6 - 1/64, units of 2^-60

struct FixedState {
    int64_t S[2];        // units of 2^-60
    double m0, m3;
    uint64_t m1;         // m1 = m1 2^e1
    int e1;
    uint64_t c32;        // 3/2 + N/2, units of 2^-58
};

// |q| i / 2 in units of 2^-60; 2^63 - 1 when it is 8 and more.
LSKUM_HD int64_t fixed_S(const double q, uint64_t y64, int ye, int64_t d1) {
    const uint64_t b = dword(q);
    const uint64_t m = (b << 11) | (uint64_t(1) << 63);
    const uint64_t v = grow(mulhi(m, y64) >> 1, d1);
    // v 2^(exponent - 1086 + ye - 40 + 64 + 1 - 1)
    const int sh = 1002 - int(b >> 52 & 0x7ff) - ye;
    const int64_t a = sh < 0 ? 0x7fffffffffffffffLL : (sh > 63 ? 0 : int64_t(v >> sh));
    return b >> 63 ? -a : a;
}

// False for a state out of range: |S| of 6 and more (the table's end), a q1
// over 24 or an extreme beta; the caller takes the general evaluation.
LSKUM_HD bool fixed_state(const double q[4], FixedState& w) {
    const uint64_t b4 = dword(q[3]), b0 = dword(q[0]);
    // q4 < 0, 2^-60 <= |q4| < 2^60
    if (b4 - 0xbc30000000000000ULL >= 0x0780000000000000ULL) return false;
    if ((b0 & 0x7fffffffffffffffULL) >= 0x4038000000000000ULL) return false;
    const double nbeta = dvalue(b4 - 0x0010000000000000ULL);  // q4/2 = -beta
    // y a float estimate of i, e = 1 - beta y^2 (y^2 is exact, e rounded once):
    // i^k = y^k (1 + (k/2) e + (k (k + 2) / 8) e^2)
    const float bf = narrow(-nbeta);
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(bf));
#else
    const float y = 1.0f / std::sqrt(bf);
#endif
    const double yd = widen(y), ed = dfma(nbeta, yd * yd, 1.0);
    const uint64_t eb = dword(ed);
    const int64_t ea = int64_t(to_fixed(eb, 64)), e = eb >> 63 ? -ea : ea;  // 2^-64
    const int64_t e2 = int64_t(uint64_t((ea >> 20) * (ea >> 20)) >> 24);
    const uint32_t ym = (fbits(y) & 0x007fffffu) | 0x00800000u;
    const int ye = int(fbits(y) >> 23) - 150;  // y = ym 2^ye
    const uint64_t y64 = uint64_t(ym) << 40;
    uint64_t s64 = uint64_t(ym) * ym << 16;  // y^2 = s64 2^se
    int se = 2 * ye - 16;
    if (!(s64 >> 63)) {
        s64 <<= 1;
        --se;
    }
    const int64_t d1 = (e >> 1) + (3 * e2 >> 3);
    w.S[0] = fixed_S(q[1], y64, ye, d1);
    w.S[1] = fixed_S(q[2], y64, ye, d1);
    const uint64_t ax = uint64_t(w.S[0] < 0 ? -w.S[0] : w.S[0]), ay = uint64_t(w.S[1] < 0 ? -w.S[1] : w.S[1]);
    if (ax >= uint64_t(kFixSEnd) || ay >= uint64_t(kFixSEnd)) return false;
    const uint64_t n56 = (mulhi(ax << 1, ax << 1) >> 2) + (mulhi(ay << 1, ay << 1) >> 2);  // N, 2^-56
    if (n56 >= uint64_t(35) << 56) return false;
    w.c32 = (n56 << 1) + (uint64_t(3) << 57);
    const int64_t q57 = int64_t(to_fixed(b0, 57));
    const int64_t x = (b0 >> 63 ? -q57 : q57) + int64_t(n56 << 1);
    const int64_t l = int64_t(mulhi(uint64_t(x < 0 ? -x : x), kFixLog2e));  // 2^-56
    const int64_t z = x < 0 ? -l : l;
    const uint64_t E = exp2_fixed(uint64_t(z) << 8);  // E = E 2^(z 2^-56 rounded down, - 63)
    const uint64_t a6 = mulhi(mulhi(mulhi(s64, s64), s64), E) >> 1;
    const int x6 = 3 * se + int(z >> 56) + 130;
    w.m0 = to_double(grow(a6, 3 * e + 6 * e2), x6);
    w.m1 = grow(mulhi(a6, y64), 3 * e + (e >> 1) + (63 * e2 >> 3));
    w.e1 = x6 + ye + 24;
    w.m3 = to_double(grow(mulhi(a6, s64), 4 * e + 10 * e2), x6 + se + 64);
    return true;
}

// T, P and C at s (units of 2^-60), |s| < 6. At -|s|, where all three are small,
// in units scaled by the power of two of e^(-s^2); above zero by T(s) = s +
// T(-s), P(s) = s^2 + 1/2 - P(-s), C(s) = (7/4 + N/2) s + C(-s). Absolute errors
// of some 2^-57 next to values of 0.25 and more.
LSKUM_HD void fixed_moments(const int64_t s, const FixedState& w, double& T, double& P, double& C) {
    const uint64_t a = uint64_t(s < 0 ? -s : s) << 1;  // |s|, 2^-61
    const uint64_t s2 = mulhi(a, a);                   // 2^-58
    const int64_t z = -int64_t(mulhi(s2, kFixLog2e));  // -s^2 log2(e), 2^-57
    const int n = int(z >> 57);
    const uint64_t m = exp2_fixed(uint64_t(z) << 7);   // e^(-s^2) = 2^n m, m in 2^-63
    const FixPiece* c = kFixErfcx + int(a >> 55);
    const uint64_t h = a << 9;
    const uint32_t h32 = uint32_t(h >> 32);
    uint64_t r = c->b5 - uint32_t(uint64_t(c->b6) * h32 >> 32);
    r = c->b[4] - (r * h32 >> 32);
    r = c->b[3] - mulhi(r, h);
    r = c->b[2] - mulhi(r, h);
    r = c->b[1] - mulhi(r, h);
    r = c->b[0] - mulhi(r, h);            // erfcx(|s|), 2^-63
    const uint64_t H = mulhi(m, r);       // Phi(-|s|), 2^(n-63)
    const uint64_t aH = mulhi(a, H);      // 2^(n-60)
    uint64_t t = (mulhi(m, kFixHalfIsqPi) >> 3) - aH;  // T(-|s|), 2^(n-60)
    uint64_t p = (H >> 4) - mulhi(a, t << 3);          // P(-|s|), 2^(n-60)
    uint64_t v = mulhi(w.c32, t << 3) - (aH >> 5);     // C(-|s|), 2^(n-57)
    int et = n - 60, ep = n - 60, ev = n - 57;
    if (s >= 0) {
        t = (a >> 1) + (t >> -n);
        p = (s2 >> 1) + (uint64_t(1) << 56) - (p >> (3 - n));
        v = mulhi((w.c32 << 1) + (uint64_t(1) << 57), a) + (v >> (1 - n));
        et = -60;
        ep = -57;
        ev = -56;
    }
    T = to_double(t, et);
    P = to_double(p, ep);
    C = to_double(v, ev);
}

// d = G - d for the flux G of the state along the first axis of S, in the order mass,
// momentum along the axis, momentum across, energy, up to the sign of the first
// and the last on the negative side. A second state's d is the difference, each
// component one fused multiply-add on the first one's rounded value.
LSKUM_HD void fixed_flux(const FixedState& w, bool negative, double d[4]) {
    double T, P, C;
    fixed_moments(negative ? -w.S[0] : w.S[0], w, T, P, C);
    const int64_t b = negative ? -w.S[1] : w.S[1];
    const double mb = to_double(mulhi(w.m1, uint64_t(b < 0 ? -b : b) << 1), w.e1 + 3);
    d[0] = dfma(w.m0, T, -d[0]);
    d[1] = dfma(to_double(w.m1, w.e1), P, -d[1]);
    d[2] = dfma(b < 0 ? -mb : mb, T, -d[2]);
    d[3] = dfma(w.m3, C, -d[3]);
}

// The state's S turned into the frame of a unit normal (nx, ny): s = (ny, -nx).
// False when a component leaves the table's range.
LSKUM_HD bool fixed_turn(FixedState& w, double nx, double ny) {
    const uint64_t bx = dword(nx), by = dword(ny), mag = 0x7fffffffffffffffULL;
    if ((bx & mag) > 0x3ff8000000000000ULL || (by & mag) > 0x3ff8000000000000ULL) return false;
    const int64_t ax = int64_t(to_fixed(bx, 62)), ay = int64_t(to_fixed(by, 62));
    const int64_t x = bx >> 63 ? -ax : ax, y = by >> 63 ? -ay : ay;
    const int64_t s = (smulhi(w.S[0], y) - smulhi(w.S[1], x)) * 4, n = (smulhi(w.S[0], x) + smulhi(w.S[1], y)) * 4;
    w.S[0] = s;
    w.S[1] = n;
    return s < kFixSEnd && -s < kFixSEnd && n < kFixSEnd && -n < kFixSEnd;
}

// G(q~_j) - G(q~_0) along both axes of the frame of (nx, ny), or of x and y when
// not local; false when a state is out of range. One state after the other in a
// loop: the code fits the instruction cache next to the pair form's.
LSKUM_HD bool fixed_diff(const double tj[4], const double t0[4], bool local, double nx, double ny,
                         bool negative_s, bool negative_n, double ds[4], double dn[4]) {
    bool ok = true;
    for (int m = 0; m < 4; ++m) ds[m] = dn[m] = 0.0;
#ifdef __CUDACC__
#pragma unroll 1
#endif
    for (int j = 0; j < 2; ++j) {
        const double q[4] = {j ? tj[0] : t0[0], j ? tj[1] : t0[1], j ? tj[2] : t0[2], j ? tj[3] : t0[3]};
        FixedState w;
        if (!fixed_state(q, w) || (local && !fixed_turn(w, nx, ny))) {
            ok = false;
            break;
        }
#ifdef __CUDACC__
#pragma unroll 1
#endif
        for (int k = 0; k < 2; ++k) {  // the axis just done last in ds, so twice round restores them
            fixed_flux(w, k ? negative_n : negative_s, ds);
#ifdef __CUDACC__
#pragma unroll
#endif
            for (int m = 0; m < 4; ++m) {
                const double t = ds[m];
                ds[m] = dn[m];
                dn[m] = t;
            }
            const int64_t t = w.S[0];
            w.S[0] = w.S[1];
            w.S[1] = t;
        }
    }
    if (negative_s) {
        ds[0] = -ds[0];
        ds[3] = -ds[3];
    }
    if (negative_n) {
        dn[0] = -dn[0];
        dn[3] = -dn[3];
    }
    return ok;
}

}  // namespace lskum
