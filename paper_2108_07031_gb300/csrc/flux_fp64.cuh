// FP64 device functions of the flux kernels: q~ -> primitive state, the kinetic
// split fluxes and their differences, the SSP-RK stage epilogue.
#pragma once

#include <cmath>

#include "device_math.cuh"
#include "lskum_internal.h"
#include "math_tables.h"
#include "lskum_kernels.cuh"

namespace lskum {

namespace {

constexpr double kInvSqrtPi = 0.56418958354775628695;  // 1 / sqrt(pi)

__device__ __forceinline__ V4 ld4(const V4* p) { return *p; }

// Bit-pattern helpers: comparisons and sign flips of doubles done on the
// integer pipe, which leaves the FP64 pipe (the flux kernel's bound) alone.
constexpr int64_t kSignBit = int64_t(0x8000000000000000ULL);
constexpr int64_t kAbsMask = 0x7FFFFFFFFFFFFFFFLL;
constexpr int64_t kBits700 = 0x4085E00000000000LL;  // 700.0
constexpr int64_t kBits6 = 0x4018000000000000LL;    // 6.0, the end of the erfcx table
static_assert(kErfcxLo == 0.0 && kErfcxInvW == double(1 << kErfcxLog2InvW) && kErfcxHi == 6.0,
              "erfcx_piece assumes pieces of width 2^-kErfcxLog2InvW on [0, 6]");

__device__ __forceinline__ int64_t dbits(const double x) { return __double_as_longlong(x); }
__device__ __forceinline__ double bitsd(const int64_t b) { return __longlong_as_double(b); }

// Primitive state of one modified state q~ in the flux's frame, with the
// per-state factors the split fluxes share: sqrt(beta), 1/sqrt(pi beta),
// h = p + rho e and mhp = -p/2 (|u|^2 is frame-invariant, so these are too).
struct Prim {
    double r, u, v, p, sb, cb, h, mhp;
};

// exp(x) 2^-HALVE by Tang's table-driven method (math_tables.h): x = k ln2/N
// + r (N = 2^kExpBits = 256), |r| <= ln2/(2N), exp(x) = 2^(k div N)
// 2^((k mod N)/N) e^r with e^r - 1 from its degree-4 Taylor polynomial
// (remainder < 4e-17); max error 1.2 ulp (checked against 200-bit arithmetic
// with exact FMA emulation). About 9 FP64 operations against the library's
// ~18; the power of two, including the optional halving, is an integer add
// to the exponent field (the result stays normal for |x| <= 700). Outside
// that range the library exp.
template <int HALVE>
__device__ __forceinline__ double exp_tab(const double x) {
    if ((dbits(x) & kAbsMask) > kBits700) return HALVE ? 0.5 * exp(x) : exp(x);
    const double shifter = 6755399441055744.0;  // 1.5 * 2^52: rounds k into the low bits
    double kd = fma(x, kInvLn2ByN, shifter);
    const int64_t k = dbits(kd) - 0x4338000000000000LL;
    kd -= shifter;
    const double r = fma(-kd, kLn2ByNLo, fma(-kd, kLn2ByNHi, x));
    const double p = r * fma(r, fma(r, fma(r, 1.0 / 24.0, 1.0 / 6.0), 0.5), 1.0);
    const double t = kExp2Tab[k & ((1 << kExpBits) - 1)];
    const double res = fma(t, p, t);
    return bitsd(dbits(res) + (((k >> kExpBits) - HALVE) << 52));
}

// q~ -> primitive (inverse of Eq. 26); velocities in the global frame. With
// gamma = 1.4 (1/(gamma-1) = 5/2) the factor beta^(-1/(gamma-1)) of the
// density is (1/beta)^2 / sqrt(beta), so no logarithm is needed; 1/sqrt(beta)
// is needed by the split fluxes anyway.
template <bool G14>
__device__ __forceinline__ Prim q_to_prim(const double t0, const double t1, const double t2,
                                          const double t3, const double gm1_inv) {
    Prim w;
    const double beta = -0.5 * t3;
    const double isb = rsqrt(beta);
    w.sb = beta * isb;
    w.cb = isb * kInvSqrtPi;
    // 1/beta from (1/sqrt(beta))^2 and one Newton step, i2 (1 + (1 - beta
    // i2)): the residual 1 - beta i2 comes exact from the FMA, so the step
    // leaves ~0.5 ulp, as good as an IEEE division (u, v, p and the density's
    // (1/beta)^2 inherit it) for 4 FP64 instructions instead of ~7.
    const double i20 = isb * isb;
    const double i2 = fma(i20, fma(-beta, i20, 1.0), i20);  // 1 / beta
    const double inv2b = 0.5 * i2;                         // 1 / (2 beta)
    w.u = t1 * inv2b;
    w.v = t2 * inv2b;
    const double uu = fma(w.u, w.u, w.v * w.v);
    if (G14) {
        w.r = exp_tab<0>(fma(beta, uu, t0)) * (i2 * i2 * isb);
    } else {
        w.r = exp_tab<0>(t0 - log(beta) * gm1_inv + beta * uu);
    }
    w.p = w.r * inv2b;
    const double rhoe = fma(0.5 * w.r, uu, w.p * gm1_inv);
    w.h = w.p + rhoe;
    w.mhp = -0.5 * w.p;
    return w;
}

// Index of the erfcx piece holding a (0 <= a <= 6), floor(2^L a) with
// L = kErfcxLog2InvW, from the bit pattern of a = 1.f x 2^e:
// 2^L a = (2^52 + f) / 2^(52 - L - e).
__device__ __forceinline__ int erfcx_piece(const int64_t abits) {
    const int sh = (52 - kErfcxLog2InvW) - (int(abits >> 52) - 1023);
    const int64_t m = (abits & 0x000FFFFFFFFFFFFFLL) | 0x0010000000000000LL;
    const int k = sh > 52 ? 0 : int(m >> sh);
    return min(k, kErfcxPieces - 1);
}

// Kinetic split flux along the frame's first axis ("a" = ua, "b" = ub) of
// the state w, for molecules with positive (nmask = 0) or negative (nmask =
// sign bit) a-velocity. With S = ua sqrt(beta) and sg = +-1:
//   A = erfc(-sg S)/2, B = exp(-S^2)/(2 sqrt(pi beta)),
//   G = (rho (ua A + sg B), (p + rho ua^2) A + sg rho ua B, rho ub (ua A + sg B),
//        (p + rho e) ua A + sg (rho e + p/2) B).
// erfc(|S|)/2 = exp(-S^2)/2 erfcx(|S|) from the erfcx pieces for |S| <= 6, from one
// polynomial in 1/S^2 beyond, sharing exp(-S^2)/2 with B, so that ua A + sg B, a
// 72nd and less of either there, loses nothing to two roundings of it (the
// library's erfc took some 65 FP64 instructions, the polynomial 25: Mach 8 at 0.6M
// points 5.9 -> 4.5 ms a launch).
// With t = ua A + sg B the four components are G0 = rho t, G1 = ua G0 + p A,
// G2 = ub G0 and G3 = h t - (p/2) sg B (h - p/2 = rho e + p/2); split_ab
// returns t, A and sg B of one state, split_flux_diff the four differences
// between two states.
struct SplitAB {
    double t, A, Bs;
};

__device__ __forceinline__ SplitAB split_ab(const Prim& w, const double ua, const int64_t nmask) {
    const double S = ua * w.sb;
    const double eh = exp_tab<1>(-(S * S));  // exp(-S^2) / 2
    const int64_t abits = dbits(S) & kAbsMask;
    double hc;  // erfc(|S|) / 2
    if (abits <= kBits6) {
        const double* c = kErfcxC[erfcx_piece(abits)];
        const double z = bitsd(abits) - __ldg(c);
        double pv = __ldg(c + 1 + kErfcxDeg);
#pragma unroll
        for (int m = kErfcxDeg - 1; m >= 0; --m) pv = fma(pv, z, __ldg(c + 1 + m));
        hc = eh * pv;
    } else {
        const double r = 1.0 / bitsd(abits), w = r * r;
        double pv = __ldg(kErfcxTail + kErfcxTailDeg);
#pragma unroll
        for (int m = kErfcxTailDeg - 1; m >= 0; --m) pv = fma(pv, w, __ldg(kErfcxTail + m));
        hc = eh * (r * pv);
    }
    // A = erfc(x)/2 at x = -sg S: erfc(|x|)/2 for x > 0, 1 - erfc(|x|)/2 otherwise
    const int64_t xbits = dbits(S) ^ nmask ^ kSignBit;
    const double A = xbits > 0 ? hc : 1.0 - hc;
    const double Bs = bitsd(dbits(eh * w.cb) ^ nmask);  // sg B
    return SplitAB{fma(ua, A, Bs), A, Bs};
}

// G(state j) - G(state 0) along the frame's first axis (velocities uaj, ubj
// and ua0, ub0): each difference takes state 0's value, rounded once, into
// the FMA chain of state j's, so the four cost 13 FP64 operations where two
// flux evaluations and four subtractions took 16.
__device__ __forceinline__ void split_flux_diff(const Prim& wj, const Prim& w0, const double uaj,
                                                const double ubj, const double ua0, const double ub0,
                                                const SplitAB& aj, const SplitAB& a0, double d[4]) {
    const double g0j = wj.r * aj.t, g00 = w0.r * a0.t;
    d[0] = g0j - g00;
    const double g10 = fma(ua0, g00, w0.p * a0.A);
    d[1] = fma(uaj, g0j, fma(wj.p, aj.A, -g10));
    d[2] = fma(g0j, ubj, -(g00 * ub0));
    const double g30 = fma(w0.h, a0.t, w0.mhp * a0.Bs);
    d[3] = fma(wj.h, aj.t, fma(wj.mhp, aj.Bs, -g30));
}

// Modified states q~_j and q~_0 of Eq. 28 for one neighbour (half offsets
// hx, hy); returns false when they are bitwise equal: then every split-flux
// difference is exactly 0 (free-stream preservation), and the pair is skipped.
__device__ __forceinline__ bool modified_states(const bool second, const double hx, const double hy,
                                                const V8& dj, const V8& di, double tj[4],
                                                double t0[4]) {
    if (second) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            tj[m] = fma(-hx, dj.x[m], fma(-hy, dj.y[m], tj[m]));
            t0[m] = fma(-hx, di.x[m], fma(-hy, di.y[m], t0[m]));
        }
    }
    int64_t diff = 0;
#pragma unroll
    for (int m = 0; m < 4; ++m) diff |= dbits(tj[m]) ^ dbits(t0[m]);
    return diff != 0;
}

// Eq. 26 from the primitive state (rho, u, v, p).
__device__ __forceinline__ void prim_to_q(const double rho, const double u, const double v,
                                          const double p, const Physics& ph, V4& q) {
    const double beta = rho / (2.0 * p);
    q.a = log(rho) + log(beta) * ph.gm1_inv - beta * (u * u + v * v);
    q.b = 2.0 * beta * u;
    q.c = 2.0 * beta * v;
    q.d = -2.0 * beta;
}

__device__ __forceinline__ bool physical(double rho, double u, double v, double p) {
    return rho > 0.0 && p > 0.0 && isfinite(rho) && isfinite(p) && isfinite(u) && isfinite(v);
}

// Block-wide sum in a fixed order (warp shuffles, then the warps' partials
// by the first warp), so the result does not depend on timing.
template <int BLOCK>
__device__ __forceinline__ double block_sum(double x) {
    __shared__ double warp_part[BLOCK / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) warp_part[wid] = x;
    __syncthreads();
    double s = 0.0;
    if (wid == 0) {
        s = lane < BLOCK / 32 ? warp_part[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    }
    return s;  // valid in thread 0
}

// SSP-RK stage epilogue of one (point, condition), shared by the fused flux
// kernel and the split-flux ablation: mode 0 stores R; modes 1..4 apply the
// stage update, the wall condition and the next q; stage 1 also stores dt
// and U0 and returns R_rho^2 for the residue.
template <int MODE, bool G14>
__device__ __forceinline__ double stage_epilogue(const DevGeom& g, const Physics& ph,
                                                 const DevState& st, const int64_t t,
                                                 const int64_t d, const int8_t fl, const bool fixed,
                                                 const double R[4], V4* __restrict__ q_out) {
    double r2 = 0.0;
    if (MODE == 0) {
        st.R[t] = V4{R[0], R[1], R[2], R[3]};
    } else {
        V4 U = ld4(st.U + t);
        double dtv;
        if (MODE == 1) {
            const double rho = U.a, u = U.b / rho, v = U.c / rho;
            const double p = ph.gm1 * (U.d - 0.5 * rho * (u * u + v * v));
            dtv = ph.cfl * g.dmin[d] / (sqrt(u * u + v * v) + sqrt(ph.gamma * p / rho));
            st.dt[t] = dtv;
            st.U0[t] = U;
            r2 = R[0] * R[0];
        } else {
            dtv = st.dt[t];
        }
        if (!fixed) {
            const double h = 0.5 * dtv;
            if (MODE == 3) {
                const V4 U0 = ld4(st.U0 + t);
                U.a = (2.0 / 3.0) * U0.a + (1.0 / 3.0) * (U.a - h * R[0]);
                U.b = (2.0 / 3.0) * U0.b + (1.0 / 3.0) * (U.b - h * R[1]);
                U.c = (2.0 / 3.0) * U0.c + (1.0 / 3.0) * (U.c - h * R[2]);
                U.d = (2.0 / 3.0) * U0.d + (1.0 / 3.0) * (U.d - h * R[3]);
            } else {
                U.a -= h * R[0];
                U.b -= h * R[1];
                U.c -= h * R[2];
                U.d -= h * R[3];
            }
            if (fl == LSKUM_WALL) {  // remove the wall-normal momentum
                const double2 nn = g.nrm[d];
                const double tx = nn.y, ty = -nn.x;
                const double ms = U.b * tx + U.c * ty;
                U.b = ms * tx;
                U.c = ms * ty;
            }
            st.U[t] = U;
        }
        V4 qn;
        double rho, u, v, p;
        cons_to_q64<G14>(U, ph, qn, rho, u, v, p);
        q_out[t] = qn;
        if (!physical(rho, u, v, p)) atomicOr(st.status, 1);
    }

    return r2;
}

}  // namespace

}  // namespace lskum
