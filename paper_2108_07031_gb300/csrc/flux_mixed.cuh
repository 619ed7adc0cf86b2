// Split-flux differences of a neighbour pair in floats, for the mixed mode: the
// primitive form (any gamma, any step) and the form in S = u sqrt(beta) (gamma =
// 1.4, steps of S up to 1/4). Both take q~_0 and q~_j - q~_0 and subtract no two
// nearby values.
//
// Compiled by a host compiler, the same code runs on the CPU with rounded results
// in place of the hardware's approximations (the tests do).
#pragma once

#include "pair_math.cuh"
#ifndef __CUDACC__
#define __device__
#endif
#include "math_tables.h"

namespace lskum {

#ifdef __CUDACC__
using Float4 = float4;
__device__ __forceinline__ float rsqrt_f(float x) { return rsqrtf(x); }
__device__ __forceinline__ float div_f(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ float exp_f(float x) { return __expf(x); }
__device__ __forceinline__ float log_f(float x) { return __logf(x); }
__device__ __forceinline__ float ldg_f(const float* p) { return __ldg(p); }
#else
struct Float4 {
    float x, y, z, w;
};
inline float rsqrt_f(float x) { return float(1.0 / std::sqrt(double(x))); }
inline float div_f(float a, float b) { return a / b; }
inline float exp_f(float x) { return float(std::exp(double(x))); }
inline float log_f(float x) { return float(std::log(double(x))); }
inline float ldg_f(const float* p) { return *p; }
#endif

constexpr float kInvSqrtPiF = 0.56418958354775628695f;  // 1 / sqrt(pi)

// ------------------------------------------------ primitive base + difference

struct PrimPair {
    float r, u, v, p, sb;       // base state (of q~_0): density, velocity, pressure, sqrt(beta)
    float dr, du, dv, dp, dsb;  // difference state(q~_j) - state(q~_0)
    float isb, isbj;            // 1/sqrt(beta) of the base and of state j
    // frame-invariant factor both split fluxes of the pair share (base and
    // difference): h = p + rho e
    float h, dh;
};

// e^x - 1: its Taylor polynomial to x^5/120 for |x| <= 1/16 (the remainder is
// below 2e-9 of the result), the library function beyond. The arguments
// here are differences of nearby states, almost always far inside 1/16.
LSKUM_HD float expm1_f(const float x) {
    if (fabsf(x) <= 0.0625f)
        return x * fmaf(x, fmaf(x, fmaf(x, fmaf(x, 1.0f / 120.0f, 1.0f / 24.0f), 1.0f / 6.0f), 0.5f),
                        1.0f);
    return expm1f(x);
}

// ln(1 + x): its Taylor polynomial to x^6/6 for |x| <= 1/16 (remainder below
// 1e-8 of the result), the library function beyond.
LSKUM_HD float log1p_f(const float x) {
    if (fabsf(x) <= 0.0625f)
        return x * fmaf(x, fmaf(x, fmaf(x, fmaf(x, fmaf(x, -1.0f / 6.0f, 0.2f), -0.25f), 1.0f / 3.0f),
                                -0.5f),
                        1.0f);
    return log1pf(x);
}

// The FP32 quotients below are fast (reciprocal approximation times the
// numerator, ~2 ulp): every one scales a difference term, whose own FP32
// rounding error is larger.

// From the base q~_0 and the difference dq~ = q~_j - q~_0 (inverse of Eq. 26).
template <bool G14>
LSKUM_HD PrimPair prim_pair(const Float4 b, const Float4 dq, const float gm1_inv) {
    PrimPair w;
    const float beta = -0.5f * b.w;
    const float dbeta = -0.5f * dq.w;
    const float qj4 = b.w + dq.w;
    const float inv2b = div_f(-1.0f, b.w);  // 1 / (2 beta)
    w.u = b.y * inv2b;
    w.v = b.z * inv2b;
    // u = -q2/q4:  u_j - u_0 = (q2 dq4 - dq2 q4) / (q4 q4_j)
    const float rq = div_f(1.0f, b.w * qj4);
    w.du = (b.y * dq.w - dq.y * b.w) * rq;
    w.dv = (b.z * dq.w - dq.z * b.w) * rq;
    const float uj = w.u + w.du, vj = w.v + w.dv;
    const float uu0 = w.u * w.u + w.v * w.v;
    const float uuj = uj * uj + vj * vj;
    const float duu = w.du * (uj + w.u) + w.dv * (vj + w.v);
    w.isb = rsqrt_f(beta);
    w.sb = beta * w.isb;
    const float betaj = beta + dbeta;
    w.isbj = rsqrt_f(betaj);
    // sqrt(beta_j) - sqrt(beta) = dbeta / (sqrt(beta_j) + sqrt(beta))
    w.dsb = div_f(dbeta, betaj * w.isbj + w.sb);
    // ln rho = q1 - ln(beta)/(gamma-1) + beta |u|^2
    if (G14) {
        const float i2 = w.isb * w.isb;
        w.r = exp_f(b.x + beta * uu0) * (i2 * i2 * w.isb);
    } else {
        w.r = exp_f(b.x - log_f(beta) * gm1_inv + beta * uu0);
    }
    const float dlnr = dq.x - log1p_f(dbeta * (2.0f * inv2b)) * gm1_inv + (dbeta * uuj + beta * duu);
    w.dr = w.r * expm1_f(dlnr);
    // p = rho / (2 beta):  p_j - p_0 = (drho beta - rho dbeta) / (2 beta beta_j)
    w.p = w.r * inv2b;
    w.dp = (w.dr * beta - w.r * dbeta) * (inv2b * (w.isbj * w.isbj));
    // rho e = p/(gamma-1) + rho |u|^2 / 2 (|u|^2 is the same in every frame)
    const float E0 = w.p * gm1_inv + 0.5f * w.r * uu0;
    const float dE = w.dp * gm1_inv + 0.5f * (w.dr * uuj + w.r * duu);
    w.h = w.p + E0;
    w.dh = w.dp + dE;
    return w;
}

// erfc(m - h) - erfc(m + h) = (4/sqrt(pi)) e^{-m^2} (h + H2 h^3/6 + H4 h^5/120
// + H6 h^7/5040 + H8 h^9/362880) with the Hermite polynomials H_k(m): the
// even Taylor terms of e^{-t^2} about m integrated over [m - h, m + h].
// For |h| <= 1/64 the H6 and H8 terms are below 2e-11 of the first (|m| <=
// 6.5, the range where erfc is not negligible) and are left out.
LSKUM_HD float erfc_central_diff(const float m, const float h) {
    const float m2 = m * m;
    const float H2 = 4.0f * m2 - 2.0f;
    const float H4 = (16.0f * m2 - 48.0f) * m2 + 12.0f;
    const float h2 = h * h;
    float tail = H4 * (1.0f / 120.0f);
    if (fabsf(h) > 0.015625f) {
        const float H6 = ((64.0f * m2 - 480.0f) * m2 + 720.0f) * m2 - 120.0f;
        const float H8 = (((256.0f * m2 - 3584.0f) * m2 + 13440.0f) * m2 - 13440.0f) * m2 + 1680.0f;
        tail += h2 * (H6 * (1.0f / 5040.0f) + h2 * (H8 * (1.0f / 362880.0f)));
    }
    const float s = h * (1.0f + h2 * (H2 * (1.0f / 6.0f) + h2 * tail));
    return 4.0f * kInvSqrtPiF * exp_f(-m2) * s;
}

// erfc(x)/2 given e = exp(-x^2): e erfcx(|x|)/2 from the FP32 erfcx pieces
// (width 1/4, degree 5, 1.2e-7 relative) for |x| < 6, then 1 minus it for
// x < 0; the exponential is the one the split flux needs for B anyway.
LSKUM_HD float half_erfc_f(const float x, const float e) {
    const float a = fabsf(x);
    float hc;
    if (a < 6.0f) {
        const float* c = kErfcxF[int(a * kErfcxFInvW)];
        const float z = a - ldg_f(c);
        float pv = ldg_f(c + 1 + kErfcxFDeg);
#pragma unroll
        for (int m = kErfcxFDeg - 1; m >= 0; --m) pv = fmaf(pv, z, ldg_f(c + 1 + m));
        hc = 0.5f * e * pv;
    } else {
        hc = 0.5f * erfcf(a);
    }
    return x > 0.0f ? hc : 1.0f - hc;
}

// Difference of the kinetic split flux along the frame's first axis ("a",
// velocity ua, transverse ub), sign sg: dG = G(state_j) - G(state_0),
// state_j = base + difference; the frame-invariant factors come from w.
LSKUM_HD void dsplit_flux_a(const PrimPair& w, const float ua0, const float ub0,
                                              const float dua, const float dub, const float sg,
                                              float dG[4]) {
    const float r0 = w.r, dr = w.dr, p0 = w.p, dp = w.dp, sb0 = w.sb, dsb = w.dsb;
    const float isb0 = w.isb, isbj = w.isbj;
    const float sbj = sb0 + dsb;
    const float S0 = ua0 * sb0;
    const float dS = dua * sbj + ua0 * dsb;
    const float Sj = S0 + dS;
    // exponential: e_j - e_0 = e_0 expm1(-(S_j^2 - S_0^2))
    const float e0 = exp_f(-S0 * S0);
    const float de = e0 * expm1_f(-dS * (Sj + S0));
    // A = erfc(x)/2 at x = -sg S
    const float x0 = -sg * S0, dx = -sg * dS;
    const float A0 = half_erfc_f(x0, e0);  // e0 = exp(-x0^2)
    float dA;
    if (fabsf(dx) <= 0.25f) {
        // erfc(x0 + dx) - erfc(x0) = -(erfc(m - h) - erfc(m + h)), m = x0 + dx/2, h = dx/2
        dA = -0.5f * erfc_central_diff(x0 + 0.5f * dx, 0.5f * dx);
    } else {
        dA = 0.5f * (erfcf(x0 + dx) - erfcf(x0));
    }
    const float Aj = A0 + dA;
    // B = e / (2 sqrt(pi) sqrt(beta))
    const float c = 0.5f * kInvSqrtPiF;
    const float B0 = c * e0 * isb0;
    const float dB = c * (de * isbj - e0 * dsb * isbj * isb0);
    const float Bj = B0 + dB;
    // t = u_a A + sg B
    const float t0 = ua0 * A0 + sg * B0;
    const float dt = dua * Aj + ua0 * dA + sg * dB;
    const float tj = t0 + dt;
    // mass: G0 = rho t
    const float G00 = r0 * t0;
    dG[0] = dr * tj + r0 * dt;
    const float G0j = G00 + dG[0];
    // a-momentum: (p + rho u_a^2) A + sg rho u_a B = u_a G0 + p A
    dG[1] = dua * G0j + ua0 * dG[0] + (dp * Aj + p0 * dA);
    // b-momentum: rho u_b t = u_b G0
    dG[2] = dub * G0j + ub0 * dG[0];
    // energy: (p + rho e) u_a A + sg (rho e + p/2) B = h t - (p/2) sg B
    dG[3] = w.dh * tj + w.h * dt - 0.5f * sg * (dp * Bj + p0 * dB);
}

// ---------------------------------------------------------------- the form in S

// Split-flux difference in floats as flux_pair.cuh has it in pairs (the same
// variables and product rules), for gamma = 1.4.
struct MxState {
    float Sxm, Sym, dSx, dSy, Km, dK, m0, m1, m3, dm0, dm1, dm3;
};

// e^x - 1 - x, to 2^-24 of x or so.
LSKUM_HD float expm1_less_x(const float x) {
    if (fabsf(x) <= 0.0625f)
        return x * x * fmaf(x, fmaf(x, fmaf(x, 1.0f / 120.0f, 1.0f / 24.0f), 1.0f / 6.0f), 0.5f);
    return expm1f(x) - x;
}

// From q~_0 = b and d = q~_j - b. False for a large step (the series in the step
// of S) or a state without a density: prim_pair takes those.
//
// The moments' relative steps are (1 + F)(1 + P) - 1 with F = e^W - 1 and P = (1 +
// eta)^-3 - 1, and W is about 5/2 eta: the linear terms are subtracted in one
// operation, eta with a low word, and the higher ones added to that. The
// moments hold i^6 to i^8, so 1/beta and 1/sqrt(beta) are refined to half a unit in
// the last place. 2-norm of dG's error at Mach 0.63, steps of 2^-8: 1.8e-7 to 2.1e-7,
// by the primitive differences 2.6e-7 to 2.9e-7, without the two measures 4.4e-7 to
// 6.4e-7; of the residual's at 5,120 points 4.2e-7 to 5.6e-7, 4.5e-7 to 5.8e-7 and
// 5.5e-7 to 8.3e-7. The measures cost 2 % of the flux (0.6M points 142.4 -> 145.4 us).
LSKUM_HD bool mx_state(const Float4 b, const Float4 d, MxState& w) {
    const float beta = -0.5f * b.w, y = rsqrt_f(beta), z = y * y, rz = fmaf(-beta, z, 1.0f);
    const float i2 = fmaf(z, rz, z), i0 = fmaf(0.5f * y, fmaf(-beta, fmaf(y, y, -z), rz), y), ih = 0.5f * i0;
    const float t = -0.5f * d.w, eta = t * i2, a = 1.0f + eta;
    const float eta_lo = fmaf(t, fmaf(z, rz, z - i2), fmaf(t, i2, -eta));
    // e = (1 + eta)^(-1/2) - 1 and e + eta/2, with u = 1/(a + sqrt(a))
    const float sa = a * rsqrt_f(a), u = div_f(1.0f, a + sa);
    const float e2 = 0.5f * eta * eta * u * fmaf(sa, u, 1.0f), e = fmaf(-0.5f, eta, e2);
    const float Sx = b.y * ih, Sy = b.z * ih;
    w.dSx = ih * fmaf(e, b.y + d.y, d.y);
    w.dSy = ih * fmaf(e, b.z + d.z, d.z);
    w.Sxm = fmaf(0.5f, w.dSx, Sx);
    w.Sym = fmaf(0.5f, w.dSy, Sy);
    const float SS = fmaf(Sx, Sx, Sy * Sy);
    w.dK = fmaf(w.Sxm, w.dSx, w.Sym * w.dSy);
    w.Km = fmaf(0.5f, SS + w.dK, 1.5f);
    const float W = fmaf(2.0f, w.dK, d.x), F2 = expm1_less_x(W);
    const float P2 = fmaf(6.0f, e2, e * e * fmaf(e, fmaf(e, fmaf(e, e + 6.0f, 15.0f), 20.0f), 15.0f));  // P + 3 eta
    const float r0 = fmaf(-3.0f, eta, W) + (fmaf(-3.0f, eta_lo, F2 + P2) + (W + F2) * fmaf(-3.0f, eta, P2));
    const float r1 = fmaf(r0, e, r0 + e), r3 = fmaf(r1, e, r1 + e);
    const float m0 = exp_f(b.x + SS) * (i2 * i2 * i2), m1 = m0 * i0, m3 = m0 * i2;
    w.dm0 = m0 * r0;
    w.dm1 = m1 * r1;
    w.dm3 = m3 * r3;
    w.m0 = fmaf(0.5f, w.dm0, m0);
    w.m1 = fmaf(0.5f, w.dm1, m1);
    w.m3 = fmaf(0.5f, w.dm3, m3);
    return fmaxf(fabsf(w.dSx), fabsf(w.dSy)) <= 0.25f && a > 0.0f;
}

LSKUM_HD float d_prod(float xm, float dx, float ym, float dy) { return fmaf(xm, dy, ym * dx); }
LSKUM_HD float m_prod(float xm, float dx, float ym, float dy) {
    return fmaf(xm, ym, 0.25f * dx * dy);
}

// {mass, axis momentum, transverse momentum, energy} along the axis with S =
// (m, ds), transverse (bm, db), for positive molecules.
LSKUM_HD void mx_diff(const MxState& w, const float m, const float ds, const float bm,
                                        const float db, float dG[4]) {
    const float q = m * m, ex = exp_f(-q), phi = kInvSqrtPiF * ex;
    const float Phi = half_erfc_f(-m, ex);
    const float h = 0.5f * ds, t = h * h, v = phi * t;
    // Hermite polynomials of the midpoint; terms beyond t below 1e-7 for t < 2^-12
    const float k = fmaf(q, 1.0f / 3.0f, -0.5f), tk = t * k;  // H3 = 24 m k
    float cP = fmaf(t, fmaf(q, fmaf(q, 2.0f / 15.0f, -0.4f), 0.1f), fmaf(q, 2.0f / 3.0f, -1.0f / 3.0f));
    float cM = fmaf(tk, m, m), cT = m * fmaf(tk, 0.2f, 1.0f / 3.0f);
    float cU = fmaf(t, fmaf(q, 1.0f / 6.0f, -1.0f / 12.0f), 0.5f);
    if (t > 2.44140625e-4f) {
        const float t2 = t * t, H4 = fmaf(fmaf(16.0f, q, -48.0f), q, 12.0f);
        const float H5 = m * fmaf(fmaf(32.0f, q, -160.0f), q, 120.0f);
        const float H6 = fmaf(fmaf(fmaf(64.0f, q, -480.0f), q, 720.0f), q, -120.0f);
        cP = fmaf(t2, H6 * (1.0f / 5040.0f), cP);
        cM = fmaf(t2, H5 * (1.0f / 720.0f), cM);
        cT = fmaf(t2, H5 * (1.0f / 5040.0f), cT);
        cU = fmaf(t2, H4 * (1.0f / 720.0f), cU);
    }
    const float dPhi = ds * fmaf(v, cP, phi), Phim = fmaf(-v, cM, Phi);
    const float dT = ds * fmaf(-v, cT, Phi), Tm = fmaf(v, cU, fmaf(m, Phi, 0.5f * phi));
    dG[0] = d_prod(w.m0, w.dm0, Tm, dT);
    dG[1] = d_prod(w.m1, w.dm1, fmaf(0.5f, Phim, m_prod(m, ds, Tm, dT)), fmaf(0.5f, dPhi, d_prod(m, ds, Tm, dT)));
    dG[2] = d_prod(w.m1, w.dm1, m_prod(bm, db, Tm, dT), d_prod(bm, db, Tm, dT));
    dG[3] = d_prod(w.m3, w.dm3, fmaf(0.25f, m_prod(m, ds, Phim, dPhi), m_prod(w.Km, w.dK, Tm, dT)),
                   fmaf(0.25f, d_prod(m, ds, Phim, dPhi), d_prod(w.Km, w.dK, Tm, dT)));
}

}  // namespace lskum
