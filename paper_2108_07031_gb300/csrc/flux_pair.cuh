// The split-flux differences of one neighbour pair in float pairs.
//
// In the variables i = 1/sqrt(beta), S = u sqrt(beta) = q2 i/2 (q3 for the
// other axis) and E = exp(q1 + |S|^2) = rho beta^(5/2) (gamma = 1.4), with
//   Phi(S) = erfc(-S)/2,  phi(S) = exp(-S^2)/sqrt(pi) = Phi',
//   T(S) = S Phi + phi/2 (T' = Phi),
// the kinetic split flux along axis a for molecules with positive a-velocity is
//   G0 = m0 T,  Ga = m1 (S T + Phi/2),  Gb = m1 S_b T,
//   Ge = m3 ((3/2 + |S|^2/2) T + S Phi/4),   m_k = E i^(6, 7, 8);
// the other sign is the mirror image S -> -S with G0, Gb, Ge negated. So one
// state costs one reciprocal square root, one exponential and one table
// lookup per axis.
//
// Every quantity of state j minus state 0 is formed from the difference d =
// q~_j - q~_0 itself -- sums and products by D(XY) = mean(X) DY + mean(Y) DX,
// powers of i by series in the relative step of beta, E by expm1, Phi and T by
// their Taylor series about the midpoint of S, where the even derivatives
// cancel -- so dG carries an error of 2^-46 to 2^-45 of itself. A plain FP64
// evaluation subtracts two fluxes and is left with ~2^-51.5 / (relative step):
// the pair form is the more accurate one for steps up to about kPairStep (at
// 2^-6 of the primitive variables 0.9-1.6 times FP64's error, at 2^-7 0.4-0.8,
// at 2^-9 0.1-0.2; 4,000 random pairs each, Mach 0.3-0.85). Larger steps, and
// states outside a range of sizes that floats hold with room, are left to FP64.
#pragma once

#include "pair_math.cuh"
#ifndef __CUDACC__
#define __device__
#endif
#include "pair_tables.h"

namespace lskum {

// Largest step of beta (relative) and S; of ln(rho beta^(5/2)), which is several
// times the primitive variables' and enters dG only to first order. Measured
// against binary128, 2-norm of the residual's error over the FP64 kernel's: at
// 1/64 0.46-0.85 on perturbed states of 600 and 1,500 points (eight to twelve seeds),
// 0.2-0.9 on others up to 46,080, 0.65-1.05 on eight flows 100 to 1,000 iterations
// from the free stream (one component of one 1.18); at 1/40 up to 1.9 on the latter.
constexpr float kPairStep = 1.0f / 64.0f;
constexpr float kPairStepW = 4.0f * kPairStep;
constexpr float kPairMaxS = 5.9f;          // |S| inside the Phi table
constexpr float kPairMaxArg = 40.0f;       // |ln(rho beta^(5/2))|
constexpr Pf kThird = {0x1.555556p-2f, -0x1.555556p-27f};  // 1/3, 1/6, 1/24 as pairs
constexpr Pf kSixth = {0x1.555556p-3f, -0x1.555556p-28f};
constexpr Pf kTwentyFourth = {0x1.555556p-5f, -0x1.555556p-30f};
constexpr Pf k120th = {0x1.111112p-7f, -0x1.dddddep-32f};
constexpr float kPairMaxBeta = 16777216.0f, kPairMinBeta = 1.0f / 16777216.0f;

// 2^-60 <= x < 2^60: with the low words and the products' errors in range too
// (m1 lies between m0 and m3). False for NaN.
LSKUM_HD bool pair_held(float x) { return fbits(x) - 0x21800000u < 0x3c000000u; }

// exp(x) for |x| <= kPairMaxArg.
LSKUM_HD Pf exp_pair(Pf x) {
    const float kf = rsub(rfma(x.h, kPairInvLn2N, 12582912.0f), 12582912.0f);
    const int k = int(kf);
    Pf r = two_sum(rfma(-kf, kPairLn2N1, x.h), -rmul(kf, kPairLn2N2));
    const float e2 = rfma(kf, kPairLn2N2, -rmul(kf, kPairLn2N2));
    r = quick_sum(r.h, radd(r.l, rsub(x.l, rfma(kf, kPairLn2N3, e2))));
    // e^r - 1 = r + r^2 (1/2 + r/6 + ...), |r| <= ln2/128
    const float t = rmul(r.h, rfma(r.h, rfma(r.h, 1.0f / 120.0f, 1.0f / 24.0f), 1.0f / 6.0f));
    const Pf w = addq(r, mul(sq(r), quick_sum(0.5f, t)));
    const int j = k & ((1 << kPairExpBits) - 1);
    const Pf T = {kPairExp2[j][0], kPairExp2[j][1]};
    const float p2 = bitsf(uint32_t((k >> kPairExpBits) + 127) << 23);
    return scale(addq(T, mul(T, w)), p2);
}

// c + x p for |x p| <= |c|.
LSKUM_HD Pf step(float c, Pf x, Pf p) { return addq(c, mul(x, p)); }
LSKUM_HD Pf step(Pf c, Pf x, Pf p) { return addq(c, mul(x, p)); }

// Phi and phi at s, |s| <= kPairMaxS.
LSKUM_HD void phi_pair(Pf s, Pf& Phi, Pf& phi) {
    const int k = int(rmul(rsub(s.h, kPhiLo), kPhiInvW));
    const float c = rfma(float(k) + 0.5f, 1.0f / kPhiInvW, kPhiLo);
    Pf z = quick_sum(-c, s.h);  // exact: |c| >= |s.h|, or the two are within a factor of two
    z = quick_sum(z.h, radd(z.l, s.l));
#ifdef __CUDA_ARCH__
    const float4* row = reinterpret_cast<const float4*>(kPhiTab[k]);
    const float4 u = __ldg(row), v = __ldg(row + 1), w = __ldg(row + 2);
    const float a3 = w.x, a4 = w.y, a5 = w.z, a6 = w.w;
    const Pf a0 = {u.x, u.y}, a1 = {u.z, u.w}, a2 = {v.x, v.y}, b2 = {v.z, v.w};
#else
    const float* t = kPhiTab[k];
    const float a3 = t[8], a4 = t[9], a5 = t[10], a6 = t[11];
    const Pf a0 = {t[0], t[1]}, a1 = {t[2], t[3]}, a2 = {t[4], t[5]}, b2 = {t[6], t[7]};
#endif
    const float x = z.h;
    const float f = rfma(x, rfma(x, rfma(x, a6, a5), a4), a3);
    Pf p = add(a2, Pf{rmul(x, f), 0.0f});
    p = add(a1, mul(z, p));
    Phi = add(a0, mul(z, p));
    const float g = rfma(x, rfma(x, 6.0f * a6, 5.0f * a5), 4.0f * a4);
    p = add(b2, Pf{rmul(x, g), 0.0f});
    p = add(scale(a2, 2.0f), mul(z, p));
    phi = add(a1, mul(z, p));
}

// What both axes of a pair share: means (suffix m) and differences (prefix d).
struct PairState {
    Pf Sxm, Sym, dSx, dSy;  // S along the two axes of the frame
    Pf Km, dK;              // 3/2 + |S|^2/2
    Pf m0, m1, m3, dm0, dm1, dm3;
};

// From q~_0 = b and d = q~_j - b. False if the pair is not this form's (a
// step over kPairStep or a state out of range; NaN included).
LSKUM_HD bool pair_state(const Pf b[4], const Pf d[4], PairState& w) {
    const Pf beta = scale(b[3], -0.5f);
    bool ok = beta.h >= kPairMinBeta && beta.h <= kPairMaxBeta;
    Pf i0, i2;
    rsqrt_pair(beta, i0, i2);
    const Pf ih = scale(i0, 0.5f);
    const Pf eta = norm(mul(scale(d[3], -0.5f), i2));  // dbeta / beta
    // e = i_j / i_0 - 1 = (1 + eta)^(-1/2) - 1
    const float x = eta.h;
    const float te = rmul(x, rfma(x, rfma(x, rfma(x, rfma(x, 0.176197052f, -0.185470581f), 0.196380615f),
                                          -0.20947265625f), 0.2255859375f));
    const Pf Q = step(0.375f, eta, step(-0.3125f, eta, step(0.2734375f, eta, quick_sum(-0.24609375f, te))));
    const Pf e = norm(addq(scale(eta, -0.5f), mul(sq(eta), Q)));
    const Pf Sx = mul(b[1], ih), Sy = mul(b[2], ih);
    w.dSx = mul(ih, add(d[1], mul(e, add(b[1], d[1]))));
    w.dSy = mul(ih, add(d[2], mul(e, add(b[2], d[2]))));
    w.Sxm = add(Sx, scale(w.dSx, 0.5f));
    w.Sym = add(Sy, scale(w.dSy, 0.5f));
    const Pf SS = add(sq(Sx), sq(Sy));
    const Pf dSS = scale(add(mul(w.Sxm, w.dSx), mul(w.Sym, w.dSy)), 2.0f);
    w.dK = scale(dSS, 0.5f);
    w.Km = addq(1.5f, scale(add(SS, w.dK), 0.5f));
    const Pf arg = add(b[0], SS), W = norm(add(d[0], dSS));
    ok = ok && fabsf(x) <= kPairStep && fabsf(w.dSx.h) <= kPairStep && fabsf(w.dSy.h) <= kPairStep &&
         fabsf(W.h) <= kPairStepW && fabsf(arg.h) <= kPairMaxArg &&
         rfma(w.Sxm.h, w.Sxm.h, rmul(w.Sym.h, w.Sym.h)) <= kPairMaxS * kPairMaxS;  // in every frame
    if (!ok) return false;
    // relative step r0 of m0 = E i^6: (1 + F)(1 + P) - 1 with F = e^W - 1 and P
    // = (1 + e)^6 - 1. W and 6 e are several times their sum, so the linear
    // terms are added first, apart from the higher ones.
    const float tf = rmul(W.h, rfma(W.h, rfma(W.h, 1.0f / 40320.0f, 1.0f / 5040.0f), 1.0f / 720.0f));
    const Pf F2 = mul(sq(W), step(0.5f, W, step(kSixth, W, step(kTwentyFourth, W, addq(k120th, Pf{tf, 0.0f})))));
    const Pf P2 = mul(sq(e), step(15.0f, e, step(20.0f, e, quick_sum(15.0f, rmul(e.h, radd(e.h, 6.0f))))));
    const Pf e6 = mul(e, 6.0f);
    const Pf r0 = norm(add(add(W, e6), add(add(F2, P2), mul(add(W, F2), add(e6, P2)))));
    const Pf r1 = norm(add(add(r0, e), mul(r0, e)));
    const Pf r3 = norm(add(add(r1, e), mul(r1, e)));
    const Pf m0 = norm(mul(exp_pair(arg), mul(sq(i2), i2))), m1 = norm(mul(m0, i0)), m3 = mul(m1, i0);
    // beta and ln E near their ends together: moments that floats do not hold
    if (!(pair_held(m0.h) && pair_held(m3.h))) return false;
    w.dm0 = mul(m0, r0);
    w.dm1 = mul(m1, r1);
    w.dm3 = mul(m3, r3);
    w.m0 = addq(m0, scale(w.dm0, 0.5f));
    w.m1 = addq(m1, scale(w.dm1, 0.5f));
    w.m3 = addq(m3, scale(w.dm3, 0.5f));
    return true;
}

// mean and difference of a product of two quantities from theirs
LSKUM_HD Pf d_prod(Pf xm, Pf dx, Pf ym, Pf dy) { return add(mul(xm, dy), mul(ym, dx)); }
LSKUM_HD Pf m_prod(Pf xm, Pf dx, Pf ym, Pf dy) { return add(mul(xm, ym), scale(mul(dx, dy), 0.25f)); }

// dG = G(state j) - G(state 0) of the split flux along the axis with S = (Sm,
// dS) (mean, difference) and transverse (Bm, dB), for positive molecules: {mass,
// axis momentum, transverse momentum, energy}. For negative ones pass -Sm, -dS
// and negate all but the axis momentum.
LSKUM_HD void split_diff(const PairState& w, Pf Sm, Pf dS, Pf Bm, Pf dB, Pf dG[4]) {
    Pf Phi, phi;
    phi_pair(Sm, Phi, phi);
    const Pf h = scale(dS, 0.5f), hh = sq(h), v = mul(phi, hh);
    const float m = Sm.h, q = rmul(m, m), t = hh.h;
    // Hermite polynomials of the midpoint: the higher terms in float
    const Pf H2_6 = mul(addq(Pf{-1.0f, 0.0f}, scale(sq(Sm), 2.0f)), kThird);  // (4 m^2 - 2) / 6
    const float H3 = rmul(m, rfma(8.0f, q, -12.0f)), H4 = rfma(rfma(16.0f, q, -48.0f), q, 12.0f);
    const float H5 = rmul(m, rfma(rfma(32.0f, q, -160.0f), q, 120.0f));
    const float H6 = rfma(rfma(rfma(64.0f, q, -480.0f), q, 720.0f), q, -120.0f);
    const Pf cP = add(H2_6, Pf{rmul(t, rfma(rmul(t, H6), 1.0f / 5040.0f, rmul(H4, 1.0f / 120.0f))), 0.0f});
    const Pf cM = add(Sm, Pf{rmul(t, rfma(rmul(t, H5), 1.0f / 720.0f, rmul(H3, 1.0f / 24.0f))), 0.0f});
    const Pf cT = add(mul(Sm, kThird), Pf{rmul(t, rfma(rmul(t, H5), 1.0f / 5040.0f, rmul(H3, 1.0f / 120.0f))), 0.0f});
    const Pf cU = quick_sum(0.5f, rmul(t, rfma(rmul(t, H4), 1.0f / 720.0f, rmul(H2_6.h, 0.25f))));
    const Pf dPhi = mul(dS, add(phi, mul(v, cP)));
    const Pf Phim = add(Phi, neg(mul(v, cM)));
    const Pf dT = mul(dS, add(Phi, neg(mul(v, cT))));
    const Pf Tm = add(add(mul(Sm, Phi), scale(phi, 0.5f)), mul(v, cU));

    dG[0] = d_prod(w.m0, w.dm0, Tm, dT);
    const Pf dX = add(d_prod(Sm, dS, Tm, dT), scale(dPhi, 0.5f));
    const Pf Xm = add(m_prod(Sm, dS, Tm, dT), scale(Phim, 0.5f));
    dG[1] = d_prod(w.m1, w.dm1, Xm, dX);
    const Pf dY = d_prod(Bm, dB, Tm, dT), Ym = m_prod(Bm, dB, Tm, dT);
    dG[2] = d_prod(w.m1, w.dm1, Ym, dY);
    const Pf dZ = add(d_prod(w.Km, w.dK, Tm, dT), scale(d_prod(Sm, dS, Phim, dPhi), 0.25f));
    const Pf Zm = add(m_prod(w.Km, w.dK, Tm, dT), scale(m_prod(Sm, dS, Phim, dPhi), 0.25f));
    dG[3] = d_prod(w.m3, w.dm3, Zm, dZ);
}

}  // namespace lskum
