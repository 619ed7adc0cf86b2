// Mixed-precision kernels of the q-LSKUM hot path (sm_103a).
//
// FP32 for the stencil, least-squares and split-flux arithmetic; FP64 for
// the state accumulation U += dt R, float pairs (2^-46) for the q-variables
// derived from U, which are stored as such, FP64 for the 2x2
// least-squares determinants (folded into weights on the host in FP64 and
// stored as FP32), the residue and the force integral.
//
// Differences are what the method consumes -- q_j - q_i in the
// least-squares sums and G(q~_j) - G(q~_0) in the split-flux derivatives --
// and at fine resolution they are 1e-4 of the values, so FP32 values would
// lose four of their seven digits in each subtraction. The FP32 path
// therefore never subtracts two nearby values:
//   * q is stored as a pair of floats (hi + lo = the FP64 q to ~2^-48), so
//     q_j - q_i = (hi_j - hi_i) + (lo_j - lo_i) is accurate to FP32
//     precision relative to the difference itself;
//   * a pair's split fluxes are differenced in the variables of flux_pair.cuh
//     (S = u sqrt(beta), 1/sqrt(beta), E): products by the product rule, E by
//     expm1, Phi and T by their midpoint expansions; for steps of S over 1/4
//     and other gammas the primitive state of q~_j is formed as base +
//     difference (quotient identities, log1p, expm1) and each flux likewise.
// The result is the same residual as the FP64 path to about FP32 relative
// precision of the residual itself, not of the fluxes.

#include <cmath>

#include "device_math.cuh"
#include "flux_mixed.cuh"
#include "flux_pair.cuh"
#include "lskum_internal.h"
#include "lskum_kernels.cuh"
#include "pair_convert.cuh"

namespace lskum {

namespace {

// q_j - q_i from the hi/lo float pairs.
__device__ __forceinline__ float4 qdiff(const QHL& a, const QHL& b) {
    return make_float4((a.hi.x - b.hi.x) + (a.lo.x - b.lo.x), (a.hi.y - b.hi.y) + (a.lo.y - b.lo.y),
                       (a.hi.z - b.hi.z) + (a.lo.z - b.lo.z), (a.hi.w - b.hi.w) + (a.lo.w - b.lo.w));
}

// ----------------------------------------------------------- q-derivatives

// Both sweeps stream, per neighbour entry, the packed neighbour word and the
// FP32 weight pair {wx, wy}, then gather the neighbour's record with the
// index that word holds. Entries are taken in groups of kLsAhead, and the
// next group's stream loads are issued before the current group's gathers,
// so a thread has a group of DRAM loads in flight while it waits on the
// cache-resident gathers (12-13 % less time per sweep at 10M points than a
// plain unrolled loop; staging the stream or the tile's own records in
// shared memory was slower). Slots at or past the point's count c are not
// read.
constexpr int kLsAhead = 4;

__device__ __forceinline__ void load_ls_entries(const DevGeom& g, const DevGeom32& g32,
                                                const int64_t d, const int k0, const int c,
                                                uint32_t e[kLsAhead], float2 w[kLsAhead]) {
#pragma unroll
    for (int u = 0; u < kLsAhead; ++u) {
        if (k0 + u < c) {
            const int64_t at = int64_t(k0 + u) * g.stride + d;
            e[u] = g.nbr[at];
            w[u] = g32.lw2[at];
        }
    }
}

template <int BLOCK>
__global__ void __launch_bounds__(BLOCK) k_ls_first_mx(const DevGeom g, const DevGeom32 g32,
                                                       const QHL* __restrict__ q,
                                                       D8f* __restrict__ dq) {
    const int64_t t = int64_t(blockIdx.x) * BLOCK + threadIdx.x;  // (point, condition)
    const int64_t d = t >> g.cshift;
    const uint32_t cc = uint32_t(t) & g.cmask;
    if (d >= g.n) return;
    const int c = g.cnt[d];
    const QHL qi = q[t];
    float4 ax = make_float4(0.f, 0.f, 0.f, 0.f), ay = ax;
    uint32_t en[kLsAhead] = {};
    float2 wn[kLsAhead] = {};
    load_ls_entries(g, g32, d, 0, c, en, wn);
    for (int k0 = 0; k0 < c; k0 += kLsAhead) {
        uint32_t ec[kLsAhead];
        float2 wc[kLsAhead];
#pragma unroll
        for (int u = 0; u < kLsAhead; ++u) {
            ec[u] = en[u];
            wc[u] = wn[u];
        }
        load_ls_entries(g, g32, d, k0 + kLsAhead, c, en, wn);
#pragma unroll
        for (int u = 0; u < kLsAhead; ++u) {
            if (k0 + u < c) {
                const float wx = wc[u].x, wy = wc[u].y;
                const float4 dqv = qdiff(q[sidx(g, ec[u] & kIndexMask, cc)], qi);
                ax.x = fmaf(wx, dqv.x, ax.x); ax.y = fmaf(wx, dqv.y, ax.y);
                ax.z = fmaf(wx, dqv.z, ax.z); ax.w = fmaf(wx, dqv.w, ax.w);
                ay.x = fmaf(wy, dqv.x, ay.x); ay.y = fmaf(wy, dqv.y, ay.y);
                ay.z = fmaf(wy, dqv.z, ay.z); ay.w = fmaf(wy, dqv.w, ay.w);
            }
        }
    }
    dq[t] = D8f{ax, ay};
}

// One Jacobi sweep of Eq. 29 as the first-order derivative of the stage
// (dq_first, the sum of wx_j (q_j - q_i)) minus the sum of wx_j (hdx_j
// (qx_j - qx_i) + hdy_j (qy_j - qy_i)): the q gathers and their float-pair
// differences are done once per stage, not per sweep; the derivative
// differences stay differences (exact in FP32 for nearby values). The
// per-neighbour stream is the 8-byte weight pair; the half offsets come from
// the gathered coordinate pairs of the neighbour (cache-resident: the
// neighbours of a warp's points are close in the Hilbert order).
template <int BLOCK>
__global__ void __launch_bounds__(BLOCK) k_ls_inner_mx(const DevGeom g, const DevGeom32 g32,
                                                       const D8f* __restrict__ dq_first,
                                                       const D8f* __restrict__ din,
                                                       D8f* __restrict__ dout) {
    const int64_t t = int64_t(blockIdx.x) * BLOCK + threadIdx.x;  // (point, condition)
    const int64_t d = t >> g.cshift;
    const uint32_t cc = uint32_t(t) & g.cmask;
    if (d >= g.n) return;
    const int c = g.cnt[d];
    const D8f di = din[t];
    const float4 pi = g32.xyhl[d];
    float4 ax = make_float4(0.f, 0.f, 0.f, 0.f), ay = ax;
    uint32_t en[kLsAhead] = {};
    float2 wn[kLsAhead] = {};
    load_ls_entries(g, g32, d, 0, c, en, wn);
    for (int k0 = 0; k0 < c; k0 += kLsAhead) {
        uint32_t ec[kLsAhead];
        float2 wc[kLsAhead];
#pragma unroll
        for (int u = 0; u < kLsAhead; ++u) {
            ec[u] = en[u];
            wc[u] = wn[u];
        }
        load_ls_entries(g, g32, d, k0 + kLsAhead, c, en, wn);
#pragma unroll
        for (int u = 0; u < kLsAhead; ++u) {
            if (k0 + u < c) {
                const uint32_t j = ec[u] & kIndexMask;
                const float wx = wc[u].x, wy = wc[u].y;
                const float4 pj = g32.xyhl[j];
                const D8f dj = din[sidx(g, j, cc)];
                const float hx = 0.5f * ((pj.x - pi.x) + (pj.z - pi.z));
                const float hy = 0.5f * ((pj.y - pi.y) + (pj.w - pi.w));
                // (dx (qx_j - qx_i) + dy (qy_j - qy_i)) / 2, the Eq. 28 correction
                const float t0 = fmaf(hx, dj.x.x - di.x.x, hy * (dj.y.x - di.y.x));
                const float t1 = fmaf(hx, dj.x.y - di.x.y, hy * (dj.y.y - di.y.y));
                const float t2 = fmaf(hx, dj.x.z - di.x.z, hy * (dj.y.z - di.y.z));
                const float t3 = fmaf(hx, dj.x.w - di.x.w, hy * (dj.y.w - di.y.w));
                ax.x = fmaf(wx, t0, ax.x); ax.y = fmaf(wx, t1, ax.y);
                ax.z = fmaf(wx, t2, ax.z); ax.w = fmaf(wx, t3, ax.w);
                ay.x = fmaf(wy, t0, ay.x); ay.y = fmaf(wy, t1, ay.y);
                ay.z = fmaf(wy, t2, ay.z); ay.w = fmaf(wy, t3, ay.w);
            }
        }
    }
    const D8f f = dq_first[t];
    dout[t] = D8f{make_float4(f.x.x - ax.x, f.x.y - ax.y, f.x.z - ax.z, f.x.w - ax.w),
                  make_float4(f.y.x - ay.x, f.y.y - ay.y, f.y.z - ay.z, f.y.w - ay.w)};
}

// The same sweeps with four threads a (point, condition), a component of q each,
// to the same bits: for clouds that one thread a point does not fill the chip
// with (see kMxSplitSweep).
template <int BLOCK>
__global__ void __launch_bounds__(BLOCK) k_ls_first_mx4(const DevGeom g, const DevGeom32 g32,
                                                        const QHL* __restrict__ q, D8f* __restrict__ dq) {
    const int64_t t = (int64_t(blockIdx.x) * BLOCK + threadIdx.x) / 4;  // (point, condition)
    const int m = threadIdx.x % 4;
    const int64_t d = t >> g.cshift;
    const uint32_t cc = uint32_t(t) & g.cmask;
    if (d >= g.n) return;
    const float* qm = reinterpret_cast<const float*>(q) + m;
    const float hi = qm[8 * t], lo = qm[8 * t + 4];
    float ax = 0.f, ay = 0.f;
    const int c = g.cnt[d];
#pragma unroll 4
    for (int k = 0; k < c; ++k) {
        const int64_t at = int64_t(k) * g.stride + d;
        const float* qj = qm + 8 * sidx(g, g.nbr[at] & kIndexMask, cc);
        const float2 w = g32.lw2[at];
        const float e = (qj[0] - hi) + (qj[4] - lo);
        ax = fmaf(w.x, e, ax);
        ay = fmaf(w.y, e, ay);
    }
    float* o = reinterpret_cast<float*>(dq + t) + m;
    o[0] = ax;
    o[4] = ay;
}

template <int BLOCK>
__global__ void __launch_bounds__(BLOCK) k_ls_inner_mx4(const DevGeom g, const DevGeom32 g32,
                                                        const D8f* __restrict__ dq_first,
                                                        const D8f* __restrict__ din,
                                                        D8f* __restrict__ dout) {
    const int64_t t = (int64_t(blockIdx.x) * BLOCK + threadIdx.x) / 4;  // (point, condition)
    const int m = threadIdx.x % 4;
    const int64_t d = t >> g.cshift;
    const uint32_t cc = uint32_t(t) & g.cmask;
    if (d >= g.n) return;
    const float* im = reinterpret_cast<const float*>(din) + m;
    const float xi = im[8 * t], yi = im[8 * t + 4];
    const float4 pi = g32.xyhl[d];
    float ax = 0.f, ay = 0.f;
    const int c = g.cnt[d];
#pragma unroll 4
    for (int k = 0; k < c; ++k) {
        const int64_t at = int64_t(k) * g.stride + d;
        const uint32_t j = g.nbr[at] & kIndexMask;
        const float2 w = g32.lw2[at];
        const float4 pj = g32.xyhl[j];
        const float* dj = im + 8 * sidx(g, j, cc);
        const float hx = 0.5f * ((pj.x - pi.x) + (pj.z - pi.z));
        const float hy = 0.5f * ((pj.y - pi.y) + (pj.w - pi.w));
        const float v = fmaf(hx, dj[0] - xi, hy * (dj[4] - yi));
        ax = fmaf(w.x, v, ax);
        ay = fmaf(w.y, v, ay);
    }
    const float* f = reinterpret_cast<const float*>(dq_first + t) + m;
    float* o = reinterpret_cast<float*>(dout + t) + m;
    o[0] = f[0] - ax;
    o[4] = f[4] - ay;
}

__device__ __forceinline__ QHL split_hl(const V4& q) {
    const Pf a = nearest_pair(q.a), b = nearest_pair(q.b), c = nearest_pair(q.c), d = nearest_pair(q.d);
    return QHL{make_float4(a.h, b.h, c.h, d.h), make_float4(a.l, b.l, c.l, d.l)};
}

// 1/b and ln of a mantissa product in float pairs, for the next stage's
// q-variables: FP64 from here on would hold the kernel to the FP64 pipe (45
// operations a point, 0.3 ms at 2.5M points).
__device__ __forceinline__ Pf recip_pair(const Pf b) {
    float y;
    asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(b.h));
    const float r = rfma(-b.l, y, rfma(-b.h, y, 1.0f));
    return quick_sum(y, rmul(y, rfma(r, r, r)));
}

// e ln2 for an integer e, |e| < 2^12.
__device__ __forceinline__ Pf times_ln2(const float e) {
    return add(Pf{rmul(e, kPairLn2Hi), 0.0f}, mul(Pf{kPairLn2Mid, kPairLn2Lo}, e));  // the first is exact
}

// ln x for a normal x > 0: x = 2^e m, F = 1/m to eight bits, r = m F - 1 (exact
// but for m's low part, |r| <= 2^-7), ln x = e ln2 - ln F + log1p(r).
__device__ __forceinline__ Pf log_pair(const Pf x) {
    const int e = int(fbits(x.h) >> 23) - 127;
    const float sc = bitsf(uint32_t(127 - e) << 23);
    const Pf m = scale(x, sc);
    const float* t = kPairLog[(fbits(m.h) >> 16) & 127u];
    const Pf r = quick_sum(rfma(m.h, __ldg(t), -1.0f), rmul(m.l, __ldg(t)));
    const float q = r.h;
    const float tail = rmul(rmul(q, rmul(q, q)), rfma(q, rfma(q, rfma(q, -1.0f / 6.0f, 0.2f), -0.25f), 1.0f / 3.0f));
    Pf s = addq(r, scale(sq(r), -0.5f));
    s.l = radd(s.l, tail);
    return add(add(times_ln2(float(e)), Pf{__ldg(t + 1), __ldg(t + 2)}), s);
}

// q-variables (Eq. 26, gamma = 1.4) of the conserved state in float pairs, to
// ~2^-46 (their pairs are what is stored). False for a state whose sizes
// floats do not hold with room (the caller takes FP64).
__device__ __forceinline__ bool q_of_cons_pair(const V4& U, QHL& q) {
    const Pf rho = split_pair(U.a), mx = split_pair(U.b), my = split_pair(U.c), en = split_pair(U.d);
    const Pf m2 = add(sq(mx), sq(my));
    const Pf rp = mul(sub(mul(en, rho), scale(m2, 0.5f)), Pf{0.4f, float(0.4 - double(0.4f))});  // rho p
    if (!(rho.h > 1e-7f && rho.h < 1e7f && rp.h > 1e-14f && rp.h < 1e14f && m2.h < 1e14f)) return false;
    const Pf ir = recip_pair(norm(rp));
    const Pf ip = norm(mul(rho, ir));  // 1/p
    const Pf b2 = mul(rho, ip);        // 2 beta
    // ln rho + 2.5 ln beta = ln(rho^2 beta^5) / 2, powers of two kept apart
    const int er = int(fbits(rho.h) >> 23) - 127, eb = int(fbits(b2.h) >> 23) - 127;
    const Pf rm = scale(rho, bitsf(uint32_t(127 - er) << 23)), bm = norm(scale(b2, bitsf(uint32_t(127 - eb) << 23)));
    const Pf L = log_pair(norm(mul(sq(rm), mul(sq(sq(bm)), bm))));
    const Pf ln = add(times_ln2(float(2 * er + 5 * (eb - 1))), L);
    const Pf q1 = norm(scale(sub(ln, mul(m2, ir)), 0.5f));  // |m|^2 / (2 rho p) = beta |u|^2
    const Pf q2 = norm(mul(mx, ip)), q3 = norm(mul(my, ip)), q4 = norm(b2);
    q.hi = make_float4(q1.h, q2.h, q3.h, -q4.h);
    q.lo = make_float4(q1.l, q2.l, q3.l, -q4.l);
    return true;
}

__device__ __forceinline__ bool physical(double rho, double u, double v, double p) {
    return rho > 0.0 && p > 0.0 && isfinite(rho) && isfinite(p) && isfinite(u) && isfinite(v);
}

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
    return s;
}

// ------------------------------------------------------- flux residual + RK

struct MxFrame {
    float tx, ty, nx, ny;
    bool local;
};

// One entry by the primitive differences: any gamma, any step.
template <bool G14>
__device__ __forceinline__ float4 entry_prim(const float4 base, const float4 dlt, const float gm1_inv,
                                          const MxFrame f, const uint32_t e, const float ws, const float wn) {
    PrimPair w = prim_pair<G14>(base, dlt, gm1_inv);
    if (f.local) {
        const float s0 = w.u * f.tx + w.v * f.ty, n0 = w.u * f.nx + w.v * f.ny;
        const float ds = w.du * f.tx + w.dv * f.ty, dn = w.du * f.nx + w.dv * f.ny;
        w.u = s0; w.v = n0; w.du = ds; w.dv = dn;
    }
    const uint32_t sc = (e >> kIndexBits) & 3u, nc = (e >> (kIndexBits + 2)) & 3u;
    float4 R = make_float4(0.f, 0.f, 0.f, 0.f);
    float dG[4];
    if (sc) {
        dsplit_flux_a(w, w.u, w.v, w.du, w.dv, sc == 1u ? 1.f : -1.f, dG);
        R = make_float4(ws * dG[0], ws * dG[1], ws * dG[2], ws * dG[3]);
    }
    if (nc) {
        dsplit_flux_a(w, w.v, w.u, w.dv, w.du, nc == 1u ? 1.f : -1.f, dG);
        R = make_float4(fmaf(wn, dG[0], R.x), fmaf(wn, dG[2], R.y), fmaf(wn, dG[1], R.z), fmaf(wn, dG[3], R.w));
    }
    return R;
}

// For gamma = 1.4, where few entries need it: out of the loop's code.
__device__ __noinline__ float4 entry_prim_g14(const float4 base, const float4 dlt, const MxFrame f,
                                              const uint32_t e, const float ws, const float wn) {
    return entry_prim<true>(base, dlt, 2.5f, f, e, ws, wn);
}

// -x where the sign bit of m is set.
__device__ __forceinline__ float flip(const float x, const uint32_t m) {
    return __uint_as_float(__float_as_uint(x) ^ (m & 0x80000000u));
}

constexpr int kMxClasses = 4;
// Four threads share a point up to this many (point, condition) pairs: one a
// point leaves SMs idle there. Microseconds a launch, one thread / four: 5,120
// points 35 / 17, 46,080 38 / 27, 79,948 42 / 33, 150,598 54.8 / 55.1.
constexpr int64_t kMxSplitPairs = 1 << 17;
// The same for the sweeps, whose set-up weighs more: the iteration of 5,120
// points takes 127 / 120 us, of 30,070 155 / 150; a sweep of 79,948 12 / 16.
constexpr int64_t kMxSplitSweep = 1 << 15;

// Issue-bound (76 % of the slots at 0.6M points, FP64 pipe 15 %: 145 us a launch;
// with the primitive differences, and q and every conversion on the FP64 pipe,
// 172 us and 57 %; 2.5M points 608 -> 530). Each neighbour entry's stream loads
// (packed word, FP32 constants) are issued one entry ahead, so that only the
// gathers they index are waited on; registers capped at 72. A point's
// entries are summed by class (slot mod kMxClasses) and the classes in order, by
// one thread of a point or by kMxClasses, to the same bits.
template <int MODE, int BLOCK, bool G14, int LANES>
__global__ void __launch_bounds__(BLOCK, 896 / BLOCK) k_flux_mx(const DevGeom g, const DevGeom32 g32,
                                                   const Physics ph, const DevState st,
                                                   const QHL* __restrict__ q_in,
                                                   const D8f* __restrict__ dq,
                                                   QHL* __restrict__ q_out) {
    const int64_t t = (int64_t(blockIdx.x) * BLOCK + threadIdx.x) / LANES;  // (point, condition)
    const int64_t d = t >> g.cshift;
    const uint32_t cc = uint32_t(t) & g.cmask;
    const int part = LANES == 1 ? 0 : threadIdx.x % LANES;
    const bool live = d < g.n;
    const int8_t fl = live ? g.flag[d] : int8_t(LSKUM_INTERIOR);
    const bool fixed = ph.outer_fixed && fl == LSKUM_OUTER;
    float R[4] = {0.f, 0.f, 0.f, 0.f};
    MxFrame f = {1.f, 0.f, 0.f, 1.f, fl != LSKUM_INTERIOR};
    if (live && !fixed) {
        if (f.local) {
            const double2 nn = g.nrm[d];
            f.nx = float(nn.x);
            f.ny = float(nn.y);
            f.tx = f.ny;
            f.ty = -f.nx;
        }
        const QHL qi = q_in[t];
        const D8f di = dq[t];
        const float4 qiv = make_float4(qi.hi.x + qi.lo.x, qi.hi.y + qi.lo.y, qi.hi.z + qi.lo.z,
                                       qi.hi.w + qi.lo.w);
        const float gm1_inv = float(ph.gm1_inv);
        const bool second = ph.order == 2;
        const int c = g.cnt[d];
        int k = part, r = part;  // the class r's next entry
        float S[4] = {0.f, 0.f, 0.f, 0.f};
        uint32_t e_next = 0u;
        float4 fw_next = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k < c) {
            e_next = g.nbr[int64_t(k) * g.stride + d];
            fw_next = g32.fxw[int64_t(k) * g.stride + d];
        }
        while (k < c) {
            const uint32_t e = e_next;
            const float4 fw = fw_next;
            k += kMxClasses;
            bool last = false;  // of its class
            if (k >= c) {
                last = true;
                k = LANES == 1 && r + 1 < kMxClasses ? ++r : c;
            }
            if (k < c) {  // the next entry's stream, in flight during this one
                const int64_t at = int64_t(k) * g.stride + d;
                e_next = g.nbr[at];
                fw_next = g32.fxw[at];
            }
            const int64_t jt = sidx(g, e & kIndexMask, cc);
            const float4 dqv = qdiff(q_in[jt], qi);
            float4 base = qiv, dlt = dqv;
            if (second) {
                const float hx = fw.z, hy = fw.w;
                const D8f dj = dq[jt];
                // q~_0 = q_i - (dx q_x,i + dy q_y,i)/2; dq~ = q~_j - q~_0 (Eq. 28)
                base.x = qiv.x - (hx * di.x.x + hy * di.y.x);
                base.y = qiv.y - (hx * di.x.y + hy * di.y.y);
                base.z = qiv.z - (hx * di.x.z + hy * di.y.z);
                base.w = qiv.w - (hx * di.x.w + hy * di.y.w);
                dlt.x = dqv.x - (hx * (dj.x.x - di.x.x) + hy * (dj.y.x - di.y.x));
                dlt.y = dqv.y - (hx * (dj.x.y - di.x.y) + hy * (dj.y.y - di.y.y));
                dlt.z = dqv.z - (hx * (dj.x.z - di.x.z) + hy * (dj.y.z - di.y.z));
                dlt.w = dqv.w - (hx * (dj.x.w - di.x.w) + hy * (dj.y.w - di.y.w));
            }
            MxState w;
            if (G14 && mx_state(base, dlt, w)) {
                if (f.local) {
                    const float sm = w.Sxm * f.tx + w.Sym * f.ty, nm = w.Sxm * f.nx + w.Sym * f.ny;
                    const float sd = w.dSx * f.tx + w.dSy * f.ty, nd = w.dSx * f.nx + w.dSy * f.ny;
                    w.Sxm = sm; w.Sym = nm; w.dSx = sd; w.dSy = nd;
                }
                // an entry outside a stencil has weight 0 there
                float dG[4];
                uint32_t neg = e << (30 - kIndexBits);  // the sign bit: code 2
                float wf = flip(fw.x, neg);
                mx_diff(w, flip(w.Sxm, neg), flip(w.dSx, neg), w.Sym, w.dSy, dG);
                S[0] = fmaf(wf, dG[0], S[0]);
                S[1] = fmaf(fw.x, dG[1], S[1]);
                S[2] = fmaf(wf, dG[2], S[2]);
                S[3] = fmaf(wf, dG[3], S[3]);
                neg = e << (28 - kIndexBits);
                wf = flip(fw.y, neg);
                mx_diff(w, flip(w.Sym, neg), flip(w.dSy, neg), w.Sxm, w.dSx, dG);
                S[0] = fmaf(wf, dG[0], S[0]);
                S[1] = fmaf(wf, dG[2], S[1]);
                S[2] = fmaf(fw.y, dG[1], S[2]);
                S[3] = fmaf(wf, dG[3], S[3]);
            } else if (!(dlt.x == 0.f && dlt.y == 0.f && dlt.z == 0.f && dlt.w == 0.f)) {
                const float4 a = G14 ? entry_prim_g14(base, dlt, f, e, fw.x, fw.y)
                                     : entry_prim<false>(base, dlt, gm1_inv, f, e, fw.x, fw.y);
                S[0] += a.x;
                S[1] += a.y;
                S[2] += a.z;
                S[3] += a.w;
            }
            if (last) {
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    R[m] = LANES == 1 ? R[m] + S[m] : S[m];
                    S[m] = 0.f;
                }
            }
        }
    }
    if (LANES > 1) {
#pragma unroll
        for (int r = 1; r < LANES; ++r)
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const float o = __shfl_down_sync(0xffffffffu, R[m], r);
                if (part == 0) R[m] += o;
            }
    }
    // the stage update: a thread for each point
    int64_t tu = t, du = d;
    int8_t flu = fl;
    bool update = live;
    if (LANES > 1) {
        __shared__ float s_R[BLOCK / LANES][4];
        if (part == 0)
#pragma unroll
            for (int m = 0; m < 4; ++m) s_R[threadIdx.x / LANES][m] = R[m];
        __syncthreads();
        tu = int64_t(blockIdx.x) * (BLOCK / LANES) + threadIdx.x;
        du = tu >> g.cshift;
        update = threadIdx.x < BLOCK / LANES && du < g.n;
        if (update) {
            flu = g.flag[du];
#pragma unroll
            for (int m = 0; m < 4; ++m) R[m] = s_R[threadIdx.x][m];
        }
    }
    double r2 = 0.0;
    if (update) {
        const bool fixu = ph.outer_fixed && flu == LSKUM_OUTER;
        if (flu != LSKUM_INTERIOR && !fixu) {  // momentum back to the global frame
            const double2 nn = g.nrm[du];
            const float nx = float(nn.x), ny = float(nn.y);
            const float rs = R[1], rn = R[2];
            R[1] = rs * ny + rn * nx;
            R[2] = rn * ny - rs * nx;
        }
        // FP64: state accumulation, wall condition, residue; the next q in pairs
        const double R0 = widen(R[0]), R1 = widen(R[1]), R2 = widen(R[2]), R3 = widen(R[3]);
        if (MODE == 0) {
            st.R[tu] = V4{R[0], R[1], R[2], R[3]};
        } else {
            V4 U = st.U[tu];
            double dtv;
            if (MODE == 1) {
                // local time step in FP32: it sets the pseudo-time path, not
                // the steady state, and FP32 square roots and quotients cost
                // a fraction of the FP64 pipe's
                const float rho = float(U.a), irho = 1.0f / rho;
                const float u = float(U.b) * irho, v = float(U.c) * irho;
                const float uu = fmaf(u, u, v * v);
                const float p = float(ph.gm1) * (float(U.d) - 0.5f * rho * uu);
                dtv = double(float(ph.cfl * g.dmin[du]) /
                             (sqrtf(uu) + sqrtf(float(ph.gamma) * p * irho)));
                st.dt[tu] = dtv;
                st.U0[tu] = U;
                r2 = R0 * R0;
            } else {
                dtv = st.dt[tu];
            }
            if (!fixu) {
                const double h = 0.5 * dtv;
                if (MODE == 3) {
                    const V4 U0 = st.U0[tu];
                    U.a = (2.0 / 3.0) * U0.a + (1.0 / 3.0) * (U.a - h * R0);
                    U.b = (2.0 / 3.0) * U0.b + (1.0 / 3.0) * (U.b - h * R1);
                    U.c = (2.0 / 3.0) * U0.c + (1.0 / 3.0) * (U.c - h * R2);
                    U.d = (2.0 / 3.0) * U0.d + (1.0 / 3.0) * (U.d - h * R3);
                } else {
                    U.a -= h * R0;
                    U.b -= h * R1;
                    U.c -= h * R2;
                    U.d -= h * R3;
                }
                if (flu == LSKUM_WALL) {
                    const double2 nn = g.nrm[du];
                    const double tx = nn.y, ty = -nn.x;
                    const double ms = U.b * tx + U.c * ty;
                    U.b = ms * tx;
                    U.c = ms * ty;
                }
                st.U[tu] = U;
            }
            QHL qn;
            if (!(G14 && q_of_cons_pair(U, qn))) {
                V4 q;
                double rho, u, v, p;
                cons_to_q64<G14>(U, ph, q, rho, u, v, p);
                qn = split_hl(q);
                if (!physical(rho, u, v, p)) atomicOr(st.status, 1);
            }
            q_out[tu] = qn;
        }
    }
    if (MODE == 1) {
        if (g.cshift == 0) {
            const double s = block_sum<BLOCK>(r2);
            if (threadIdx.x == 0) st.partials[blockIdx.x] = s;
        } else if (update) {
            st.r2[tu] = r2;
        }
    }
}

__global__ void k_q_from_U_mx(const DevGeom g, const Physics ph, const V4* __restrict__ U,
                              QHL* __restrict__ q) {
    const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if ((t >> g.cshift) >= g.n) return;
    V4 qn;
    double rho, u, v, p;
    if (fabs(ph.gm1_inv - 2.5) < 1e-12)
        cons_to_q64<true>(U[t], ph, qn, rho, u, v, p);
    else
        cons_to_q64<false>(U[t], ph, qn, rho, u, v, p);
    q[t] = split_hl(qn);
}

__global__ void k_gather_dq_mx(const DevGeom g, const D8f* __restrict__ src, V4* __restrict__ qx,
                               V4* __restrict__ qy) {
    const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t d = t >> g.cshift;
    if (d >= g.n) return;
    const int64_t at = int64_t(uint32_t(t) & g.cmask) * g.n + g.dev_to_user[d];
    const D8f s = src[t];
    qx[at] = V4{s.x.x, s.x.y, s.x.z, s.x.w};
    qy[at] = V4{s.y.x, s.y.y, s.y.z, s.y.w};
}

inline unsigned grid_for(int64_t n, int block) { return unsigned((n + block - 1) / block); }
inline unsigned grid_nc(const DevGeom& g, int block) { return grid_for(g.n << g.cshift, block); }
inline int mx_flux_lanes(const DevGeom& g) { return (g.n << g.cshift) <= kMxSplitPairs ? kMxClasses : 1; }
inline bool mx_sweep_four(const DevGeom& g) { return (g.n << g.cshift) <= kMxSplitSweep; }

template <int BLOCK, bool G14, int LANES>
void flux_mx_dispatch(int mode, const DevGeom& g, const DevGeom32& g32, const Physics& ph,
                      const DevState& st, const QHL* q_in, const D8f* dq, QHL* q_out,
                      cudaStream_t s) {
    const unsigned grid = grid_for((g.n << g.cshift) * LANES, BLOCK);
    switch (mode) {
        case 0: k_flux_mx<0, BLOCK, G14, LANES><<<grid, BLOCK, 0, s>>>(g, g32, ph, st, q_in, dq, q_out); break;
        case 1: k_flux_mx<1, BLOCK, G14, LANES><<<grid, BLOCK, 0, s>>>(g, g32, ph, st, q_in, dq, q_out); break;
        case 2: k_flux_mx<2, BLOCK, G14, LANES><<<grid, BLOCK, 0, s>>>(g, g32, ph, st, q_in, dq, q_out); break;
        case 3: k_flux_mx<3, BLOCK, G14, LANES><<<grid, BLOCK, 0, s>>>(g, g32, ph, st, q_in, dq, q_out); break;
        default: k_flux_mx<4, BLOCK, G14, LANES><<<grid, BLOCK, 0, s>>>(g, g32, ph, st, q_in, dq, q_out); break;
    }
}

template <int BLOCK, bool G14>
void flux_mx_lanes(int mode, const DevGeom& g, const DevGeom32& g32, const Physics& ph, const DevState& st,
                   const QHL* q_in, const D8f* dq, QHL* q_out, cudaStream_t s) {
    if (mx_flux_lanes(g) > 1)
        flux_mx_dispatch<BLOCK, G14, kMxClasses>(mode, g, g32, ph, st, q_in, dq, q_out, s);
    else
        flux_mx_dispatch<BLOCK, G14, 1>(mode, g, g32, ph, st, q_in, dq, q_out, s);
}

}  // namespace

int64_t mx_flux_blocks(const DevGeom& g, int block) {
    return grid_for((g.n << g.cshift) * mx_flux_lanes(g), block);
}

cudaError_t launch_ls_first_mx(const DevGeom& g, const DevGeom32& g32, const QHL* q, D8f* dq,
                               int block, cudaStream_t s) {
    const bool four = mx_sweep_four(g);
    const unsigned grid = grid_for((g.n << g.cshift) * (four ? 4 : 1), block);
    if (block == 256) {
        if (four) k_ls_first_mx4<256><<<grid, 256, 0, s>>>(g, g32, q, dq);
        else k_ls_first_mx<256><<<grid, 256, 0, s>>>(g, g32, q, dq);
    } else {
        if (four) k_ls_first_mx4<kDefaultBlock><<<grid, kDefaultBlock, 0, s>>>(g, g32, q, dq);
        else k_ls_first_mx<kDefaultBlock><<<grid, kDefaultBlock, 0, s>>>(g, g32, q, dq);
    }
    return cudaGetLastError();
}

cudaError_t launch_ls_inner_mx(const DevGeom& g, const DevGeom32& g32, const D8f* dq_first,
                               const D8f* din, D8f* dout, int block, cudaStream_t s) {
    const bool four = mx_sweep_four(g);
    const unsigned grid = grid_for((g.n << g.cshift) * (four ? 4 : 1), block);
    if (block == 256) {
        if (four) k_ls_inner_mx4<256><<<grid, 256, 0, s>>>(g, g32, dq_first, din, dout);
        else k_ls_inner_mx<256><<<grid, 256, 0, s>>>(g, g32, dq_first, din, dout);
    } else {
        if (four) k_ls_inner_mx4<kDefaultBlock><<<grid, kDefaultBlock, 0, s>>>(g, g32, dq_first, din, dout);
        else k_ls_inner_mx<kDefaultBlock><<<grid, kDefaultBlock, 0, s>>>(g, g32, dq_first, din, dout);
    }
    return cudaGetLastError();
}

cudaError_t launch_flux_mx(int mode, const DevGeom& g, const DevGeom32& g32, const Physics& ph,
                           const DevState& st, const QHL* q_in, const D8f* dq, QHL* q_out,
                           int block, cudaStream_t s) {
    const bool g14 = fabs(ph.gm1_inv - 2.5) < 1e-12;
    if (block == 256) {
        if (g14) flux_mx_lanes<256, true>(mode, g, g32, ph, st, q_in, dq, q_out, s);
        else flux_mx_lanes<256, false>(mode, g, g32, ph, st, q_in, dq, q_out, s);
    } else {
        if (g14) flux_mx_lanes<kDefaultBlock, true>(mode, g, g32, ph, st, q_in, dq, q_out, s);
        else flux_mx_lanes<kDefaultBlock, false>(mode, g, g32, ph, st, q_in, dq, q_out, s);
    }
    return cudaGetLastError();
}

cudaError_t launch_q_from_U_mx(const DevGeom& g, const Physics& ph, const V4* U, QHL* q,
                               cudaStream_t s) {
    k_q_from_U_mx<<<grid_nc(g, 256), 256, 0, s>>>(g, ph, U, q);
    return cudaGetLastError();
}

cudaError_t launch_dq_to_user_mx(const DevGeom& g, const D8f* src, V4* qx_user, V4* qy_user, cudaStream_t s) {
    k_gather_dq_mx<<<grid_nc(g, 256), 256, 0, s>>>(g, src, qx_user, qy_user);
    return cudaGetLastError();
}

}  // namespace lskum
