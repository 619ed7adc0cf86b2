// FP64 device kernels of the q-LSKUM hot path (sm_103a).
//
// Mapping: one thread per point (the sweeps: four, a component each), points in
// Hilbert-curve order (set-up), so a warp's points and their stencils are
// spatially close. Per-slot data
// (packed neighbour entry, half offsets, least-squares weights) is slot-major
// [slot][point]: consecutive threads read consecutive words (coalesced). The
// gathered per-point records are AoS: q (32 B) and (q_x, q_y) (64 B), so a
// neighbour gather is one or two full sectors.
//
// Per stage (Algorithm 2 re-fused):
//   ls_first  : q_x, q_y from Eq. 11 (full stencil), weights precomputed
//   ls_inner  : Jacobi sweep of Eq. 29 with dq~ of Eq. 28 (x inner_iters)
//   flux<k>   : residual of Eq. 12 -- per neighbour q~_j and q~_0 (Eq. 28),
//               their primitive states, the kinetic split fluxes G+-(q~)
//               along s and n (Eq. 27), accumulated with the precomputed
//               split-stencil weights (Eq. 24 over the Eq. 14 stencils) --
//               fused with the SSP-RK stage update, the wall condition, the
//               next stage's q-variables (Eq. 26), the stage-1 local time
//               step and the stage-1 partial sums of the residue.
//   residue   : fixed-order reduction of the partial sums (deterministic).
//
// The arithmetic is FP64 throughout, and the FP64 pipe, not HBM, bounds the flux
// kernel; for gamma = 1.4 lskum_kernels_pair.cu has the flux off that pipe.

#include <cmath>

#include "flux_fp64.cuh"

namespace lskum {

namespace {

// ----------------------------------------------------------- q-derivatives
//
// Four threads a (point, condition), one for each component of q: a gathered
// record is one coalesced read of its four threads where a thread of its own
// for each point made 32 scattered ones a load, and a small cloud fills four
// times the SMs: 5,120 points 15 -> 10 us the first-order sweep, 20 -> 14 an
// inner one; at 0.6M points and more both forms are bound by the FP64 pipe
// (190 and 285 us). A component's sum keeps the slot order.

// Stores a component's derivatives, with PAIRS also as float pairs (hi and lo each
// rounded to nearest) for the pair-form flux kernel.
template <bool PAIRS>
__device__ __forceinline__ void store_dq(V8* p, DQP* pairs, const int m, const double x, const double y) {
    p->x[m] = x;
    p->y[m] = y;
    if (PAIRS) {
        float4 v;
        v.x = __double2float_rn(x);
        v.y = __double2float_rn(x - double(v.x));
        v.z = __double2float_rn(y);
        v.w = __double2float_rn(y - double(v.z));
        pairs->c[m] = v;
    }
}

template <int BLOCK, bool PAIRS>
__global__ void __launch_bounds__(BLOCK) k_ls_first(const DevGeom g, const V4* __restrict__ q,
                                                    V8* __restrict__ dq, DQP* __restrict__ pairs) {
    const int64_t t = (int64_t(blockIdx.x) * BLOCK + threadIdx.x) / 4;  // (point, condition)
    const int m = threadIdx.x % 4;
    const int64_t d = t >> g.cshift;
    const uint32_t cc = uint32_t(t) & g.cmask;
    if (d >= g.n) return;
    const double* qm = reinterpret_cast<const double*>(q) + m;
    const double qi = qm[4 * t];
    double ax = 0.0, ay = 0.0;
    const int c = g.cnt[d];
#pragma unroll 4
    for (int k = 0; k < c; ++k) {
        const int64_t at = int64_t(k) * g.stride + d;
        const uint32_t j = g.nbr[at] & kIndexMask;
        const double wx = g.wx[at], wy = g.wy[at];
        const double e = qm[4 * sidx(g, j, cc)] - qi;
        ax += wx * e;
        ay += wy * e;
    }
    store_dq<PAIRS>(dq + t, pairs + t, m, ax, ay);
}

// One Jacobi sweep of Eq. 29. With dq~_j = (q_j - q_i) - (hdx_j (qx_j - qx_i)
// + hdy_j (qy_j - qy_i)) (Eq. 28, hdx = dx/2) the sweep is
//   q_x = sum_j wx_j (q_j - q_i) - [sum_j (a_j qx_j + b_j qy_j) - (A qx_i + B qy_i)]
// with a_j = wx_j hdx_j, b_j = wx_j hdy_j, A = sum_j a_j, B = sum_j b_j (and
// c, d, C, D from wy for q_y). The first sum is the first-order derivative of
// the same stage (dq_first), so a sweep gathers only the neighbours'
// derivatives: 4 FMAs per component and neighbour instead of 7 FP64
// operations. The bracket is ~1e-4 of q_x at 10M points and is formed to
// ~1e-12 of itself, so q_x keeps FP64 accuracy. `pairs` may be the memory of
// dq_first: a record is read by its own four threads only, before they write it.
template <int BLOCK, bool PAIRS>
__global__ void __launch_bounds__(BLOCK) k_ls_inner(const DevGeom g, const V8* dq_first,
                                                    const V8* __restrict__ din,
                                                    V8* __restrict__ dout, DQP* pairs) {
    const int64_t t = (int64_t(blockIdx.x) * BLOCK + threadIdx.x) / 4;  // (point, condition)
    const int m = threadIdx.x % 4;
    const int64_t d = t >> g.cshift;
    const uint32_t cc = uint32_t(t) & g.cmask;
    if (d >= g.n) return;
    double ax = 0.0, ay = 0.0;
    const int c = g.cnt[d];
#pragma unroll 4
    for (int k = 0; k < c; ++k) {
        const int64_t at = int64_t(k) * g.stride + d;
        const uint32_t j = g.nbr[at] & kIndexMask;
        const V4 p = g.lcoef[at];
        const V8* dj = din + sidx(g, j, cc);
        const double x = dj->x[m], y = dj->y[m];
        ax = fma(p.a, x, fma(p.b, y, ax));
        ay = fma(p.c, x, fma(p.d, y, ay));
    }
    const V4 S = g.lsum[d];
    const double xi = din[t].x[m], yi = din[t].y[m];
    const double fx = dq_first[t].x[m], fy = dq_first[t].y[m];
    if (PAIRS) __syncwarp(0xfu << (threadIdx.x & 28));
    store_dq<PAIRS>(dout + t, pairs + t, m, fx - (ax - fma(S.a, xi, S.b * yi)), fy - (ay - fma(S.c, xi, S.d * yi)));
}

// ------------------------------------------------------- flux residual + RK

// Every gamma but 1.4, and 1.4 on clouds of sizes that k_flux_pair does not take
// (HostLayout::held).
template <int MODE, int BLOCK, bool G14>
__global__ void __launch_bounds__(BLOCK) k_flux(const DevGeom g, const Physics ph,
                                                const DevState st, const V4* __restrict__ q_in,
                                                const V8* __restrict__ dq, V4* __restrict__ q_out) {
    const int64_t t = int64_t(blockIdx.x) * BLOCK + threadIdx.x;  // (point, condition)
    const int64_t d = t >> g.cshift;
    const uint32_t cc = uint32_t(t) & g.cmask;
    double r2 = 0.0;
    if (d < g.n) {
        const int8_t fl = g.flag[d];
        const bool fixed = ph.outer_fixed && fl == LSKUM_OUTER;
        double R[4] = {0.0, 0.0, 0.0, 0.0};
        if (!fixed) {
            double tx = 1.0, ty = 0.0, nx = 0.0, ny = 1.0;
            const bool local = fl != LSKUM_INTERIOR;
            if (local) {
                const double2 nn = g.nrm[d];
                nx = nn.x;
                ny = nn.y;
                tx = ny;
                ty = -nx;
            }
            const V4 qi = ld4(q_in + t);
            const V8 di = dq[t];
            const double qiv[4] = {qi.a, qi.b, qi.c, qi.d};
            const bool second = ph.order == 2;
            const int c = g.cnt[d];
            for (int k = 0; k < c; ++k) {
                const int64_t at = int64_t(k) * g.stride + d;
                const uint32_t e = g.nbr[at];
                const uint32_t j = e & kIndexMask;
                const uint32_t sc = (e >> kIndexBits) & 3u;
                const uint32_t nc = (e >> (kIndexBits + 2)) & 3u;
                const int64_t jt = sidx(g, j, cc);
                const V4 qj = ld4(q_in + jt);
                double tj[4] = {qj.a, qj.b, qj.c, qj.d};
                double t0[4] = {qiv[0], qiv[1], qiv[2], qiv[3]};
                // equal modified states give dG = 0 exactly (free-stream preservation);
                // the two inlined flux evaluations below need not round identically
                if (!modified_states(second, second ? g.hdx[at] : 0.0, second ? g.hdy[at] : 0.0,
                                     second ? dq[jt] : di, di, tj, t0))
                    continue;
                Prim wj = q_to_prim<G14>(tj[0], tj[1], tj[2], tj[3], ph.gm1_inv);
                Prim w0 = q_to_prim<G14>(t0[0], t0[1], t0[2], t0[3], ph.gm1_inv);
                if (local) {  // velocities into (s, n)
                    const double sj = wj.u * tx + wj.v * ty, nj = wj.u * nx + wj.v * ny;
                    const double s0 = w0.u * tx + w0.v * ty, n0 = w0.u * nx + w0.v * ny;
                    wj.u = sj; wj.v = nj;
                    w0.u = s0; w0.v = n0;
                }
                if (sc) {
                    const int64_t nmask = sc == 1u ? 0 : kSignBit;
                    double dg[4];
                    split_flux_diff(wj, w0, wj.u, wj.v, w0.u, w0.v, split_ab(wj, wj.u, nmask),
                                    split_ab(w0, w0.u, nmask), dg);
                    const double w = g.ws[at];
                    R[0] = fma(w, dg[0], R[0]);
                    R[1] = fma(w, dg[1], R[1]);
                    R[2] = fma(w, dg[2], R[2]);
                    R[3] = fma(w, dg[3], R[3]);
                }
                if (nc) {
                    const int64_t nmask = nc == 1u ? 0 : kSignBit;
                    double dg[4];
                    // along n: "a" = n-velocity, "b" = s-velocity
                    split_flux_diff(wj, w0, wj.v, wj.u, w0.v, w0.u, split_ab(wj, wj.v, nmask),
                                    split_ab(w0, w0.v, nmask), dg);
                    const double w = g.wn[at];
                    R[0] = fma(w, dg[0], R[0]);
                    R[1] = fma(w, dg[2], R[1]);  // s-momentum
                    R[2] = fma(w, dg[1], R[2]);  // n-momentum
                    R[3] = fma(w, dg[3], R[3]);
                }
            }
            if (local) {  // momentum back to the global frame
                const double rs = R[1], rn = R[2];
                R[1] = rs * tx + rn * nx;
                R[2] = rs * ty + rn * ny;
            }
        }
        r2 = stage_epilogue<MODE, G14>(g, ph, st, t, d, fl, fixed, R, q_out);
    }
    if (MODE == 1) {
        if (g.cshift == 0) {  // one condition: fused block partial sums
            const double s = block_sum<BLOCK>(r2);
            if (threadIdx.x == 0) st.partials[blockIdx.x] = s;
        } else if (d < g.n) {  // several: per (point, condition), reduced per condition
            st.r2[t] = r2;
        }
    }
}

// ------------------------------------------------ split-flux kernels (ablation)
// The paper's kernel splitting (Section 5, the four split-flux kernels Gx+,
// Gx-, Gy+, Gy-): one kernel per split-flux derivative dGs+/ds, dGs-/ds,
// dGn+/dn, dGn-/dn, each adding its stencil's contribution to the residual
// (local frame) in Racc, then one kernel for the stage update. An ablation of
// the fused kernel: a neighbour's two q~ -> primitive maps are computed once
// per stencil it belongs to (twice), and Racc makes four extra round trips.
template <int PART, int BLOCK, bool G14>
__global__ void __launch_bounds__(BLOCK) k_flux_part(const DevGeom g, const Physics ph,
                                                     const V4* __restrict__ q_in,
                                                     const V8* __restrict__ dq,
                                                     V4* __restrict__ Racc) {
    const int64_t t = int64_t(blockIdx.x) * BLOCK + threadIdx.x;
    const int64_t d = t >> g.cshift;
    const uint32_t cc = uint32_t(t) & g.cmask;
    if (d >= g.n) return;
    const int8_t fl = g.flag[d];
    double R[4] = {0.0, 0.0, 0.0, 0.0};
    if (!(ph.outer_fixed && fl == LSKUM_OUTER)) {
        double tx = 1.0, ty = 0.0, nx = 0.0, ny = 1.0;
        const bool local = fl != LSKUM_INTERIOR;
        if (local) {
            const double2 nn = g.nrm[d];
            nx = nn.x;
            ny = nn.y;
            tx = ny;
            ty = -nx;
        }
        const V4 qi = ld4(q_in + t);
        const V8 di = dq[t];
        const double qiv[4] = {qi.a, qi.b, qi.c, qi.d};
        const bool second = ph.order == 2;
        const uint32_t want = (PART % 2 == 0) ? 1u : 2u;
        const int64_t nmask = (PART % 2 == 0) ? 0 : kSignBit;
        const int c = g.cnt[d];
        for (int k = 0; k < c; ++k) {
            const int64_t at = int64_t(k) * g.stride + d;
            const uint32_t e = g.nbr[at];
            const uint32_t code = PART < 2 ? ((e >> kIndexBits) & 3u) : ((e >> (kIndexBits + 2)) & 3u);
            if (code != want) continue;
            const uint32_t j = e & kIndexMask;
            const int64_t jt = sidx(g, j, cc);
            const V4 qj = ld4(q_in + jt);
            double tj[4] = {qj.a, qj.b, qj.c, qj.d};
            double t0[4] = {qiv[0], qiv[1], qiv[2], qiv[3]};
            if (!modified_states(second, second ? g.hdx[at] : 0.0, second ? g.hdy[at] : 0.0,
                                 second ? dq[jt] : di, di, tj, t0))
                continue;
            Prim wj = q_to_prim<G14>(tj[0], tj[1], tj[2], tj[3], ph.gm1_inv);
            Prim w0 = q_to_prim<G14>(t0[0], t0[1], t0[2], t0[3], ph.gm1_inv);
            if (local) {
                const double sj = wj.u * tx + wj.v * ty, nj = wj.u * nx + wj.v * ny;
                const double s0 = w0.u * tx + w0.v * ty, n0 = w0.u * nx + w0.v * ny;
                wj.u = sj; wj.v = nj;
                w0.u = s0; w0.v = n0;
            }
            double dg[4];
            if (PART < 2) {
                split_flux_diff(wj, w0, wj.u, wj.v, w0.u, w0.v, split_ab(wj, wj.u, nmask),
                                split_ab(w0, w0.u, nmask), dg);
                const double w = g.ws[at];
                R[0] = fma(w, dg[0], R[0]);
                R[1] = fma(w, dg[1], R[1]);
                R[2] = fma(w, dg[2], R[2]);
                R[3] = fma(w, dg[3], R[3]);
            } else {
                split_flux_diff(wj, w0, wj.v, wj.u, w0.v, w0.u, split_ab(wj, wj.v, nmask),
                                split_ab(w0, w0.v, nmask), dg);
                const double w = g.wn[at];
                R[0] = fma(w, dg[0], R[0]);
                R[1] = fma(w, dg[2], R[1]);
                R[2] = fma(w, dg[1], R[2]);
                R[3] = fma(w, dg[3], R[3]);
            }
        }
    }
    if (PART == 0) {
        Racc[t] = V4{R[0], R[1], R[2], R[3]};
    } else {
        V4 a = Racc[t];
        a.a += R[0];
        a.b += R[1];
        a.c += R[2];
        a.d += R[3];
        Racc[t] = a;
    }
}

template <int MODE, int BLOCK, bool G14>
__global__ void __launch_bounds__(BLOCK) k_stage_split(const DevGeom g, const Physics ph,
                                                       const DevState st, const V4* __restrict__ Racc,
                                                       V4* __restrict__ q_out) {
    const int64_t t = int64_t(blockIdx.x) * BLOCK + threadIdx.x;
    const int64_t d = t >> g.cshift;
    double r2 = 0.0;
    if (d < g.n) {
        const int8_t fl = g.flag[d];
        const bool fixed = ph.outer_fixed && fl == LSKUM_OUTER;
        double R[4] = {0.0, 0.0, 0.0, 0.0};
        if (!fixed) {
            const V4 a = Racc[t];
            R[0] = a.a;
            R[1] = a.b;
            R[2] = a.c;
            R[3] = a.d;
            if (fl != LSKUM_INTERIOR) {
                const double2 nn = g.nrm[d];
                const double tx = nn.y, ty = -nn.x;
                const double rs = R[1], rn = R[2];
                R[1] = rs * tx + rn * nn.x;
                R[2] = rs * ty + rn * nn.y;
            }
        }
        r2 = stage_epilogue<MODE, G14>(g, ph, st, t, d, fl, fixed, R, q_out);
    }
    if (MODE == 1) {
        if (g.cshift == 0) {
            const double s = block_sum<BLOCK>(r2);
            if (threadIdx.x == 0) st.partials[blockIdx.x] = s;
        } else if (d < g.n) {
            st.r2[t] = r2;
        }
    }
}

// Residue = sqrt(sum of the per-block partials) / N, summed in block order by
// one block (deterministic), appended to the history ring buffer.
__global__ void __launch_bounds__(kReduceBlock) k_residue(const DevState st, int nblocks,
                                                          int64_t n) {
    double s = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += kReduceBlock) s += st.partials[b];
    s = block_sum<kReduceBlock>(s);
    if (threadIdx.x == 0) {
        const unsigned long long it = *st.iter_counter;
        const double r = sqrt(s) / double(n);
        st.res_hist[it % (unsigned long long)st.res_cap] = r;
        *st.iter_counter = it + 1;
        if (!isfinite(r)) atomicOr(st.status, 1);
    }
}

// ------------------------------------------------------------ state I/O

__global__ void k_set_uniform(const DevGeom g, const Physics ph, const V4* __restrict__ Wc,
                              V4* U, V4* q) {
    const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t d = t >> g.cshift;
    if (d >= g.n) return;
    const V4 W = Wc[uint32_t(t) & g.cmask];
    V4 u;
    u.a = W.a;
    u.b = W.a * W.b;
    u.c = W.a * W.c;
    u.d = W.d * ph.gm1_inv + 0.5 * W.a * (W.b * W.b + W.c * W.c);
    U[t] = u;
    // q straight from the given primitive state (no round trip through U)
    V4 qq;
    prim_to_q(W.a, W.b, W.c, W.d, ph, qq);
    q[t] = qq;
}

// W_user is condition-major in the caller's point order: [condition][point].
__global__ void k_set_prim(const DevGeom g, const Physics ph, const V4* __restrict__ W_user,
                           V4* U, V4* q, int* status) {
    const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t d = t >> g.cshift;
    if (d >= g.n) return;
    const int64_t cc = int64_t(uint32_t(t) & g.cmask);
    const V4 W = W_user[cc * g.n + g.dev_to_user[d]];
    if (!physical(W.a, W.b, W.c, W.d)) atomicOr(status, 2);
    V4 u;
    u.a = W.a;
    u.b = W.a * W.b;
    u.c = W.a * W.c;
    u.d = W.d * ph.gm1_inv + 0.5 * W.a * (W.b * W.b + W.c * W.c);
    U[t] = u;
    // q straight from the given primitive state (no round trip through U)
    V4 qq;
    prim_to_q(W.a, W.b, W.c, W.d, ph, qq);
    q[t] = qq;
}

__global__ void k_get_prim(const DevGeom g, const Physics ph, const V4* __restrict__ U,
                           V4* __restrict__ W_user) {
    const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t d = t >> g.cshift;
    if (d >= g.n) return;
    const int64_t cc = int64_t(uint32_t(t) & g.cmask);
    const V4 u = U[t];
    const double rho = u.a, uu = u.b / rho, vv = u.c / rho;
    const double p = ph.gm1 * (u.d - 0.5 * rho * (uu * uu + vv * vv));
    W_user[cc * g.n + g.dev_to_user[d]] = V4{rho, uu, vv, p};
}

__global__ void k_q_from_U(const DevGeom g, const Physics ph, const V4* __restrict__ U,
                           V4* __restrict__ q) {
    const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if ((t >> g.cshift) >= g.n) return;
    V4 qq;
    double rho, uu, vv, p;
    if (fabs(ph.gm1_inv - 2.5) < 1e-12)
        cons_to_q64<true>(U[t], ph, qq, rho, uu, vv, p);
    else
        cons_to_q64<false>(U[t], ph, qq, rho, uu, vv, p);
    q[t] = qq;
}

__global__ void k_gather(const DevGeom g, const V4* __restrict__ src, V4* __restrict__ dst) {
    const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t d = t >> g.cshift;
    if (d >= g.n) return;
    const int64_t cc = int64_t(uint32_t(t) & g.cmask);
    dst[cc * g.n + g.dev_to_user[d]] = src[t];
}

// Derivatives in the caller's order, q_x and q_y apart (n x 4 each a condition).
__global__ void k_gather_dq(const DevGeom g, const V8* __restrict__ src, V4* __restrict__ qx,
                            V4* __restrict__ qy) {
    const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t d = t >> g.cshift;
    if (d >= g.n) return;
    const int64_t at = int64_t(uint32_t(t) & g.cmask) * g.n + g.dev_to_user[d];
    const V8 s = src[t];
    qx[at] = V4{s.x[0], s.x[1], s.x[2], s.x[3]};
    qy[at] = V4{s.y[0], s.y[1], s.y[2], s.y[3]};
}

// Residue per condition (C > 1), phase 1: block b reduces a contiguous range
// of points for every condition into cpartials[b][c] (rows in a fixed order).
__global__ void __launch_bounds__(512) k_residue_cond_p1(const DevGeom g, const DevState st) {
    __shared__ double part[16][33];
    const int64_t C = int64_t(1) << g.cshift;
    const int64_t rows_per_block = (g.n + gridDim.x - 1) / gridDim.x;
    const int64_t r0 = int64_t(blockIdx.x) * rows_per_block;
    const int64_t r1 = min(g.n, r0 + rows_per_block);
    for (int64_t c0 = 0; c0 < C; c0 += 32) {
        const int64_t c = c0 + threadIdx.x;
        double s = 0.0;
        if (c < C)
            for (int64_t r = r0 + threadIdx.y; r < r1; r += 16) s += st.r2[(r << g.cshift) | c];
        part[threadIdx.y][threadIdx.x] = s;
        __syncthreads();
        if (threadIdx.y == 0 && c < C) {
            double tot = 0.0;
            for (int k = 0; k < 16; ++k) tot += part[k][threadIdx.x];
            st.cpartials[int64_t(blockIdx.x) * C + c] = tot;
        }
        __syncthreads();
    }
}

// Phase 2 (one block): sum the block partials of each condition, append
// sqrt(sum)/N per condition to the history. The block's threads share out the
// partials of a condition (every kCondSumThreads / C-th each, then their sums in
// order): a chain of loads a condition took 14 us longer for 64 of them.
constexpr int kCondSumThreads = 1024;  // at least the conditions

__global__ void __launch_bounds__(kCondSumThreads) k_residue_cond_p2(const DevGeom g, const DevState st,
                                                                     int nblocks) {
    __shared__ double part[kCondSumThreads];
    const int C = 1 << g.cshift, groups = kCondSumThreads >> g.cshift;
    const unsigned long long it = *st.iter_counter;
    const int c = threadIdx.x & (C - 1);
    double s = 0.0;
#pragma unroll 8
    for (int b = threadIdx.x >> g.cshift; b < nblocks; b += groups) s += st.cpartials[int64_t(b) * C + c];
    part[threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.x < C) {
        s = 0.0;
        for (int k = 0; k < groups; ++k) s += part[(k << g.cshift) + c];
        const double r = sqrt(s) / double(g.n);
        st.res_hist[int64_t(it % (unsigned long long)(st.res_cap / C)) * C + c] = r;
        if (!isfinite(r)) atomicOr(st.status, 1);
    }
    if (threadIdx.x == 0) *st.iter_counter = it + 1;
}

// Pressure force on the wall loops: F = -sum (p_i - p_inf) n_i ds_i; one
// block per condition.
__global__ void __launch_bounds__(kReduceBlock) k_forces(const DevGeom g, const Physics ph,
                                                         const DevState st) {
    const uint32_t cc = blockIdx.x;
    double fx = 0.0, fy = 0.0;
    for (int64_t k = threadIdx.x; k < g.n_wall; k += kReduceBlock) {
        const int32_t d = g.wall_id[k];
        const V4 u = st.U[sidx(g, d, cc)];
        const double rho = u.a, uu = u.b / rho, vv = u.c / rho;
        const double p = ph.gm1 * (u.d - 0.5 * rho * (uu * uu + vv * vv));
        const double2 nds = g.wall_nds[k];
        fx -= (p - ph.p_inf) * nds.x;
        fy -= (p - ph.p_inf) * nds.y;
    }
    fx = block_sum<kReduceBlock>(fx);
    __syncthreads();
    fy = block_sum<kReduceBlock>(fy);
    if (threadIdx.x == 0) {
        st.force_out[2 * cc] = fx;
        st.force_out[2 * cc + 1] = fy;
    }
}

inline unsigned grid_for(int64_t n, int block) { return unsigned((n + block - 1) / block); }
// threads over all (point, condition) pairs
inline unsigned grid_nc(const DevGeom& g, int block) { return grid_for(g.n << g.cshift, block); }

}  // namespace

cudaError_t launch_ls_first(const DevGeom& g, const V4* q, V8* dq, DQP* pairs, int block,
                            cudaStream_t s) {
    const unsigned grid = grid_for((g.n << g.cshift) * 4, block);
    if (block == 256) {
        if (pairs) k_ls_first<256, true><<<grid, 256, 0, s>>>(g, q, dq, pairs);
        else k_ls_first<256, false><<<grid, 256, 0, s>>>(g, q, dq, nullptr);
    } else {
        if (pairs) k_ls_first<kDefaultBlock, true><<<grid, kDefaultBlock, 0, s>>>(g, q, dq, pairs);
        else k_ls_first<kDefaultBlock, false><<<grid, kDefaultBlock, 0, s>>>(g, q, dq, nullptr);
    }
    return cudaGetLastError();
}

cudaError_t launch_ls_inner(const DevGeom& g, const V8* dq_first, const V8* din, V8* dout, DQP* pairs,
                            int block, cudaStream_t s) {
    const unsigned grid = grid_for((g.n << g.cshift) * 4, block);
    if (block == 256) {
        if (pairs) k_ls_inner<256, true><<<grid, 256, 0, s>>>(g, dq_first, din, dout, pairs);
        else k_ls_inner<256, false><<<grid, 256, 0, s>>>(g, dq_first, din, dout, nullptr);
    } else {
        if (pairs) k_ls_inner<kDefaultBlock, true><<<grid, kDefaultBlock, 0, s>>>(g, dq_first, din, dout, pairs);
        else k_ls_inner<kDefaultBlock, false><<<grid, kDefaultBlock, 0, s>>>(g, dq_first, din, dout, nullptr);
    }
    return cudaGetLastError();
}

template <int BLOCK, bool G14>
static void flux_dispatch(int mode, const DevGeom& g, const Physics& ph, const DevState& st,
                          const V4* q_in, const V8* dq, V4* q_out, cudaStream_t s) {
    const unsigned grid = grid_nc(g, BLOCK);
    switch (mode) {
        case 0: k_flux<0, BLOCK, G14><<<grid, BLOCK, 0, s>>>(g, ph, st, q_in, dq, q_out); break;
        case 1: k_flux<1, BLOCK, G14><<<grid, BLOCK, 0, s>>>(g, ph, st, q_in, dq, q_out); break;
        case 2: k_flux<2, BLOCK, G14><<<grid, BLOCK, 0, s>>>(g, ph, st, q_in, dq, q_out); break;
        case 3: k_flux<3, BLOCK, G14><<<grid, BLOCK, 0, s>>>(g, ph, st, q_in, dq, q_out); break;
        default: k_flux<4, BLOCK, G14><<<grid, BLOCK, 0, s>>>(g, ph, st, q_in, dq, q_out); break;
    }
}

cudaError_t launch_flux(int mode, const DevGeom& g, const Physics& ph, const DevState& st,
                        const V4* q_in, const V8* dq, V4* q_out, int block, cudaStream_t s) {
    // gamma = 1.4: log-free density (see q_to_prim)
    const bool g14 = fabs(ph.gm1_inv - 2.5) < 1e-12;
    if (block == 256) {
        if (g14) flux_dispatch<256, true>(mode, g, ph, st, q_in, dq, q_out, s);
        else flux_dispatch<256, false>(mode, g, ph, st, q_in, dq, q_out, s);
    } else {
        if (g14) flux_dispatch<kDefaultBlock, true>(mode, g, ph, st, q_in, dq, q_out, s);
        else flux_dispatch<kDefaultBlock, false>(mode, g, ph, st, q_in, dq, q_out, s);
    }
    return cudaGetLastError();
}

template <int BLOCK, bool G14>
static void flux_split_dispatch(int mode, const DevGeom& g, const Physics& ph, const DevState& st,
                                const V4* q_in, const V8* dq, V4* q_out, cudaStream_t s) {
    const unsigned grid = grid_nc(g, BLOCK);
    V4* Racc = st.R;  // accumulator (R is an output only of the evaluation mode)
    k_flux_part<0, BLOCK, G14><<<grid, BLOCK, 0, s>>>(g, ph, q_in, dq, Racc);
    k_flux_part<1, BLOCK, G14><<<grid, BLOCK, 0, s>>>(g, ph, q_in, dq, Racc);
    k_flux_part<2, BLOCK, G14><<<grid, BLOCK, 0, s>>>(g, ph, q_in, dq, Racc);
    k_flux_part<3, BLOCK, G14><<<grid, BLOCK, 0, s>>>(g, ph, q_in, dq, Racc);
    switch (mode) {
        case 0: k_stage_split<0, BLOCK, G14><<<grid, BLOCK, 0, s>>>(g, ph, st, Racc, q_out); break;
        case 1: k_stage_split<1, BLOCK, G14><<<grid, BLOCK, 0, s>>>(g, ph, st, Racc, q_out); break;
        case 2: k_stage_split<2, BLOCK, G14><<<grid, BLOCK, 0, s>>>(g, ph, st, Racc, q_out); break;
        case 3: k_stage_split<3, BLOCK, G14><<<grid, BLOCK, 0, s>>>(g, ph, st, Racc, q_out); break;
        default: k_stage_split<4, BLOCK, G14><<<grid, BLOCK, 0, s>>>(g, ph, st, Racc, q_out); break;
    }
}

cudaError_t launch_flux_split(int mode, const DevGeom& g, const Physics& ph, const DevState& st,
                              const V4* q_in, const V8* dq, V4* q_out, int block, cudaStream_t s) {
    const bool g14 = fabs(ph.gm1_inv - 2.5) < 1e-12;
    if (block == 256) {
        if (g14) flux_split_dispatch<256, true>(mode, g, ph, st, q_in, dq, q_out, s);
        else flux_split_dispatch<256, false>(mode, g, ph, st, q_in, dq, q_out, s);
    } else {
        if (g14) flux_split_dispatch<kDefaultBlock, true>(mode, g, ph, st, q_in, dq, q_out, s);
        else flux_split_dispatch<kDefaultBlock, false>(mode, g, ph, st, q_in, dq, q_out, s);
    }
    return cudaGetLastError();
}

cudaError_t launch_residue(const DevState& st, int nblocks, int64_t n, cudaStream_t s) {
    k_residue<<<1, kReduceBlock, 0, s>>>(st, nblocks, n);
    return cudaGetLastError();
}

cudaError_t launch_residue_cond(const DevGeom& g, const DevState& st, cudaStream_t s) {
    k_residue_cond_p1<<<kCondReduceBlocks, dim3(32, 16), 0, s>>>(g, st);
    k_residue_cond_p2<<<1, kCondSumThreads, 0, s>>>(g, st, kCondReduceBlocks);
    return cudaGetLastError();
}

cudaError_t launch_set_uniform(const DevGeom& g, const Physics& ph, const V4* W_cond, V4* U, V4* q,
                               cudaStream_t s) {
    k_set_uniform<<<grid_nc(g, 256), 256, 0, s>>>(g, ph, W_cond, U, q);
    return cudaGetLastError();
}

cudaError_t launch_set_prim(const DevGeom& g, const Physics& ph, const V4* W_user, V4* U, V4* q,
                            int* status, cudaStream_t s) {
    k_set_prim<<<grid_nc(g, 256), 256, 0, s>>>(g, ph, W_user, U, q, status);
    return cudaGetLastError();
}

cudaError_t launch_get_prim(const DevGeom& g, const Physics& ph, const V4* U, V4* W_user,
                            cudaStream_t s) {
    k_get_prim<<<grid_nc(g, 256), 256, 0, s>>>(g, ph, U, W_user);
    return cudaGetLastError();
}

cudaError_t launch_q_from_U(const DevGeom& g, const Physics& ph, const V4* U, V4* q, cudaStream_t s) {
    k_q_from_U<<<grid_nc(g, 256), 256, 0, s>>>(g, ph, U, q);
    return cudaGetLastError();
}

cudaError_t launch_gather_v4(const DevGeom& g, const V4* src, V4* dst, cudaStream_t s) {
    k_gather<<<grid_nc(g, 256), 256, 0, s>>>(g, src, dst);
    return cudaGetLastError();
}

cudaError_t launch_gather_dq(const DevGeom& g, const V8* src, V4* qx, V4* qy, cudaStream_t s) {
    k_gather_dq<<<grid_nc(g, 256), 256, 0, s>>>(g, src, qx, qy);
    return cudaGetLastError();
}

cudaError_t launch_forces(const DevGeom& g, const Physics& ph, const DevState& st, cudaStream_t s) {
    k_forces<<<unsigned(1u << g.cshift), kReduceBlock, 0, s>>>(g, ph, st);
    return cudaGetLastError();
}

}  // namespace lskum
