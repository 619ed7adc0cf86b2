// The FP64 path's flux kernel for gamma = 1.4, its per-neighbour work in float
// pairs (flux_pair.cuh).
//
// What bounds it: instruction issue (66 % of the slots at 2.5M points). A
// split-flux difference costs 225 FP64 instructions per neighbour entry, and the
// FP64 pipe issues two per clock and SM where the FP32 pipes issue 128. The pair
// form takes about 1,850 FP32 instructions: at 2.5M points 2.88 ms a launch
// instead of 14.75, at 0.6M 0.91 instead of 3.58, at 5,120 0.050 instead of
// 0.148. Entries that are not the pair form's (large steps: a quarter at 0.6M,
// most at 5,120) are noted in a bit mask and evaluated after the loop from the
// doubles, in 64-bit fixed point (flux_fixed.cuh), a warp's entries spread evenly
// over its lanes; the stage update, the next stage's q-variables and the residue
// stay FP64.

#include "flux_fixed.cuh"
#include "flux_fp64.cuh"
#include "flux_pair.cuh"
#include "pair_convert.cuh"

namespace lskum {

namespace {

constexpr int kClasses = 4;
// Up to this many (point, condition) pairs four threads share a point. One
// thread a point leaves SMs idle on a small cloud (5,120 points: 40 blocks),
// and blocks of 128 points whose entries all have large steps are too large a
// unit of work to balance; beyond it the four-fold set-up of a point costs more.
// Microseconds a launch, one thread / four: 5,120 points 141 / 50, 46,080
// 208 / 151, 150,598 384 / 359, 220,080 457 / 478, 600,138 909 / 1,051.
constexpr int64_t kSplitPairs = 3 << 16;

// The double of which h + l is the pair and r what it exceeds them by, in units of
// its last place (lskum_setup.cpp); h and l are finite.
__device__ __forceinline__ double whole(const float h, const float l, const signed char r) {
    return bitsd(dbits(widen(h) + widen(l)) + r);
}

__device__ __forceinline__ Pf dx_of(const float4& c) { return Pf{c.x, c.y}; }
__device__ __forceinline__ Pf dy_of(const float4& c) { return Pf{c.z, c.w}; }

// The two states' split fluxes by primitive variables in FP64, for states that
// the fixed-point form does not take: |S| or ln(rho beta^2.5) out of its tables.
__device__ __noinline__ void general_diff(const double* tj, const double* t0, const bool local,
                                          const double2 nn, const uint32_t sc, const uint32_t nc,
                                          const double gm1_inv, double* ds, double* dn) {
    Prim wj = q_to_prim<true>(tj[0], tj[1], tj[2], tj[3], gm1_inv);
    Prim w0 = q_to_prim<true>(t0[0], t0[1], t0[2], t0[3], gm1_inv);
    if (local) {
        const double nx = nn.x, ny = nn.y, tx = ny, ty = -nx;
        const double sj = wj.u * tx + wj.v * ty, nj = wj.u * nx + wj.v * ny;
        const double s0 = w0.u * tx + w0.v * ty, n0 = w0.u * nx + w0.v * ny;
        wj.u = sj; wj.v = nj;
        w0.u = s0; w0.v = n0;
    }
    const int64_t sm = sc == 2u ? kSignBit : 0, nm = nc == 2u ? kSignBit : 0;
    split_flux_diff(wj, w0, wj.u, wj.v, w0.u, w0.v, split_ab(wj, wj.u, sm), split_ab(w0, w0.u, sm), ds);
    split_flux_diff(wj, w0, wj.v, wj.u, w0.v, w0.u, split_ab(wj, wj.v, nm), split_ab(w0, w0.v, nm), dn);
}

// ws dGs + wn dGn of entry k of point d to FP64's accuracy, in the point's frame:
// what k_flux adds for that entry. 48 FP64 instructions and some 1,700 on the
// integer pipe (flux_fixed.cuh), where k_flux's formulas take 230 FP64 ones.
__device__ __forceinline__ void entry_fp64(const DevGeom& g, const DevGeomPair& gp, const Physics& ph,
                                           const V4* __restrict__ q_in, const V8* __restrict__ dq,
                                           const int64_t t, const int k, double c[4]) {
    const int64_t d = t >> g.cshift;
    const int64_t at = int64_t(k) * g.stride + d;
    const uint32_t e = g.nbr[at];
    const int64_t jt = sidx(g, e & kIndexMask, uint32_t(t) & g.cmask);
    const V4 qi = ld4(q_in + t), qj = ld4(q_in + jt);
    double tj[4] = {qj.a, qj.b, qj.c, qj.d};
    double t0[4] = {qi.a, qi.b, qi.c, qi.d};
    c[0] = c[1] = c[2] = c[3] = 0.0;
    const char4 rest = gp.rest[at];
    double hx = 0.0, hy = 0.0;
    const bool second = ph.order == 2;
    if (second) {
        const float4 hp = gp.half[at];
        hx = whole(hp.x, hp.y, rest.x);
        hy = whole(hp.z, hp.w, rest.y);
    }
    if (!modified_states(second, hx, hy, dq[second ? jt : t], dq[t], tj, t0)) return;
    const uint32_t sc = e >> kIndexBits & 3u, nc = e >> (kIndexBits + 2) & 3u;
    const bool local = g.flag[d] != LSKUM_INTERIOR;
    const double2 nn = local ? g.nrm[d] : make_double2(0.0, 1.0);
    double ds[4], dn[4];
    if (!fixed_diff(tj, t0, local, nn.x, nn.y, sc == 2u, nc == 2u, ds, dn)) {
        const double gj[4] = {tj[0], tj[1], tj[2], tj[3]}, g0[4] = {t0[0], t0[1], t0[2], t0[3]};
        double rs[4], rn[4];
        general_diff(gj, g0, local, nn, sc, nc, ph.gm1_inv, rs, rn);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            ds[m] = sc ? rs[m] : 0.0;
            dn[m] = nc ? rn[m] : 0.0;
        }
    }
    const float4 wp = gp.weight[at];
    // an entry outside a stencil has weight 0 there
    const double ws = whole(wp.x, wp.y, rest.z), wn = whole(wp.z, wp.w, rest.w);
    c[0] = fma(wn, dn[0], ws * ds[0]);
    c[1] = fma(wn, dn[2], ws * ds[1]);
    c[2] = fma(wn, dn[1], ws * ds[2]);
    c[3] = fma(wn, dn[3], ws * ds[3]);
}

// The pair-form part of one point's entries first, first + kClasses, ...: adds to
// acc; returns the entries left over as a bit mask.
struct PairPoint {
    V4 q;
    DQP dq;
    Pf qp[4], nx, ny;
    bool local;
};

__device__ __forceinline__ uint32_t entries_pair(const DevGeom& g, const DevGeomPair& gp, const bool second,
                                                 const V4* __restrict__ q_in, const DQP* __restrict__ dq,
                                                 const int64_t d, const uint32_t cc, const PairPoint& P,
                                                 const int first, const int c, Pf acc[4]) {
    uint32_t left = 0;
    // for the first look at a step: 1/q4 and 1/(2 sqrt(beta)), floats; no step is
    // small enough at a point with |S| well beyond the pair form's
    const float iq4 = __fdividef(1.0f, P.qp[3].h), isq = rsqrtf(-2.0f * P.qp[3].h);
    const float s1 = isq * P.qp[1].h, s2 = isq * P.qp[2].h;
    const float look = s1 * s1 + s2 * s2 <= 1.1f * kPairMaxS * kPairMaxS ? 1.25f * kPairStep : -1.0f;
    for (int k = first; k < c; k += kClasses) {
        const int64_t at = int64_t(k) * g.stride + d;
        const uint32_t e = g.nbr[at];
        const int64_t jt = sidx(g, e & kIndexMask, cc);
        const V4 qj = ld4(q_in + jt);
        Pf b[4] = {P.qp[0], P.qp[1], P.qp[2], P.qp[3]};
        Pf dd[4] = {split_pair(qj.a - P.q.a), split_pair(qj.b - P.q.b), split_pair(qj.c - P.q.c),
                    split_pair(qj.d - P.q.d)};
        float4 hp = make_float4(0.f, 0.f, 0.f, 0.f);
        DQP dj = P.dq;
        float f0 = dd[0].h, f1 = dd[1].h, f2 = dd[2].h, f3 = dd[3].h;
        if (second) {
            hp = gp.half[at];
            dj = dq[jt];
            f0 -= hp.x * (dj.c[0].x - P.dq.c[0].x) + hp.z * (dj.c[0].z - P.dq.c[0].z);
            f1 -= hp.x * (dj.c[1].x - P.dq.c[1].x) + hp.z * (dj.c[1].z - P.dq.c[1].z);
            f2 -= hp.x * (dj.c[2].x - P.dq.c[2].x) + hp.z * (dj.c[2].z - P.dq.c[2].z);
            f3 -= hp.x * (dj.c[3].x - P.dq.c[3].x) + hp.z * (dj.c[3].z - P.dq.c[3].z);
        }
        // a step well over the limits is not taken through the pair arithmetic
        // to find that out: d(ln beta), dS and d(q1 + |S|^2) in floats
        const float fe = f3 * iq4, g1 = f1 - 0.5f * fe * P.qp[1].h, g2 = f2 - 0.5f * fe * P.qp[2].h;
        const float fw = f0 - iq4 * (P.qp[1].h * g1 + P.qp[2].h * g2);
        if (!(fmaxf(fmaxf(fabsf(fe), fabsf(fw) * (kPairStep / kPairStepW)),
                    isq * fmaxf(fabsf(g1), fabsf(g2))) <= look)) {
            left |= 1u << k;
            continue;
        }
        if (second) {  // q~ of Eq. 28
            const Pf hx = {hp.x, hp.y}, hy = {hp.z, hp.w};
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const Pf c0 = add(mul(hx, dx_of(P.dq.c[m])), mul(hy, dy_of(P.dq.c[m])));
                const Pf cj = add(mul(hx, dx_of(dj.c[m])), mul(hy, dy_of(dj.c[m])));
                b[m] = sub(b[m], c0);
                dd[m] = sub(dd[m], sub(cj, c0));
            }
        }
        PairState w;
        if (!pair_state(b, dd, w)) {
            left |= 1u << k;
            continue;
        }
        if (P.local) {  // into (s, n): s = (n_y, -n_x)
            const Pf sm = sub(mul(w.Sxm, P.ny), mul(w.Sym, P.nx)), nm = add(mul(w.Sxm, P.nx), mul(w.Sym, P.ny));
            const Pf sd = sub(mul(w.dSx, P.ny), mul(w.dSy, P.nx)), nd = add(mul(w.dSx, P.nx), mul(w.dSy, P.ny));
            w.Sxm = sm; w.Sym = nm;
            w.dSx = sd; w.dSy = nd;
        }
        // an entry outside a stencil has weight 0 there
        const float4 wp = gp.weight[at];
        Pf dG[4];
        float sg = ((e >> kIndexBits) & 3u) == 2u ? -1.f : 1.f;
        Pf wt = {wp.x, wp.y}, wf = scale(wt, sg);
        split_diff(w, scale(w.Sxm, sg), scale(w.dSx, sg), w.Sym, w.dSy, dG);
        acc[0] = add(acc[0], mul(wf, dG[0]));
        acc[1] = add(acc[1], mul(wt, dG[1]));
        acc[2] = add(acc[2], mul(wf, dG[2]));
        acc[3] = add(acc[3], mul(wf, dG[3]));
        sg = ((e >> (kIndexBits + 2)) & 3u) == 2u ? -1.f : 1.f;
        wt = {wp.z, wp.w};
        wf = scale(wt, sg);
        split_diff(w, scale(w.Sym, sg), scale(w.dSy, sg), w.Sxm, w.dSx, dG);
        acc[0] = add(acc[0], mul(wf, dG[0]));
        acc[1] = add(acc[1], mul(wf, dG[2]));
        acc[2] = add(acc[2], mul(wt, dG[1]));
        acc[3] = add(acc[3], mul(wf, dG[3]));
    }
    return left;
}

// A point's entries fall into kClasses classes (k mod kClasses), each summed in
// slot order, the classes' sums then added in order: LANES = 1 thread of a point
// takes them one after the other, LANES = kClasses threads one each, to the
// same bits.
template <int MODE, int BLOCK, int LANES>
__global__ void __launch_bounds__(BLOCK) k_flux_pair(const DevGeom g, const DevGeomPair gp,
                                                     const Physics ph, const DevState st,
                                                     const V4* __restrict__ q_in,
                                                     const V8* __restrict__ dq,
                                                     const DQP* __restrict__ dqp,
                                                     V4* __restrict__ q_out) {
    static_assert(LANES == 1 || LANES == kClasses, "a thread takes all classes of a point or one");
    // per warp: the large-step entries of one pass of its lanes (owner lane, slot) and their results
    __shared__ uint16_t s_item[BLOCK / 32][32];
    __shared__ double s_res[BLOCK / 32][4][33];
    __shared__ double s_R[BLOCK / LANES][4];  // a point's sums
    const int64_t t = (int64_t(blockIdx.x) * BLOCK + threadIdx.x) / LANES;  // (point, condition)
    const int64_t d = t >> g.cshift;
    const uint32_t cc = uint32_t(t) & g.cmask;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int part = LANES == 1 ? 0 : lane % LANES;
    const bool live = d < g.n;
    const int8_t fl = live ? g.flag[d] : int8_t(LSKUM_INTERIOR);
    const bool fixed = ph.outer_fixed && fl == LSKUM_OUTER;
    const bool local = fl != LSKUM_INTERIOR;
    uint32_t left = 0;  // entries with large steps
    Pf acc[4] = {};
    if (live && !fixed) {
        PairPoint P;
        P.q = ld4(q_in + t);
        P.dq = dqp[t];
        P.local = local;
        const double2 nn = local ? g.nrm[d] : make_double2(0.0, 1.0);
        P.nx = split_pair(nn.x);
        P.ny = split_pair(nn.y);
        P.qp[0] = split_pair(P.q.a);
        P.qp[1] = split_pair(P.q.b);
        P.qp[2] = split_pair(P.q.c);
        P.qp[3] = split_pair(P.q.d);
        const int c = g.cnt[d];
        const bool second = ph.order == 2;
#pragma unroll 1
        for (int r = part; r < kClasses; r += LANES) {
            Pf sum[4] = {};
            left |= entries_pair(g, gp, second, q_in, dqp, d, cc, P, r, c, sum);
#pragma unroll
            for (int m = 0; m < 4; ++m) acc[m] = LANES == 1 ? add(acc[m], sum[m]) : sum[m];
        }
    }
    if (LANES > 1) {
#pragma unroll
        for (int r = 1; r < LANES; ++r)
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const Pf o = {__shfl_down_sync(0xffffffffu, acc[m].h, r),
                              __shfl_down_sync(0xffffffffu, acc[m].l, r)};
                if (part == 0) acc[m] = add(acc[m], o);
            }
    }
    double R[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) R[m] = double(acc[m].h) + double(acc[m].l);
    // entries with large steps: the warp's lanes share them out evenly, 32 a time, and
    // a point's are added class by class, its four components by four lanes (by one
    // lane they were more FP64 instructions than the entries themselves: 56 a pass
    // of 32 entries, 14 entries a point)
    const int mine = __popc(left);
    int upto = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane >= o) upto += v;
    }
    const int total = __shfl_sync(0xffffffffu, upto, 31);
    constexpr int kWarpPoints = 32 / LANES;
    double(*const sum)[4] = s_R + warp * kWarpPoints;
    if (LANES > 1 || total > 0) {
        if (part == 0)
#pragma unroll
            for (int m = 0; m < 4; ++m) sum[lane / LANES][m] = R[m];
        int at = upto - mine;  // positions of the lane's entries: at .. upto - 1
        const int begin = at;
        uint32_t cls = 0x11111111u;  // the class whose entries are listed next
        for (int base = 0; base < total; base += 32) {
            const int end = min(total, base + 32);
            while (left && at < end) {
                if (LANES == 1)
                    while (!(left & cls)) cls <<= 1;
                const int k = __ffs(int(LANES == 1 ? left & cls : left)) - 1;
                s_item[warp][at - base] = uint16_t((lane << 5) | k);
                left &= ~(1u << k);
                ++at;
            }
            __syncwarp();
            if (base + lane < total) {
                const int item = s_item[warp][lane];
                double c[4];
                entry_fp64(g, gp, ph, q_in, dq, t - lane / LANES + (item >> 5) / LANES, item & 31, c);
#pragma unroll
                for (int m = 0; m < 4; ++m) s_res[warp][m][lane] = c[m];
            }
            __syncwarp();
            const int first = (s_item[warp][0] >> 5) / LANES, last = (s_item[warp][end - 1 - base] >> 5) / LANES;
            for (int p0 = first; p0 <= last; p0 += 8) {  // eight points a time
                const int p = p0 + lane / 4, m = lane % 4, own = min(p, kWarpPoints - 1) * LANES;
                const int from = __shfl_sync(0xffffffffu, begin, own);
                const int to = __shfl_sync(0xffffffffu, upto, own + LANES - 1);
                if (p <= last) {
                    double r = sum[p][m];
                    for (int i = max(from, base); i < min(to, end); ++i) r += s_res[warp][m][i - base];
                    sum[p][m] = r;
                }
            }
            __syncwarp();
        }
        if (LANES == 1)
#pragma unroll
            for (int m = 0; m < 4; ++m) R[m] = sum[lane][m];
    }
    // the stage update: a thread for each point
    int64_t tu = t;
    bool update = live;
    if (LANES > 1) {
        __syncthreads();
        tu = int64_t(blockIdx.x) * (BLOCK / LANES) + threadIdx.x;
        update = threadIdx.x < BLOCK / LANES && (tu >> g.cshift) < g.n;
    }
    double r2 = 0.0;
    if (update) {
        const int64_t du = tu >> g.cshift;
        const int8_t flu = LANES > 1 ? g.flag[du] : fl;
        const bool fixu = ph.outer_fixed && flu == LSKUM_OUTER;
        if (LANES > 1)
#pragma unroll
            for (int m = 0; m < 4; ++m) R[m] = s_R[threadIdx.x][m];
        if (flu != LSKUM_INTERIOR && !fixu) {  // momentum back to the global frame
            const double2 nn = g.nrm[du];
            const double rs = R[1], rn = R[2];
            R[1] = rs * nn.y + rn * nn.x;
            R[2] = rn * nn.y - rs * nn.x;
        }
        r2 = stage_epilogue<MODE, true>(g, ph, st, tu, du, flu, fixu, R, q_out);
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

inline unsigned pair_grid(const DevGeom& g, int block, int lanes) {
    return unsigned(((g.n << g.cshift) * lanes + block - 1) / block);
}

template <int BLOCK, int LANES>
void pair_dispatch(int mode, const DevGeom& g, const DevGeomPair& gp, const Physics& ph,
                   const DevState& st, const V4* q_in, const V8* dq, const DQP* dqp, V4* q_out,
                   cudaStream_t s) {
    const unsigned grid = pair_grid(g, BLOCK, LANES);
    switch (mode) {
        case 0: k_flux_pair<0, BLOCK, LANES><<<grid, BLOCK, 0, s>>>(g, gp, ph, st, q_in, dq, dqp, q_out); break;
        case 1: k_flux_pair<1, BLOCK, LANES><<<grid, BLOCK, 0, s>>>(g, gp, ph, st, q_in, dq, dqp, q_out); break;
        case 2: k_flux_pair<2, BLOCK, LANES><<<grid, BLOCK, 0, s>>>(g, gp, ph, st, q_in, dq, dqp, q_out); break;
        case 3: k_flux_pair<3, BLOCK, LANES><<<grid, BLOCK, 0, s>>>(g, gp, ph, st, q_in, dq, dqp, q_out); break;
        default: k_flux_pair<4, BLOCK, LANES><<<grid, BLOCK, 0, s>>>(g, gp, ph, st, q_in, dq, dqp, q_out); break;
    }
}

}  // namespace

int pair_flux_lanes(const DevGeom& g) {
    return (g.n << g.cshift) <= kSplitPairs ? kClasses : 1;
}

int64_t pair_flux_blocks(const DevGeom& g, int block) {
    return pair_grid(g, block, pair_flux_lanes(g));
}

cudaError_t launch_flux_pair(int mode, const DevGeom& g, const DevGeomPair& gp, const Physics& ph,
                             const DevState& st, const V4* q_in, const V8* dq, const DQP* dqp, V4* q_out,
                             int block, cudaStream_t s) {
    const bool split = pair_flux_lanes(g) > 1;
    if (block == 256) {
        if (split) pair_dispatch<256, kClasses>(mode, g, gp, ph, st, q_in, dq, dqp, q_out, s);
        else pair_dispatch<256, 1>(mode, g, gp, ph, st, q_in, dq, dqp, q_out, s);
    } else {
        if (split) pair_dispatch<kDefaultBlock, kClasses>(mode, g, gp, ph, st, q_in, dq, dqp, q_out, s);
        else pair_dispatch<kDefaultBlock, 1>(mode, g, gp, ph, st, q_in, dq, dqp, q_out, s);
    }
    return cudaGetLastError();
}

}  // namespace lskum
