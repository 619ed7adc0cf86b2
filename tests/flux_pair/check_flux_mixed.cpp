// Errors of the two FP32 forms of the split-flux differences (flux_mixed.cuh,
// compiled for the host) against binary128, for random neighbour pairs of one
// step size. Usage: check_flux_mixed MACH LOG2_STEP PAIRS -> "taken s[4]
// primitive[4]": the pairs that the form in S took, and both forms' errors, 2-norms
// over that of dG.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "../../paper_2108_07031_gb300/csrc/flux_mixed.cuh"
#include "reference_flux.h"

using lskum::Float4;

int main(int argc, char** argv) {
    if (argc < 4) return 2;
    const double mach = std::atof(argv[1]), step = std::ldexp(1.0, std::atoi(argv[2]));
    std::mt19937_64 rng(7);
    std::uniform_real_distribution<double> U(-1, 1);
    double sum[4] = {}, err[4] = {}, prim[4] = {};
    int taken = 0;
    for (int t = 0; t < std::atoi(argv[3]); ++t) {
        double w[2][4], q[2][4];
        for (int m = 0; m < 4; ++m) {
            const bool velocity = m == 1 || m == 2;
            const double base = m == 0 ? 1 + 0.05 * U(rng) : m == 3 ? (1 + 0.05 * U(rng)) / 1.4 : mach * U(rng);
            w[0][m] = base;
            w[1][m] = base + step * U(rng) * (velocity ? 1.0 : base);
        }
        for (int k = 0; k < 2; ++k) {
            const double b = w[k][0] / (2 * w[k][3]);
            q[k][0] = std::log(w[k][0]) + 2.5 * std::log(b) - b * (w[k][1] * w[k][1] + w[k][2] * w[k][2]);
            q[k][1] = 2 * b * w[k][1];
            q[k][2] = 2 * b * w[k][2];
            q[k][3] = -2 * b;
        }
        float b[4], d[4];
        Real x0[4], x1[4], g0[4], g1[4];
        for (int m = 0; m < 4; ++m) {
            b[m] = float(q[0][m]);
            d[m] = float(q[1][m] - q[0][m]);
            x0[m] = b[m];
            x1[m] = Real(b[m]) + Real(d[m]);
        }
        const Float4 base = {b[0], b[1], b[2], b[3]}, diff = {d[0], d[1], d[2], d[3]};
        lskum::MxState s;
        if (!lskum::mx_state(base, diff, s)) continue;
        ++taken;
        const int axis = t & 1, sign = t & 2 ? -1 : 1;
        const float sg = float(sign);
        float g[4], h[4];
        lskum::mx_diff(s, sg * (axis ? s.Sym : s.Sxm), sg * (axis ? s.dSy : s.dSx), axis ? s.Sxm : s.Sym,
                       axis ? s.dSx : s.dSy, g);
        const lskum::PrimPair p = lskum::prim_pair<true>(base, diff, 2.5f);
        if (axis) lskum::dsplit_flux_a(p, p.v, p.u, p.dv, p.du, sg, h);
        else lskum::dsplit_flux_a(p, p.u, p.v, p.du, p.dv, sg, h);
        flux<Real>(x0, axis, sign, g0);
        flux<Real>(x1, axis, sign, g1);
        for (int m = 0; m < 4; ++m) {
            const Real exact = g1[m] - g0[m], got = Real(g[m]) * (m == 1 ? 1 : sign);
            sum[m] += double(exact * exact);
            err[m] += double((got - exact) * (got - exact));
            prim[m] += double((h[m] - exact) * (h[m] - exact));
        }
    }
    std::printf("%d", taken);
    for (int m = 0; m < 4; ++m) std::printf(" %.3e", std::sqrt(err[m] / std::fmax(sum[m], 1e-300)));
    for (int m = 0; m < 4; ++m) std::printf(" %.3e", std::sqrt(prim[m] / std::fmax(sum[m], 1e-300)));
    std::printf("\n");
    return 0;
}
