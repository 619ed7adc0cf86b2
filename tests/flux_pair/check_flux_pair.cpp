// Error of the pair-form split-flux differences (flux_pair.cuh, compiled for the
// host) against the direct evaluation of the two fluxes in binary128, and of a
// plain double evaluation, for random neighbour pairs of one step size.
// Usage: check_flux_pair MACH LOG2_STEP PAIRS -> "taken pair[4] double[4]": the
// pairs the form took, and 2-norms of the errors over the 2-norm of dG.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "../../paper_2108_07031_gb300/csrc/flux_pair.cuh"
#include "reference_flux.h"

using lskum::Pf;

static Pf pair(double x) {
    const float h = float(x);
    return Pf{h, float(x - double(h))};
}

int main(int argc, char** argv) {
    if (argc < 4) return 2;
    const double mach = std::atof(argv[1]), step = std::ldexp(1.0, std::atoi(argv[2]));
    std::mt19937_64 rng(7);
    std::uniform_real_distribution<double> U(-1, 1);
    double sum[4] = {}, err[4] = {}, err64[4] = {};
    int taken = 0;
    for (int t = 0; t < std::atoi(argv[3]); ++t) {
        double w[2][4], q[2][4];
        for (int m = 0; m < 4; ++m) {
            const double base = m == 0 ? 1 + 0.1 * U(rng) : m == 3 ? (1 + 0.1 * U(rng)) / 1.4 : mach * U(rng);
            w[0][m] = base;
            w[1][m] = base + step * U(rng) * (m == 0 || m == 3 ? base : std::max(mach, 0.1));
        }
        for (int k = 0; k < 2; ++k) {
            const double b = w[k][0] / (2 * w[k][3]);
            q[k][0] = std::log(w[k][0]) + 2.5 * std::log(b) - b * (w[k][1] * w[k][1] + w[k][2] * w[k][2]);
            q[k][1] = 2 * b * w[k][1];
            q[k][2] = 2 * b * w[k][2];
            q[k][3] = -2 * b;
        }
        Pf b[4], d[4], g[4];
        Real x0[4], x1[4], g0[4], g1[4];
        double y0[4], y1[4], h0[4], h1[4];
        for (int m = 0; m < 4; ++m) {
            b[m] = pair(q[0][m]);
            d[m] = pair(q[1][m] - q[0][m]);
            x0[m] = Real(b[m].h) + Real(b[m].l);
            x1[m] = x0[m] + Real(d[m].h) + Real(d[m].l);
            y0[m] = double(x0[m]);
            y1[m] = double(x1[m]);
        }
        lskum::PairState s;
        if (!lskum::pair_state(b, d, s)) continue;
        ++taken;
        const int axis = t & 1, sign = t & 2 ? -1 : 1;
        const float sg = float(sign);
        const Pf S = axis ? s.Sym : s.Sxm, dS = axis ? s.dSy : s.dSx;
        split_diff(s, scale(S, sg), scale(dS, sg), axis ? s.Sxm : s.Sym, axis ? s.dSx : s.dSy, g);
        flux<Real>(x0, axis, sign, g0);
        flux<Real>(x1, axis, sign, g1);
        flux<double>(y0, axis, sign, h0);
        flux<double>(y1, axis, sign, h1);
        for (int m = 0; m < 4; ++m) {
            const Real exact = g1[m] - g0[m];
            const Real got = (Real(g[m].h) + Real(g[m].l)) * (m == 1 ? 1 : sign);
            sum[m] += double(exact * exact);
            err[m] += double((got - exact) * (got - exact));
            err64[m] += double((h1[m] - h0[m] - exact) * (h1[m] - h0[m] - exact));
        }
    }
    std::printf("%d", taken);
    for (int m = 0; m < 4; ++m) std::printf(" %.3e", std::sqrt(err[m] / std::fmax(sum[m], 1e-300)));
    for (int m = 0; m < 4; ++m) std::printf(" %.3e", std::sqrt(err64[m] / std::fmax(sum[m], 1e-300)));
    std::printf("\n");
    return 0;
}
