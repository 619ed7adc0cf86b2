// Errors of the fixed-point split-flux differences (flux_fixed.cuh, compiled for
// the host) and of a plain double evaluation against binary128, for random
// neighbour pairs. Usage: check_flux_fixed MACH LOG2_STEP PAIRS -> "taken fixed[4]
// double[4]": the pairs the form took, and the errors' 2-norms over that of G (of the momentum
// along the axis for both momenta).
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "../../paper_2108_07031_gb300/csrc/flux_fixed.cuh"
#include "reference_flux.h"

int main(int argc, char** argv) {
    if (argc < 4) return 2;
    const double mach = std::atof(argv[1]), step = std::ldexp(1.0, std::atoi(argv[2]));
    std::mt19937_64 rng(11);
    std::uniform_real_distribution<double> U(-1, 1);
    double sum[4] = {}, err[4] = {}, err64[4] = {};
    int taken = 0;
    for (int t = 0; t < std::atoi(argv[3]); ++t) {
        double q[2][4];
        for (int k = 0; k < 2; ++k) {
            const double x = k ? step : 0.0;
            const double rho = 1 + 0.3 * U(rng) * x, p = (1 + 0.3 * U(rng) * x) / 1.4;
            const double u = mach * U(rng) + x * U(rng), v = mach * U(rng) + x * U(rng), b = rho / (2 * p);
            q[k][0] = std::log(rho) + 2.5 * std::log(b) - b * (u * u + v * v);
            q[k][1] = 2 * b * u;
            q[k][2] = 2 * b * v;
            q[k][3] = -2 * b;
        }
        const int axis = t & 1, sign = t & 2 ? -1 : 1;
        double ds[4], dn[4], h0[4], h1[4];
        const double* d = axis ? dn : ds;
        if (!lskum::fixed_diff(q[1], q[0], false, 0.0, 1.0, sign < 0, sign < 0, ds, dn)) continue;
        ++taken;
        Real g0[4], g1[4], x0[4], x1[4];
        for (int m = 0; m < 4; ++m) {
            x0[m] = q[0][m];
            x1[m] = q[1][m];
        }
        flux<Real>(x0, axis, sign, g0);
        flux<Real>(x1, axis, sign, g1);
        flux<double>(q[0], axis, sign, h0);
        flux<double>(q[1], axis, sign, h1);
        for (int m = 0; m < 4; ++m) {
            const Real exact = g1[m] - g0[m];
            const int k = m == 2 ? 1 : m;  // both momenta by the larger one
            sum[m] += double(g1[k] * g1[k]);
            err[m] += double((d[m] - exact) * (d[m] - exact));
            err64[m] += double((h1[m] - h0[m] - exact) * (h1[m] - h0[m] - exact));
        }
    }
    std::printf("%d", taken);
    for (int m = 0; m < 4; ++m) std::printf(" %.3e", std::sqrt(err[m] / std::fmax(sum[m], 1e-300)));
    for (int m = 0; m < 4; ++m) std::printf(" %.3e", std::sqrt(err64[m] / std::fmax(sum[m], 1e-300)));
    std::printf("\n");
    return 0;
}
