// The pair form (flux_pair.cuh, compiled for the host) over its whole range of
// beta and ln(rho beta^2.5), the corners included, at steps of 2^-10 and |S| = 0.3
// and 4. Prints "taken bad worst": the neighbour pairs it took, those of them with a
// flux difference that is not finite, and the largest error of a component over
// that component of G.
#include <cmath>
#include <cstdio>
#include <initializer_list>

#include "../../paper_2108_07031_gb300/csrc/flux_pair.cuh"
#include "reference_flux.h"

using lskum::Pf;

static Pf pair(double x) {
    const float h = float(x);
    return Pf{h, float(x - double(h))};
}

int main() {
    int taken = 0, bad = 0;
    double worst = 0.0;
    for (int e = -26; e <= 26; ++e)
        for (int a = -82; a <= 82; ++a)
            for (double S : {0.3, 4.0}) {
                const double beta = std::ldexp(1.3, e), arg = 0.5 * a, up = 1.0 + std::ldexp(1.0, -10);
                const double q[4] = {arg - S * S, 2 * S * std::sqrt(beta), 0.1 * std::sqrt(beta), -2 * beta};
                const double r[4] = {q[0] + std::ldexp(1.0, -11), q[1] * up, q[2], q[3] * up};
                Pf b[4], d[4], g[4];
                Real x0[4], x1[4], g0[4], g1[4];
                for (int m = 0; m < 4; ++m) {
                    b[m] = pair(q[m]);
                    d[m] = pair(r[m] - q[m]);
                    x0[m] = Real(b[m].h) + Real(b[m].l);
                    x1[m] = x0[m] + Real(d[m].h) + Real(d[m].l);
                }
                lskum::PairState s;
                if (!lskum::pair_state(b, d, s)) continue;
                ++taken;
                split_diff(s, s.Sxm, s.dSx, s.Sym, s.dSy, g);
                flux<Real>(x0, 0, 1, g0);
                flux<Real>(x1, 0, 1, g1);
                bool finite = true;
                for (int m = 0; m < 4; ++m) {
                    finite = finite && std::isfinite(g[m].h) && std::isfinite(g[m].l);
                    const double err = double((Real(g[m].h) + Real(g[m].l) - (g1[m] - g0[m])) / g0[m]);
                    if (std::isfinite(err)) worst = std::fmax(worst, std::fabs(err));
                }
                bad += !finite;
            }
    std::printf("%d %d %.3e\n", taken, bad, worst);
    return 0;
}
