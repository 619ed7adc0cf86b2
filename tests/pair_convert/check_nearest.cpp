// Largest |x - (hi + lo)| / |x| of nearest_pair over a million doubles, in units of 2^-49.
#include <cmath>
#include <cstdio>
#include <random>

#include "../../paper_2108_07031_gb300/csrc/pair_convert.cuh"

int main() {
    std::mt19937_64 rng(9);
    double worst = 0.0;
    for (int t = 0; t < 1000000; ++t) {
        const uint64_t r = rng();
        double x = std::ldexp(1.0 + double(r >> 12) * 0x1p-52, int(r % 41) - 20);
        if (r & 2048) x = -x;
        const lskum::Pf p = lskum::nearest_pair(x);
        worst = std::fmax(worst, std::fabs((x - double(p.h)) - double(p.l)) / std::fabs(x) * 0x1p49);
    }
    std::printf("%.6f\n", worst);
    return 0;
}
