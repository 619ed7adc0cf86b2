// The set-up's float pairs with their rests (lskum_setup.cpp). Without arguments: the
// number of random doubles that hi + lo + rest does not give back bit for bit. With
// an exponent: whether the pair form holds a small cloud scaled by 2^exponent.
#include <cstdio>
#include <cstdlib>
#include <random>

#include "../../paper_2108_07031_gb300/csrc/lskum_setup.cpp"

static int held(double scale) {
    constexpr int nt = 24, nr = 5, n = nt * nr;  // rings around a cylinder
    std::vector<double> xy, nrm;
    std::vector<int8_t> flag;
    std::vector<int32_t> off{0}, idx;
    for (int i = 0; i < n; ++i) {
        const double a = 2 * M_PI * (i % nt) / nt, r = scale * (1.0 + 0.3 * (i / nt));
        xy.insert(xy.end(), {r * std::cos(a), r * std::sin(a)});
        nrm.insert(nrm.end(), {std::cos(a), std::sin(a)});
        flag.push_back(i < nt ? LSKUM_WALL : i >= n - nt ? LSKUM_OUTER : LSKUM_INTERIOR);
        for (int k = -1; k <= 1; ++k)
            for (int t = -2; t <= 2; ++t)
                if ((k || t) && i / nt + k >= 0 && i / nt + k < nr) idx.push_back((i / nt + k) * nt + (i + t + nt) % nt);
        off.push_back(int32_t(idx.size()));
    }
    lskum_options o{};
    o.gamma = 1.4;
    o.order = 2;
    o.wall_factor = 2.0;
    o.n_conditions = 1;
    lskum::HostLayout L;
    std::string err;
    const int rc = lskum::build_layout(n, xy.data(), nrm.data(), flag.data(), off.data(), idx.data(), o, true, L, err);
    if (rc) std::fprintf(stderr, "%s\n", err.c_str());
    return rc ? -1 : L.held;
}

int main(int argc, char** argv) {
    if (argc > 1) {
        std::printf("%d\n", held(std::ldexp(1.0, std::atoi(argv[1]))));
        return 0;
    }
    std::mt19937_64 rng(5);
    int wrong = 0;
    for (int t = 0; t < 1000000; ++t) {
        const uint64_t r = rng();
        double x = std::ldexp(1.0 + double(r >> 12) * 0x1p-52, int(r % 120) - 60);
        if (r & 2048) x = -x;
        float f[2];
        int8_t rest;
        const bool ok = lskum::split(x, f, &rest);
        const double sum = double(f[0]) + double(f[1]);
        int64_t bits;
        std::memcpy(&bits, &sum, 8);
        bits += rest;
        wrong += !ok || std::memcmp(&bits, &x, 8) != 0;
    }
    std::printf("%d\n", wrong);
    return 0;
}
