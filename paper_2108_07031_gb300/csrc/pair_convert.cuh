// Conversions between FP64 and floats by integer operations: the hardware's run
// at the FP64 pipe's rate, 1/64 of the FP32 and integer pipes'.
#pragma once

#include "pair_math.cuh"

namespace lskum {

LSKUM_HD uint64_t dword(double x) {
#ifdef __CUDA_ARCH__
    return uint64_t(__double_as_longlong(x));
#else
    uint64_t u;
    std::memcpy(&u, &x, 8);
    return u;
#endif
}
LSKUM_HD double dvalue(uint64_t u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(int64_t(u));
#else
    double x;
    std::memcpy(&x, &u, 8);
    return x;
#endif
}

#ifdef __CUDACC__
// x as a pair to 2^-48: the leading 24 bits truncated, the other 29 rounded to a float.
// Integer operations only (the conversions between FP64 and FP32 run at the
// FP64 pipe's rate). |x| below 2^-74 gives zero, above 2^127 or not finite NaN.
__device__ __forceinline__ Pf split_pair(const double x) {
    const uint32_t hi = uint32_t(__double2hiint(x)), lo = uint32_t(__double2loint(x));
    const uint32_t mag = hi & 0x7fffffffu;
    const uint32_t hb = (hi & 0x80000000u) | ((__funnelshift_l(lo, hi, 3) ^ 0x40000000u) & 0x7fffffffu);
    Pf r;
    r.h = bitsf(hb);
    r.l = rmul(__uint2float_rn(lo & 0x1fffffffu), bitsf((hb & 0xff800000u) - (52u << 23)));
    if (mag - 0x3b500000u >= 0x0ca00000u) {  // exponent outside [-74, 127)
        const bool small = mag < 0x3b500000u;
        r.h = small ? 0.f : __int_as_float(0x7fc00000);
        r.l = 0.f;
    }
    return r;
}
#endif

// x as the nearest pair, to 2^-49: where the conversions' rate does not matter.
LSKUM_HD Pf nearest_pair(const double x) {
    const float h = float(x);
    return {h, float(x - double(h))};
}

// The double equal to a float, infinities and NaN included, by integer
// operations; subnormals give zero.
LSKUM_HD double widen(const float x) {
    const uint32_t u = fbits(x), mag = u & 0x7fffffffu;
    const bool zero = mag < 0x00800000u;
    const uint32_t rebias = mag >= 0x7f800000u ? 0x70000000u : 0x38000000u;
    return dvalue(uint64_t((u & 0x80000000u) | (zero ? 0u : (mag >> 3) + rebias)) << 32 |
                  (zero ? 0u : u << 29));
}

// x truncated to a float, for 2^-100 < |x| < 2^100; smaller ones give zero.
LSKUM_HD float narrow(const double x) {
    const uint64_t u = dword(x);
    const uint32_t hi = uint32_t(u >> 32), mag = uint32_t((u & 0x7fffffffffffffffULL) >> 29) - 0xc0000000u;
    return (hi & 0x7fffffffu) < 0x39b00000u ? 0.f : bitsf((hi & 0x80000000u) | (mag & 0x7fffffffu));
}

}  // namespace lskum
