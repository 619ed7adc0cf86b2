// Float-pair arithmetic: a value as an unevaluated sum h + l of two floats,
// |l| up to a few ulps of h (Dekker 1971, Knuth's two-sum, products by one
// fused multiply-add). Sums and products are not renormalised: about 2^-47
// relative, 4 FP32 instructions per product and 8 per sum, where one FP64
// instruction costs 64 FP32 issue slots on this GPU.
//
// Compiled by a host compiler, the same code runs on the CPU (the tests do).
#pragma once

#ifdef __CUDACC__
#define LSKUM_HD __device__ __forceinline__
#else
#define LSKUM_HD inline
#endif

#include <cmath>
#include <cstdint>
#include <cstring>

namespace lskum {

// Single roundings that the compiler must neither contract nor reorder.
LSKUM_HD float radd(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    return a + b;
#endif
}
LSKUM_HD float rsub(float a, float b) { return radd(a, -b); }
LSKUM_HD float rmul(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    return a * b;
#endif
}
LSKUM_HD float rfma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
    return __fmaf_rn(a, b, c);
#else
    return std::fmaf(a, b, c);
#endif
}
LSKUM_HD uint32_t fbits(float x) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    uint32_t u;
    std::memcpy(&u, &x, 4);
    return u;
#endif
}
LSKUM_HD float bitsf(uint32_t u) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float x;
    std::memcpy(&x, &u, 4);
    return x;
#endif
}

struct Pf {
    float h, l;
};

LSKUM_HD Pf two_sum(float a, float b) {
    const float s = radd(a, b), t = rsub(s, a);
    return {s, radd(rsub(a, rsub(s, t)), rsub(b, t))};
}
LSKUM_HD Pf quick_sum(float a, float b) {  // |a| >= |b| or a == 0
    const float s = radd(a, b);
    return {s, rsub(b, rsub(s, a))};
}
LSKUM_HD Pf norm(Pf a) { return quick_sum(a.h, a.l); }  // |l| to half an ulp of h
LSKUM_HD Pf neg(Pf a) { return {-a.h, -a.l}; }
LSKUM_HD Pf add(Pf a, Pf b) {
    Pf s = two_sum(a.h, b.h);
    s.l = radd(s.l, radd(a.l, b.l));
    return s;
}
LSKUM_HD Pf sub(Pf a, Pf b) { return add(a, neg(b)); }
LSKUM_HD Pf addq(Pf a, Pf b) {  // |a| >= |b|
    Pf s = quick_sum(a.h, b.h);
    s.l = radd(s.l, radd(a.l, b.l));
    return s;
}
LSKUM_HD Pf addq(float a, Pf b) {
    Pf s = quick_sum(a, b.h);
    s.l = radd(s.l, b.l);
    return s;
}
LSKUM_HD Pf mul(Pf a, Pf b) {
    const float p = rmul(a.h, b.h);
    return {p, rfma(a.l, b.h, rfma(a.h, b.l, rfma(a.h, b.h, -p)))};
}
LSKUM_HD Pf mul(Pf a, float b) {
    const float p = rmul(a.h, b);
    return {p, rfma(a.l, b, rfma(a.h, b, -p))};
}
LSKUM_HD Pf sq(Pf a) {
    const float p = rmul(a.h, a.h);
    return {p, rfma(radd(a.h, a.h), a.l, rfma(a.h, a.h, -p))};
}
LSKUM_HD Pf scale(Pf a, float s) { return {rmul(a.h, s), rmul(a.l, s)}; }  // s a power of two

// i = 1/sqrt(b) and i2 = 1/b for normal b. With the hardware estimate y of i,
// s = y^2 rounded and e its rounding error, u = 1 - b s = t - m (t exact, m
// small) and q = 1 - b y^2 = u - b e: two terms of the series of 1/(1 - u) and
// 1/sqrt(1 - q), the leading products with their rounding errors.
LSKUM_HD void rsqrt_pair(Pf b, Pf& i, Pf& i2) {
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(b.h));
#else
    const float y = 1.0f / std::sqrt(b.h);
#endif
    const float s = rmul(y, y), e = rfma(y, y, -s);
    const float p = rmul(b.h, s);
    const float t = rsub(1.0f, p), m = rfma(b.l, s, rfma(b.h, s, -p));
    const float u = rsub(t, m);
    float c = rmul(s, t), d = rfma(s, t, -c);
    i2 = quick_sum(s, c);
    i2 = quick_sum(i2.h, radd(i2.l, rfma(s, rfma(u, u, -m), d)));
    const float n = rfma(b.h, e, m), q = rsub(t, n);
    const float th = rmul(0.5f, t);
    c = rmul(y, th);
    d = rfma(y, th, -c);
    i = quick_sum(y, c);
    i = quick_sum(i.h, radd(i.l, rfma(y, rfma(rmul(0.375f, q), q, rmul(-0.5f, n)), d)));
}

}  // namespace lskum
