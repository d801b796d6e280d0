// Double-float arithmetic (a value as the unevaluated sum of two FP32 numbers, about 46 bits) for the Gaussian draws: FP64
// runs at two lanes a clock an SM on this part, so FP64 logarithms and sines bound the draws at 1.16 ms for 256^3.
// Error-free transformations of Dekker (1971) and Knuth (TAOCP vol. 2, 4.2.2) with a fused multiply-add for products; the
// functions are Taylor and atanh series whose leading terms are double-float and whose small terms are FP32.  Relative errors:
// radii 2.2e-13, cosines and sines 5e-14 (checked on the host, which is what the host branches are for).
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace pb {
namespace dd {

struct F2 {
    float h, l;
};
#ifdef __CUDA_ARCH__
__device__ __forceinline__ float add_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float sqrt_(float a) { return __fsqrt_rn(a); }
__device__ __forceinline__ float div_(float a, float b) { return __fdividef(a, b); }   // a few ulp: corrected below
__device__ __forceinline__ int clz_(unsigned long long v) { return __clzll((long long)v); }
#else
inline float add_(float a, float b) { return a + b; }
inline float mul_(float a, float b) { return a * b; }
inline float fma_(float a, float b, float c) { return fmaf(a, b, c); }
inline float sqrt_(float a) { return sqrtf(a); }
inline float div_(float a, float b) { return a / b; }
inline int clz_(unsigned long long v) { return __builtin_clzll(v); }
#endif
#define PB_HD __host__ __device__ __forceinline__

PB_HD F2 quick_sum(float a, float b) {               // |a| >= |b|
    const float s = add_(a, b);
    return F2{s, add_(b, -add_(s, -a))};
}
PB_HD F2 two_sum(float a, float b) {
    const float s = add_(a, b), v = add_(s, -a);
    return F2{s, add_(add_(a, -add_(s, -v)), add_(b, -v))};
}
PB_HD F2 two_prod(float a, float b) {
    const float p = mul_(a, b);
    return F2{p, fma_(a, b, -p)};
}
PB_HD F2 mul(F2 a, F2 b) {
    F2 p = two_prod(a.h, b.h);
    p.l = fma_(a.h, b.l, fma_(a.l, b.h, p.l));
    return quick_sum(p.h, p.l);
}
PB_HD F2 add(F2 a, F2 b) {
    F2 s = two_sum(a.h, b.h);
    s.l = add_(s.l, add_(a.l, b.l));
    return quick_sum(s.h, s.l);
}
PB_HD F2 neg(F2 a) { return F2{-a.h, -a.l}; }
// c + x for a double constant c.
PB_HD F2 split(double c) { return F2{(float)c, (float)(c - (double)(float)c)}; }

// The integer v < 2^48 as a double-float (exact).
PB_HD F2 from_int(unsigned long long v) {
    const float h = (float)(v >> 24) * 16777216.f, l = (float)(v & 0xFFFFFFull);
    return quick_sum(h, l);
}

// sqrt(-2 ln u) for u = v 2^-33, v odd, 0 < v < 2^33.
PB_HD F2 radius(unsigned long long v) {
    const int e = 63 - clz_(v);                       // v = m 2^e, 1 <= m < 2
    // m (exact: at most 33 bits), and the half of it above sqrt 2
    F2 m = from_int(v);
    int k = e;
    float sc = 1.f;
#ifdef __CUDA_ARCH__
    sc = __int_as_float((127 - e) << 23);
#else
    sc = ldexpf(1.f, -e);
#endif
    m.h *= sc;
    m.l *= sc;
    if (m.h > 1.41421356f) {
        m.h *= 0.5f;
        m.l *= 0.5f;
        ++k;
    }
    // f = (m - 1) / (m + 1); both sums are exact to double-float
    const F2 num = add(m, F2{-1.f, 0.f}), den = add(m, F2{1.f, 0.f});
    const float q1 = div_(num.h, den.h);
    const F2 r1 = add(num, neg(mul(F2{q1, 0.f}, den)));
    const float q2 = div_(r1.h, den.h);
    const F2 r2 = add(r1, neg(mul(F2{q2, 0.f}, den)));
    const F2 f = add(quick_sum(q1, q2), F2{div_(r2.h, den.h), 0.f});
    // ln m = 2 f (1 + t/3 + t^2/5 + ..), t = f^2 <= 0.0295
    const F2 t = mul(f, f);
    const float g = fma_(t.h, fma_(t.h, fma_(t.h, fma_(t.h, 1.f / 15.f, 1.f / 13.f), 1.f / 11.f), 1.f / 9.f), 1.f / 7.f);
    const F2 a = add(split(1.0 / 5.0), two_prod(t.h, g));
    const F2 b = add(split(1.0 / 3.0), mul(t, a));
    const F2 s = mul(t, b);
    const F2 lnm = mul(F2{2.f * f.h, 2.f * f.l}, add(F2{1.f, 0.f}, s));
    // ln u = ln m + (k - 33) ln 2, ln 2 in three parts (the products of the first are exact)
    const float n = (float)(k - 33);
    const float l1 = 0.693145751953125f;              // 15 bits
    const double l2 = 0.69314718055994530942 - 0.693145751953125;
    F2 ln = add(F2{n * l1, 0.f}, mul(F2{n, 0.f}, split(l2)));
    ln = add(ln, lnm);
    const F2 x = F2{-2.f * ln.h, -2.f * ln.l};
    const float r = sqrt_(x.h);
    // r + (x - r^2) / (2 r)
    const F2 rr = two_prod(r, r);
    const float d = add_(add_(add_(x.h, -rr.h), -rr.l), x.l);
    return quick_sum(r, div_(d, 2.f * r));
}

// cos and sin of 2 pi v 2^-33, v odd, 0 < v < 2^33.
PB_HD void sincos_turn(unsigned long long v, F2& c, F2& s) {
    const int o = (int)(v >> 30);                     // octant
    const unsigned long long rem = v & 0x3FFFFFFFull;
    const unsigned long long w = (o & 1) ? 0x40000000ull - rem : rem;   // 0 < w < 2^30
    F2 x = from_int(w);
    const float sc = 9.31322574615478515625e-10f;     // 2^-30
    x.h *= sc;
    x.l *= sc;
    const F2 th = mul(x, split(0.78539816339744830962));
    const F2 t = mul(th, th);                         // <= 0.617
    // sin th = th (1 - t/6 + t^2/120 - t^3/5040 + t^4/362880 - ..)
    const float gs = fma_(t.h, fma_(t.h, fma_(t.h, -1.f / 1307674368000.f, 1.f / 6227020800.f), -1.f / 39916800.f), 1.f / 362880.f);
    F2 p = add(split(-1.0 / 5040.0), two_prod(t.h, gs));
    p = add(split(1.0 / 120.0), mul(t, p));
    p = add(split(-1.0 / 6.0), mul(t, p));
    p = add(F2{1.f, 0.f}, mul(t, p));
    const F2 sn = mul(th, p);
    // cos th = 1 - t/2 + t^2/24 - t^3/720 + t^4/40320 - t^5/3628800 + ..
    const float gc =
        fma_(t.h, fma_(t.h, fma_(t.h, 1.f / 20922789888000.f, -1.f / 87178291200.f), 1.f / 479001600.f), -1.f / 3628800.f);
    F2 q = add(split(1.0 / 40320.0), two_prod(t.h, gc));
    q = add(split(-1.0 / 720.0), mul(t, q));
    q = add(split(1.0 / 24.0), mul(t, q));
    q = add(F2{-0.5f, 0.f}, mul(t, q));
    const F2 cs = add(F2{1.f, 0.f}, mul(t, q));
    // octants: (o + 1) & 2 exchanges the two; signs by the quadrant
    const bool swap = ((o + 1) & 2) != 0;
    c = swap ? sn : cs;
    s = swap ? cs : sn;
    if (o >= 2 && o < 6) c = neg(c);
    if (o >= 4) s = neg(s);
}

// The product of two double-floats rounded to FP32; sure = false where a relative error of 2^-39 (1.8e-12) in the product
// could change the rounding (Ziv's test): 0.5 % of 128 values hold such a one.
PB_HD float round_prod(F2 a, F2 b, bool& sure) {
    const F2 p = mul(a, b);
    const float e = mul_(fabsf(p.h), 1.8189894035458564758e-12f);
    const float z = add_(p.h, add_(p.l, e));
    sure = sure && z == add_(p.h, add_(p.l, -e));
    return z;
}

#undef PB_HD
}  // namespace dd
}  // namespace pb
