// Pairs of FP32 numbers (h + l, |l| <= ulp(h) / 2: 48 bits) for the few places of the FP32 path
// that take their values from FP64: the phases of the initial conditions, their spectral filter
// and their placement.  FP64 arithmetic runs at a small fraction of the FP32 rate on this part.
// Sums, products and quotients of pairs are within 2^-44 of their value; the functions below end
// their series in single numbers and are within 2^-33 (logarithm and cosine 6e-11, sine 7e-12),
// so that a value rounded to FP32 is what the FP64 value gives but for one in ten thousand, and a
// neighbour of it there, off by at most 0.502 units.
//
// Error-free sums and products after Knuth and Dekker (the product by fused multiply-add).
#pragma once

#include <stdint.h>

namespace pm {

struct df {
    float h, l;
};

// The pair nearest a double.
__host__ __device__ constexpr df df_of(double v) { return df{(float)v, (float)(v - (double)(float)v)}; }

#ifdef __CUDACC__

__device__ __forceinline__ df two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return df{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
// |a| >= |b| (or a = 0)
__device__ __forceinline__ df quick_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return df{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ df two_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return df{p, fmaf(a, b, -p)};
}
__device__ __forceinline__ df operator*(df a, df b) {
    df p = two_prod(a.h, b.h);
    p.l = fmaf(a.h, b.l, fmaf(a.l, b.h, p.l));
    return quick_sum(p.h, p.l);
}
__device__ __forceinline__ df operator*(float a, df b) {
    df p = two_prod(a, b.h);
    p.l = fmaf(a, b.l, p.l);
    return quick_sum(p.h, p.l);
}
__device__ __forceinline__ df operator+(df a, df b) {
    df s = two_sum(a.h, b.h);
    s.l = __fadd_rn(s.l, __fadd_rn(a.l, b.l));
    return quick_sum(s.h, s.l);
}
// The FP32 number nearest the pair.
__device__ __forceinline__ float round_df(df a) { return __fadd_rn(a.h, a.l); }
// Nearest integer of a pair with |a| < 2^30.
__device__ __forceinline__ int df2int_rn(df a) {
    const int i = __float2int_rn(a.h);
    return i + __float2int_rn(__fadd_rn(__fsub_rn(a.h, (float)i), a.l));
}
// a / n for an exact n: the quotient of the leading parts, then one Newton-Raphson correction
// from its remainder (the quotient's error squares to below the pair's).
__device__ __forceinline__ df df_div(df a, float n) {
    const float r = __fdividef(1.0f, n), q = __fmul_rn(a.h, r);
    return quick_sum(q, __fmul_rn(__fadd_rn(fmaf(-q, n, a.h), a.l), r));
}

// -ln((r + 1/2) 2^-32): with (r + 1/2) 2^-32 = 2^-k (1 + f), 1 + f in [1/sqrt 2, sqrt 2),
// k ln 2 - 2 artanh(s), s = f / (2 + f), artanh by its Taylor series in s^2 <= 0.0295 (to
// s^16 / 17, below 2^-44), its first two terms as pairs.
__device__ __forceinline__ df neg_log_unit(uint32_t r) {
    // v = 2 r + 1 = vh + vl exactly, 2^33 (r + 1/2) 2^-32
    const float vh = (float)(r >> 16) * 131072.0f, vl = (float)(2u * (r & 0xffffu) + 1u);
    const uint32_t bits = __float_as_uint(__fadd_rn(vh, vl));
    int e = (int)(bits >> 23) - 127;
    if ((bits & 0x7fffffu) > 0x3504f3u) e += 1;  // mantissa above sqrt 2
    const float sc = __uint_as_float((uint32_t)(127 - e) << 23);  // 2^-e
    const df f = two_sum(__fmaf_rn(vh, sc, -1.0f), __fmul_rn(vl, sc));
    // s = f / (2 + f): quotient and one correction
    df d = two_sum(2.0f, f.h);
    d.l = __fadd_rn(d.l, f.l);
    const float rd = __fdividef(1.0f, d.h), q = __fmul_rn(f.h, rd);
    const df s = quick_sum(q, __fmul_rn(fmaf(-q, d.l, __fadd_rn(fmaf(-q, d.h, f.h), f.l)), rd));
    df z = two_prod(s.h, s.h);
    z.l = fmaf(2.0f * s.h, s.l, z.l);
    float p = 1.0f / 17.0f;
    p = fmaf(p, z.h, 1.0f / 15.0f);
    p = fmaf(p, z.h, 1.0f / 13.0f);
    p = fmaf(p, z.h, 1.0f / 11.0f);
    p = fmaf(p, z.h, 1.0f / 9.0f);
    p = fmaf(p, z.h, 1.0f / 7.0f);
    p = fmaf(p, z.h, 1.0f / 5.0f);
    constexpr df third = df_of(1.0 / 3.0);
    df t = third * z;
    t.l = fmaf(__fmul_rn(z.h, z.h), p, t.l);  // z / 3 + z^2 / 5 + ...
    t = quick_sum(t.h, t.l);
    const df L = s + s * t;  // artanh(s)
    // ln 2 = 0.693145751953125 (18 bits, so that k times it is exact) + the rest
    constexpr float ln2h = 0.693145751953125f, ln2l = (float)(0.69314718055994530942 - 0.693145751953125);
    const float k = (float)(33 - e);
    df a = two_sum(__fmul_rn(k, ln2h), -2.0f * L.h);
    a.l = __fadd_rn(a.l, fmaf(k, ln2l, -2.0f * L.l));
    return quick_sum(a.h, a.l);
}

// sqrt of a positive pair: one Newton step from the reciprocal square root of its leading part.
__device__ __forceinline__ df df_sqrt(df a) {
    const float r = rsqrtf(a.h), g = __fmul_rn(a.h, r);
    return quick_sum(g, __fmul_rn(0.5f * r, __fadd_rn(fmaf(-g, g, a.h), a.l)));
}

// sin and cos of 2 pi (r + 1/2) 2^-32: the nearest quarter turn is taken off exactly in integers,
// the rest x, |x| <= pi / 4, goes through the Taylor series with their leading terms as pairs.
__device__ __forceinline__ void sincos_unit(uint32_t r, df& sn, df& cs) {
    const uint32_t k = ((r >> 29) + 1u) >> 1;  // nearest quarter turn, 0..4
    const int t = (int)(2u * r + 1u - (k << 31));
    const float th = (float)t, tl = (float)(t - (int)th);
    // x = t pi 2^-32
    constexpr df c = df_of(3.14159265358979323846 / 4294967296.0);
    df x = two_prod(th, c.h);
    x.l = fmaf(th, c.l, fmaf(tl, c.h, x.l));
    x = quick_sum(x.h, x.l);
    const df z = x * x;
    // sin x = x + x z (-1/6 + z (1/120 - z / 5040 + ...)), 1/6 and 1/120 as pairs: with the latter
    // single the sine was off by up to 6.5e-10
    float ps = 1.0f / 6227020800.0f;
    ps = fmaf(ps, z.h, -1.0f / 39916800.0f);
    ps = fmaf(ps, z.h, 1.0f / 362880.0f);
    ps = fmaf(ps, z.h, -1.0f / 5040.0f);
    constexpr df c3 = df_of(-1.0 / 6.0), c5 = df_of(1.0 / 120.0);
    df v = quick_sum(c5.h, __fmul_rn(ps, z.h));
    v.l = __fadd_rn(v.l, c5.l);
    const df s = x + x * (z * (c3 + z * v));
    // cos x = 1 - z / 2 + z^2 (1/24 - z (1/720 - z / 40320 + ...))
    float pc = -1.0f / 87178291200.0f;
    pc = fmaf(pc, z.h, 1.0f / 479001600.0f);
    pc = fmaf(pc, z.h, -1.0f / 3628800.0f);
    pc = fmaf(pc, z.h, 1.0f / 40320.0f);
    pc = fmaf(pc, z.h, -1.0f / 720.0f);
    constexpr df c4 = df_of(1.0 / 24.0);
    df w = quick_sum(c4.h, __fmul_rn(pc, z.h));
    w.l = __fadd_rn(w.l, c4.l);
    const df q = df{1.0f, 0.0f} + (df{-0.5f * z.h, -0.5f * z.l} + z * z * w);
    // rotate by k quarter turns
    const bool swap = k & 1u;
    df ss = swap ? q : s, cc = swap ? s : q;
    const float fs = (k & 2u) ? -1.0f : 1.0f, fc = ((k + 1u) & 2u) ? -1.0f : 1.0f;
    sn = df{fs * ss.h, fs * ss.l};
    cs = df{fc * cc.h, fc * cc.l};
}

#endif  // __CUDACC__

}  // namespace pm
