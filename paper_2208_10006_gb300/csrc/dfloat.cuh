// Double-FP32 ("double-float") arithmetic: a value is hi + lo with two floats,
// |lo| <= ulp(hi)/2, about 48 significant bits. Used for the ray state of the
// bounce kernel (origin, direction, unfolded length) and the reception test,
// where FP32 is too coarse and FP64 is scarce on this GPU. Built from the
// error-free transformations: Knuth's two-sum, Dekker's fast two-sum and the
// FMA-based two-product; division takes two correction steps of the quotient,
// the dot product gathers every lower-order term in one float (the compensated
// dot product of Ogita, Rump and Oishi, 2005).
#pragma once
#include <cuda_runtime.h>

namespace sbr {

struct df {
    float hi, lo;
};

__device__ __forceinline__ df df_make(float h, float l) { return df{h, l}; }

// exact split of a double into hi + lo floats
__host__ __device__ __forceinline__ df df_from_double(double x) {
    float h = (float)x;
    return df{h, (float)(x - (double)h)};
}
__device__ __forceinline__ double df_to_double(df a) { return (double)a.hi + (double)a.lo; }

#ifdef __CUDACC__
// the same split by integer operations (a double-precision conversion or
// subtraction takes some 70 FP32 slots on this GPU): the upper 24 significant
// bits by shifting, the lower 29 through an integer conversion. Values outside
// [2^-74, 2^127) keep their FP32 rounding only.
__device__ __forceinline__ df df_split(double x) {
    const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
    const unsigned e = (h >> 20) & 0x7ffu;
    if (e - 949u >= 201u) return df{__double2float_rn(x), 0.f};
    const unsigned sign = h & 0x80000000u;
    const float hi = __uint_as_float(((__funnelshift_l(l, h, 3) ^ 0x40000000u) & 0x7fffffffu) | sign);
    const float scale = __uint_as_float(((e - 948u) << 23) | sign);
    const float lo = __fmul_rn(__uint2float_rn(l & 0x1fffffffu), scale);
    const float s = __fadd_rn(hi, lo);
    return df{s, __fsub_rn(lo, __fsub_rn(s, hi))};
}
#endif

__device__ __forceinline__ df two_sum(float a, float b) {
    float s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return df{s, e};
}
// requires |a| >= |b| (or a == 0)
__device__ __forceinline__ df fast_two_sum(float a, float b) {
    float s = __fadd_rn(a, b);
    float e = __fsub_rn(b, __fsub_rn(s, a));
    return df{s, e};
}
__device__ __forceinline__ df two_prod(float a, float b) {
    float p = __fmul_rn(a, b);
    return df{p, __fmaf_rn(a, b, -p)};
}

// a + b with one two-sum on the high words and the low words added in FP32:
// the error is a few units of 2^-48 of the operands' magnitude (not of the
// result's, under cancellation), the absolute accuracy the ray state, the face
// planes and the receiver positions carry in any case
__device__ __forceinline__ df df_add(df a, df b) {
    df s = two_sum(a.hi, b.hi);
    s.lo = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
    return fast_two_sum(s.hi, s.lo);
}
__device__ __forceinline__ df df_neg(df a) { return df{-a.hi, -a.lo}; }
__device__ __forceinline__ df df_sub(df a, df b) { return df_add(a, df_neg(b)); }

__device__ __forceinline__ df df_mul(df a, df b) {
    df p = two_prod(a.hi, b.hi);
    p.lo = __fmaf_rn(a.hi, b.lo, p.lo);
    p.lo = __fmaf_rn(a.lo, b.hi, p.lo);
    return fast_two_sum(p.hi, p.lo);
}
__device__ __forceinline__ df df_mul_f(df a, float b) {
    df p = two_prod(a.hi, b);
    p.lo = __fmaf_rn(a.lo, b, p.lo);
    return fast_two_sum(p.hi, p.lo);
}
// a / b: quotient terms from one reciprocal of b.hi, each correcting the
// residual the previous ones left (computed in double-float); a term only
// needs to be close to the residual's quotient, so the reciprocal's rounding
// does not limit the result
__device__ __forceinline__ df df_div(df a, df b) {
    const float ib = __frcp_rn(b.hi);
    float q1 = a.hi * ib;
    df r = df_sub(a, df_mul_f(b, q1));
    float q2 = r.hi * ib;
    r = df_sub(r, df_mul_f(b, q2));
    float q3 = r.hi * ib;
    df q = fast_two_sum(q1, q2);
    return df_add(q, df{q3, 0.f});
}
// a b + c d, error-free on the high words, the rest gathered in one float
__device__ __forceinline__ df df_dot2(df a, df b, df c, df d) {
    const df p = two_prod(a.hi, b.hi), q = two_prod(c.hi, d.hi);
    const df s = two_sum(p.hi, q.hi);
    float e = __fadd_rn(__fadd_rn(p.lo, q.lo), s.lo);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    e = __fmaf_rn(c.hi, d.lo, e);
    e = __fmaf_rn(c.lo, d.hi, e);
    return two_sum(s.hi, e);
}
// 1 / a and sqrt(a) for normal a (a > 0 under the root): the hardware
// approximation x and one correction from its exact residual, 1 / a with the
// second-order term (relative error about 2^-45)
__device__ __forceinline__ df df_rcp(df a) {
    float x;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(x) : "f"(a.hi));
    const float r = __fmaf_rn(-a.lo, x, __fmaf_rn(-a.hi, x, 1.f));
    return fast_two_sum(x, __fmul_rn(x, __fmaf_rn(r, r, r)));
}
__device__ __forceinline__ df df_sqrt(df a) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a.hi));
    const float s = __fmul_rn(a.hi, y);
    const float r = __fadd_rn(__fmaf_rn(-s, s, a.hi), a.lo);
    return fast_two_sum(s, __fmul_rn(__fmul_rn(0.5f, y), r));
}
// length from its square: zero below the normal range (1e-19), where the two above fail
__device__ __forceinline__ df df_length(df n2) { return n2.hi >= 1.17549435e-38f ? df_sqrt(n2) : df{0.f, 0.f}; }
// log2 of a positive normal double: exponent and 2 atanh((m - 1) / (m + 1)) of
// the mantissa m in [0.71, 1.42); absolute error below 2e-11
__device__ __forceinline__ df df_log2(double x) {
    const int h = __double2hiint(x);
    const bool up = (h & 0xfffff) >= 0x6a09e;   // m >= sqrt 2
    const float e = (float)((h >> 20) - 1023 + (up ? 1 : 0));
    const df m = df_split(__hiloint2double((h & 0xfffff) | (up ? 0x3fe00000 : 0x3ff00000), __double2loint(x)));
    const df one{1.f, 0.f};
    const df s = df_mul(df_sub(m, one), df_rcp(df_add(m, one)));
    const df t = df_mul(s, s);   // at most 0.03
    float q = __fmaf_rn(1.f / 13.f, t.hi, 1.f / 11.f);
    q = __fmaf_rn(q, t.hi, 1.f / 9.f);
    q = __fmaf_rn(q, t.hi, 1.f / 7.f);
    q = __fmaf_rn(q, t.hi, 1.f / 5.f);
    const df y = df_add(s, df_mul(s, df_mul(t, df_add(df{0.333333343f, -9.93410776e-9f}, two_prod(q, t.hi)))));
    return df_add(df{e, 0.f}, df_mul(y, df{2.88539004f, 3.85192598e-8f}));   // 2 / ln 2
}
// a < b, a <= b on the represented values
__device__ __forceinline__ bool df_lt(df a, df b) { return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo); }
__device__ __forceinline__ bool df_le(df a, df b) { return a.hi < b.hi || (a.hi == b.hi && a.lo <= b.lo); }

struct df3 {
    df x, y, z;
};
__device__ __forceinline__ df3 df3_add(df3 a, df3 b) { return df3{df_add(a.x, b.x), df_add(a.y, b.y), df_add(a.z, b.z)}; }
__device__ __forceinline__ df3 df3_sub(df3 a, df3 b) { return df3{df_sub(a.x, b.x), df_sub(a.y, b.y), df_sub(a.z, b.z)}; }
__device__ __forceinline__ df3 df3_scale(df3 a, df s) { return df3{df_mul(a.x, s), df_mul(a.y, s), df_mul(a.z, s)}; }
// a.b: the three hi*hi products and their two partial sums by error-free
// transformations; their errors, the cross terms hi*lo and lo*hi are summed in
// one float and added once (not symmetric in a, b to the last bit: callers
// keep one argument order per quantity)
__device__ __forceinline__ df df3_dot(df3 a, df3 b) {
    const df px = two_prod(a.x.hi, b.x.hi), py = two_prod(a.y.hi, b.y.hi), pz = two_prod(a.z.hi, b.z.hi);
    const df s1 = two_sum(px.hi, py.hi);
    const df s2 = two_sum(s1.hi, pz.hi);
    float e = __fadd_rn(__fadd_rn(px.lo, py.lo), __fadd_rn(pz.lo, __fadd_rn(s1.lo, s2.lo)));
    e = __fmaf_rn(a.x.hi, b.x.lo, e);
    e = __fmaf_rn(a.x.lo, b.x.hi, e);
    e = __fmaf_rn(a.y.hi, b.y.lo, e);
    e = __fmaf_rn(a.y.lo, b.y.hi, e);
    e = __fmaf_rn(a.z.hi, b.z.lo, e);
    e = __fmaf_rn(a.z.lo, b.z.hi, e);
    return two_sum(s2.hi, e);   // not fast_two_sum: under cancellation |e| may exceed |s2.hi|
}
// a + b c in one pass: the product's high word error-free, its low terms and
// a.lo gathered in FP32 (the accuracy of df_mul followed by df_add)
__device__ __forceinline__ df df_fma(df a, df b, df c) {
    df p = two_prod(b.hi, c.hi);
    p.lo = __fmaf_rn(b.hi, c.lo, p.lo);
    p.lo = __fmaf_rn(b.lo, c.hi, p.lo);
    df s = two_sum(a.hi, p.hi);
    s.lo = __fadd_rn(s.lo, __fadd_rn(a.lo, p.lo));
    return fast_two_sum(s.hi, s.lo);
}
// a + b s for vectors a, b and a scalar s
__device__ __forceinline__ df3 df3_fma(df3 a, df3 b, df s) {
    return df3{df_fma(a.x, b.x, s), df_fma(a.y, b.y, s), df_fma(a.z, b.z, s)};
}
__device__ __forceinline__ float3 df3_hi(df3 a) { return make_float3(a.x.hi, a.y.hi, a.z.hi); }

// ---------------------------------------------------------------- complex, packed
// A complex double-float as (re, im) pairs of its high and low words, so that the
// two parts share packed FP32 instructions (which run at half the rate of scalar
// ones, two results each, and leave every other issue slot free).
struct cdf2 {
    float2 h, l;
};
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 dup2(float x) { return make_float2(x, x); }
__device__ __forceinline__ cdf2 cdf2_make(df re, df im) { return cdf2{make_float2(re.hi, im.hi), make_float2(re.lo, im.lo)}; }
// acc += u k, with ju = j u: the two products and the two sums of each part
// error-free on the high words, everything below gathered in the low word
// (27 packed instructions, about 2^-47 of the operands)
__device__ __forceinline__ void cdf2_mac(cdf2& acc, const cdf2& u, const cdf2& ju, const cdf2& k) {
    const float2 kr = dup2(k.h.x), ki = dup2(k.h.y);
    const float2 p1 = __fmul2_rn(u.h, kr), p2 = __fmul2_rn(ju.h, ki);
    float2 e = __ffma2_rn(u.h, kr, make_float2(-p1.x, -p1.y));
    e = __ffma2_rn(u.h, dup2(k.l.x), e);
    e = __ffma2_rn(u.l, kr, e);
    e = __ffma2_rn(ju.h, dup2(k.l.y), e);
    e = __ffma2_rn(ju.l, ki, e);
    e = __fadd2_rn(e, __ffma2_rn(ju.h, ki, make_float2(-p2.x, -p2.y)));
    const float2 s1 = __fadd2_rn(acc.h, p1), b1 = sub2(s1, acc.h);
    const float2 t1 = __fadd2_rn(sub2(acc.h, sub2(s1, b1)), sub2(p1, b1));
    const float2 s2 = __fadd2_rn(s1, p2), b2 = sub2(s2, s1);
    const float2 t2 = __fadd2_rn(sub2(s1, sub2(s2, b2)), sub2(p2, b2));
    const float2 lo = __fadd2_rn(__fadd2_rn(acc.l, __fadd2_rn(t1, t2)), e);
    acc.h = __fadd2_rn(s2, lo);
    acc.l = sub2(lo, sub2(acc.h, s2));
}

}  // namespace sbr
