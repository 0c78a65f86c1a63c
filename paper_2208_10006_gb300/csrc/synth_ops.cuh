// Operands of the tensor-core H(f) synthesis (Eq. 13-14), shared by the
// single-receiver and the batched forms so that both compute them with the
// same arithmetic (and therefore give bit-identical H for the same paths).
//
// Layout, for the Pr reflected paths of one receiver padded to Pp (a multiple
// of 8; padded entries are zero):
//   w   [F][Pp]  float2  g_n(f) exp(-j 2 pi f L_n / c), reflected paths only
//   wl  [F]      float2  the same for the LoS path (zero when there is none)
//   sc  [F]      float   FP16 form: the power of two that brings
//                        max_n max(|Re w|, |Im w|) into [1/2, 1) (1 if all zero)
//   dtT [Pp/4][Nt][4] float   |T_p - P1| - |T_0 - P1|   (P1 first interaction point)
//   drT [Pp/4][Nr][4] float   |R_q - Pm| - |R_0 - Pm|   (Pm last interaction point)
//   dl  [dl_size(Nr, Nt)] float, element (q, p) at dl_index: |T_p - R_q| - |T_0 - R_0|,
//                        in blocks of 8 receive x 16 transmit elements as the epilogue
//                        reads them (a lane's four of a block in 16 bytes, a warp's in 512)
// (the delay tables in groups of 4 paths, element-major within a group, so
// that consecutive threads, on consecutive elements, read consecutive 16-byte
// groups)
#pragma once
#include "dfloat.cuh"
#include "sbr_internal.cuh"
#include "synth_index.cuh"

namespace sbr {

constexpr double kInvC0 = 1.0 / kC0;

// g exp(-j 2 pi f L / c). The phase f L / c (up to ~1e6 cycles at THz) is formed in
// double-float, its integer part removed exactly; the rest r = hi + lo with hi the
// FP32 rounding of r; exp(-j 2 pi r) = exp(-j 2 pi hi) (1 - j 2 pi lo) to second
// order in lo (< 1e-13), with the FP32 sine and cosine of pi x (sincospif) for the
// hi part. No FP64 operation: one takes as long as some 70 FP32 ones on this GPU.
//
// Every operation is written with an explicit rounding intrinsic, so that the
// compiler cannot contract a multiply and an add differently in the kernels
// that share these functions (their results must agree bit for bit).
__device__ __forceinline__ float2 synth_weight(float2 g, double f, double L) {
    const df fd = df_split(f), t = df_mul(df_split(L), df{(float)kInvC0, (float)(kInvC0 - (double)(float)kInvC0)});
    const df p = two_prod(fd.hi, t.hi);
    const df r = two_sum(__fsub_rn(p.hi, rintf(p.hi)), __fmaf_rn(fd.hi, t.lo, __fmaf_rn(fd.lo, t.hi, p.lo)));
    float s, c;
    sincospif(__fmul_rn(-2.0f, r.hi), &s, &c);
    const float d = __fmul_rn(-6.283185307179586f, r.lo);   // exp(j d) ~ 1 + j d
    const float cr = __fmaf_rn(-s, d, c), ci = __fmaf_rn(c, d, s);
    return make_float2(__fmaf_rn(g.x, cr, __fmul_rn(-g.y, ci)), __fmaf_rn(g.x, ci, __fmul_rn(g.y, cr)));
}

// the FP16 form's per-frequency scale from the largest weight component
__device__ __forceinline__ float synth_scale(float m) {
    if (!(m > 0.f)) return 1.f;
    int e;
    frexpf(m, &e);
    return ldexpf(1.f, -e);
}

// |a - b| in double-float (relative error about 2^-45)
__device__ __forceinline__ df3 df3_of(d3 v) { return df3{df_split(v.x), df_split(v.y), df_split(v.z)}; }
__device__ __forceinline__ df dist_df(const df3& a, const df3& b) {
    const df3 v = df3_sub(a, b);
    return df_length(df3_dot(v, v));
}

// element delay |E - P| - ref, ref = |E0 - P| = dist_df(E0, P) computed once
// per path, rounded to FP32
__device__ __forceinline__ float el_delay(const double* elem, const df3& P, df ref) {
    return df_sub(dist_df(df3_of(ld3(elem)), P), ref).hi;
}

}  // namespace sbr
