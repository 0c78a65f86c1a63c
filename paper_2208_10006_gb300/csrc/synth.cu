// MIMO H(f) synthesis on CUDA cores (Eq. 11-14, near-field spherical
// wavefront of Sec. I), the FP32 and FP64 forms.
//
// For the paths of one receiver, with first/last interaction points P1/Pm,
//   H[f,q,p] = sum_n w_n(f) exp(-j 2 pi f (dt_pn + dr_qn) / c),
//   w_n(f)   = g_n(f) exp(-j 2 pi frac(f L_n / c)),
//   dt_pn    = |T_p - P1| - |T_0 - P1|,  dr_qn = |R_q - Pm| - |R_0 - Pm|;
// a LoS path uses dlos_qp = |T_p - R_q| - |T_0 - R_0| instead of dt + dr.
// The phasor of a term is the product of one per (path, receive element) and one
// per (path, transmit element), so that a tile of H costs (Nr + Nt) sines and
// cosines per path and one complex multiply-add per term.
//
// The FP32 form computes in FP32 with phases reduced from double-float
// frequencies, the FP64 form in FP64 throughout (an operation of which takes as long
// as 71 FP32 ones on this GPU).
#include <algorithm>
#include <type_traits>

#include "dfloat.cuh"
#include "sbr_internal.cuh"
#include "synth_ops.cuh"

namespace sbr {

namespace {

// ---------------------------------------------------------------- delays
// |b + e| - |b| = e . (2 b + e) / (|b + e| + |b|) without the cancellation of the
// difference; e and b in double-float
__device__ __forceinline__ df length_change(const df3& b, df b_norm, const df3& e) {
    const df3 a = df3_add(b, e), s = df3_add(a, b);
    const df den = df_add(df_length(df3_dot(a, a)), b_norm);
    return den.hi > 0.f ? df_mul(df3_dot(e, s), df_rcp(den)) : df{0.f, 0.f};
}
__device__ __forceinline__ df3 df3_from(d3 v) { return df3{df_split(v.x), df_split(v.y), df_split(v.z)}; }
__device__ __forceinline__ df df3_norm(const df3& v) { return df_length(df3_dot(v, v)); }

// Element delays of the paths: FP64 (D = double), or as (hi, lo) for the FP32 form,
// where an FP32 delay alone would carry 6e-8 of its cycles into the phase. Thread per
// element over kDelayPaths paths. Double-float: the element's offset from its array's
// reference and each path's vector from the reference to its point are differences
// taken in FP64, the rest is double-float.
template <class D>
struct DelayArgs {
    int64_t P;                // paths
    const int32_t* nb;
    const double* pts;
    const double* R0;         // reference-point form: receiver reference; else null
    const int32_t* rx;        // per-element form: receiver of each path
    const double* rx_xyz;
    d3 T0;
    const double* tx_elem;
    const double* rx_elem;    // reference-point form
    int32_t Nt, Nr;
    D *dt, *dr, *dlos;        // [P][Nt], [P][Nr], [Nr][Nt]
};
constexpr int kDelayThreads = 128, kDelayPaths = 2;

// path blocks in y (then, reference-point form, receive elements in groups of
// kDelayPaths for dlos), elements (transmit, then receive) in x
template <class D>
__global__ void __launch_bounds__(kDelayThreads) k_delays(const __grid_constant__ DelayArgs<D> a) {
    ::sbr::pdl_wait();
    constexpr bool kF64 = std::is_same<D, double>::value;
    __shared__ typename std::conditional<kF64, d3, df3>::type s_b[2][kDelayPaths];   // FP64: the points themselves
    __shared__ typename std::conditional<kF64, double, df>::type s_n[2][kDelayPaths];
    const int64_t blocks = (a.P + kDelayPaths - 1) / kDelayPaths;
    const bool los = (int64_t)blockIdx.y >= blocks;
    const int64_t n0 = ((int64_t)blockIdx.y - (los ? blocks : 0)) * kDelayPaths;
    const d3 R0 = a.R0 ? ld3(a.R0) : mk3(0, 0, 0);
    if (!los && threadIdx.x < 2 * kDelayPaths) {
        const int k = threadIdx.x % kDelayPaths, rx_side = threadIdx.x / kDelayPaths;
        const int64_t n = n0 + k;
        if (n < a.P) {
            const int m = a.nb[n];
            const d3 ref = rx_side ? R0 : a.T0;
            d3 at = ref;
            if (m > 0) at = ld3(a.pts + (n * kKmax + (rx_side ? m - 1 : 0)) * 3);
            else if (a.rx && !rx_side) at = ld3(a.rx_xyz + 3 * (int64_t)a.rx[n]);   // LoS of the path's own receiver
            if constexpr (kF64) {
                s_b[rx_side][k] = at;
                s_n[rx_side][k] = norm(ref - at);
            } else {
                s_b[rx_side][k] = df3_from(ref - at);
                s_n[rx_side][k] = df3_norm(s_b[rx_side][k]);
            }
        }
    }
    __syncthreads();
    const int64_t e = (int64_t)blockIdx.x * kDelayThreads + threadIdx.x;
    const bool rx_side = e >= a.Nt;
    if (e >= (int64_t)a.Nt + (a.R0 && !los ? a.Nr : 0)) return;
    const d3 el = rx_side ? ld3(a.rx_elem + 3 * (e - a.Nt)) : ld3(a.tx_elem + 3 * e);
    df3 off, b;   // double-float: the element's offset, the arrays' distance
    df bn;
    if constexpr (!kF64) off = df3_from(el - (rx_side ? R0 : a.T0));
    if (los) {   // |T_p - R_q| - |T_0 - R_0|
        if constexpr (!kF64) b = df3_from(a.T0 - R0), bn = df3_norm(b);
        for (int64_t q = n0; q < n0 + kDelayPaths && q < a.Nr; ++q) {
            const d3 r = ld3(a.rx_elem + 3 * q);
            if constexpr (kF64) {
                a.dlos[q * a.Nt + e] = norm(el - r) - norm(a.T0 - R0);
            } else {
                const df v = length_change(b, bn, df3_sub(off, df3_from(r - R0)));
                a.dlos[q * a.Nt + e] = make_float2(v.hi, v.lo);
            }
        }
        return;
    }
    for (int k = 0; k < kDelayPaths && n0 + k < a.P; ++k) {
        D* out = rx_side ? a.dr + (n0 + k) * a.Nr + (e - a.Nt) : a.dt + (n0 + k) * a.Nt + e;
        // a LoS path of the reference-point form takes its delay from dlos
        const bool on = a.nb[n0 + k] > 0 || a.rx;
        if constexpr (kF64) {
            *out = on ? norm(el - s_b[rx_side][k]) - s_n[rx_side][k] : 0.0;
        } else {
            const df v = on ? length_change(s_b[rx_side][k], s_n[rx_side][k], off) : df{0.f, 0.f};
            *out = make_float2(v.hi, v.lo);
        }
    }
}

template <class D>
sbr_status delays_run(const DelayArgs<D>& a, cudaStream_t s) {
    const int64_t e = (int64_t)a.Nt + (a.R0 ? a.Nr : 0);
    const int64_t y = (a.P + kDelayPaths - 1) / kDelayPaths + (a.R0 ? (a.Nr + kDelayPaths - 1) / kDelayPaths : 0);
    if (y == 0) return SBR_OK;
    // path groups in slices of at most 65535 (P up to 2^31)
    if (a.R0 && a.Nr > 65535) {
        set_error("synthesis: more than 65535 receive elements");
        return SBR_ERR_CUDA;
    }
    if (y > 65535) {
        DelayArgs<D> part = a;
        const int64_t step = 16384 * (int64_t)kDelayPaths;   // with 32768 groups of receive elements at most
        const double* r0 = a.R0;
        for (int64_t n = 0; n < a.P; n += step) {
            part.P = std::min(step, a.P - n);
            part.nb = a.nb + n;
            part.pts = a.pts + n * kKmax * 3;
            part.rx = a.rx ? a.rx + n : nullptr;
            part.dt = a.dt + n * a.Nt;
            part.dr = a.dr + n * a.Nr;
            part.R0 = r0;
            SBR_TRY(delays_run(part, s));   // (writes dlos again: the same values)
        }
        return SBR_OK;
    }
    ::sbr::note_launch();
    SBR_TRY_CUDA(::sbr::launch_pdl(k_delays<D>, dim3((unsigned)((e + kDelayThreads - 1) / kDelayThreads), (unsigned)y),
                                   dim3(kDelayThreads), 0, s, a));
    return SBR_OK;
}

// ---------------------------------------------------------------- phasors
// cycles f t modulo 1 from double-float factors, in [-0.5, 0.5] and a bit:
// absolute error about 4e-15 of the product (1e6 cycles: 4e-9)
__device__ __forceinline__ df cycles_mod1(df f, df t) {
    const df p = two_prod(f.hi, t.hi);
    return two_sum(__fsub_rn(p.hi, rintf(p.hi)), __fmaf_rn(f.hi, t.lo, __fmaf_rn(f.lo, t.hi, p.lo)));
}
// exp(-j 2 pi x) for x = foc d cycles (foc = f / c), FP32: the nearest multiple of
// a quarter turn is removed exactly (foc d - k / 4 in one fused operation, plus the
// terms of the low words), sine and cosine of the rest (|z| <= pi / 4, up to 0.89 next to
// 2^19 turns, where k comes from a product rounded to 1/8) from their Taylor series
// (remainders below 2e-9, there 8e-9). Phases beyond 2^19 turns are reduced to a turn by
// cycles_mod1.
__device__ __forceinline__ float2 phasor32(df foc, float2 d) {
    const float x4 = 4.f * __fmul_rn(foc.hi, d.x);
    if (!(fabsf(x4) < 2097152.f)) {
        float s, c;
        sincospif(-2.f * cycles_mod1(foc, df{d.x, d.y}).hi, &s, &c);
        return make_float2(c, s);
    }
    const float m = __fadd_rn(x4, 12582912.f);   // 1.5 2^23: the sum's low bits are the integer
    const float k = __fsub_rn(m, 12582912.f);
    const float r = __fmaf_rn(foc.hi, d.y, __fmaf_rn(foc.lo, d.x, __fmaf_rn(foc.hi, d.x, -0.25f * k)));
    const float z = 6.28318531f * r, z2 = z * z;
    float s = fmaf(z2, 2.75573192e-6f, -1.98412698e-4f);
    s = fmaf(s, z2, 8.33333333e-3f);
    s = fmaf(s, z2, -1.66666667e-1f);
    s = fmaf(s * z2, z, z);
    float c = fmaf(z2, -2.75573192e-7f, 2.48015873e-5f);
    c = fmaf(c, z2, -1.38888889e-3f);
    c = fmaf(c, z2, 4.16666667e-2f);
    c = fmaf(c, z2, -0.5f);
    c = fmaf(c, z2, 1.f);
    const int q = __float_as_int(m);
    // exp(-j (z + q pi / 2)): swap for odd q, then the signs
    const float a = (q & 1) ? s : c, b = (q & 1) ? c : s;
    const float re = __int_as_float(__float_as_int(a) ^ (((q + 1) & 2) << 30));
    const float im = __int_as_float(__float_as_int(b) ^ ((~q & 2) << 30));
    return make_float2(re, im);
}

// g exp(-j 2 pi x), x in [-0.5, 0.5] and a bit, rounded once: sine and cosine of the
// rest to a quarter turn with the leading terms of their series in double-float, the
// later ones (below 4e-7 of the sum) in FP32
__device__ __forceinline__ float2 turned(float2 g, df x) {
    const float k = rintf(4.f * x.hi);
    const df z = df_mul(df_add(df{__fmaf_rn(-0.25f, k, x.hi), 0.f}, df{x.lo, 0.f}), df{6.28318548f, -1.74845560e-7f});
    const df z2 = df_mul(z, z);
    const float t = z2.hi;
    float u = fmaf(t, -2.50521084e-8f, 2.75573192e-6f);    // 1/11!, 1/9!
    u = fmaf(u, t, -1.98412698e-4f);                       // 1/7!
    df s = df_add(df{8.33333377e-3f, -4.34617203e-10f}, two_prod(u, t));      // 1/5!
    s = df_fma(df{-0.166666672f, 4.96705379e-9f}, z2, s);                     // 1/3!
    s = df_fma(z, df_mul(z, z2), s);
    u = fmaf(t, 2.08767570e-9f, -2.75573192e-7f);          // 1/12!, 1/10!
    u = fmaf(u, t, 2.48015873e-5f);                        // 1/8!
    df c = df_add(df{-1.38888892e-3f, 3.36310929e-11f}, two_prod(u, t));      // 1/6!
    c = df_fma(df{4.16666679e-2f, -1.24176345e-9f}, z2, c);                   // 1/4!
    c = df_fma(df{-0.5f, 0.f}, z2, c);
    c = df_fma(df{1.f, 0.f}, z2, c);
    const int q = (int)k;
    df a = (q & 1) ? s : c, b = (q & 1) ? c : s;
    if ((q + 1) & 2) a = df_neg(a);
    if (~q & 2) b = df_neg(b);
    const df gx{g.x, 0.f}, gy{g.y, 0.f};
    return make_float2(df_dot2(gx, a, df_neg(gy), b).hi, df_dot2(gx, b, gy, a).hi);
}
__device__ __forceinline__ float2 cmul32(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// the arithmetic of the two forms: C a complex value, D an element delay
struct Form32 {
    using C = float2;
    using D = float2;
    struct Freq { df f, foc; };
    static __device__ __forceinline__ Freq freq(double f) { return Freq{df_split(f), df_split(f * kInvC0)}; }
    static __device__ __forceinline__ C phasor(const Freq& f, float2 d) { return phasor32(f.foc, d); }
    // g exp(-j 2 pi f L / c)
    static __device__ __forceinline__ C weight(float2 g, const Freq& f, double, double L) {
        return turned(g, cycles_mod1(f.f, df_split(L * kInvC0)));
    }
    static __device__ __forceinline__ C mul(C a, C b) { return cmul32(a, b); }
    static __device__ __forceinline__ void mac(C& acc, const C& a, const C& v) {
        acc.x = fmaf(a.x, v.x, fmaf(-a.y, v.y, acc.x));
        acc.y = fmaf(a.x, v.y, fmaf(a.y, v.x, acc.y));
    }
    static __device__ __forceinline__ C zero() { return make_float2(0.f, 0.f); }
    static __device__ __forceinline__ C add(C a, C b) { return make_float2(a.x + b.x, a.y + b.y); }
    static __device__ __forceinline__ float2 out(const C& a) { return a; }
};
struct Form64 {
    using C = double2;
    using D = double;
    struct Freq { double foc; };
    static __device__ __forceinline__ Freq freq(double f) { return Freq{f / kC0}; }
    static __device__ __forceinline__ C turn(double cycles) {
        double s, c;
        sincospi(-2.0 * cycles, &s, &c);
        return make_double2(c, s);
    }
    static __device__ __forceinline__ C phasor(const Freq& f, double d) { return turn(f.foc * d); }
    static __device__ __forceinline__ C weight(float2 g, const Freq&, double f, double L) {
        const double cyc = f * L / kC0;
        return mul(make_double2(g.x, g.y), turn(cyc - floor(cyc)));
    }
    static __device__ __forceinline__ C mul(C a, C b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
    static __device__ __forceinline__ void mac(C& acc, const C& a, const C& v) {
        acc.x = fma(a.x, v.x, fma(-a.y, v.y, acc.x));
        acc.y = fma(a.x, v.y, fma(a.y, v.x, acc.y));
    }
    static __device__ __forceinline__ C zero() { return make_double2(0.0, 0.0); }
    static __device__ __forceinline__ C add(C a, C b) { return make_double2(a.x + b.x, a.y + b.y); }
    static __device__ __forceinline__ float2 out(const C& a) { return make_float2((float)a.x, (float)a.y); }
};

// ---------------------------------------------------------------- reference-point form
// Block: one frequency, 8 RQ receive x 64 transmit elements; G groups of 128
// threads of RQ x 4 outputs each. Paths in chunks of G NC: all threads fill the
// chunk's weighted receive phasors and transmit phasors in shared memory (their
// delays were requested while the previous chunk was summed), then group g runs
// the outer products of its NC paths; the groups' sums are added at the end. The
// LoS path (if any, the first) is added per output. Bound by the FP32 pipe, 4
// operations a term, or the FP64 pipe, where what lies outside H is left out (its
// phasors and terms cost as much as others). RQ follows Nr (the smallest of 1,
// 2, 4, 8 that covers it: rows past Nr are computed for nothing, and a block
// shares its transmit phasors among 8 RQ rows); G follows the number of blocks, up
// to 4, so that few frequencies still fill the SMs with warps.
// Measured: FP32, F 600, 13 x 63, 129 paths: 156 us with a sine and cosine per
// term and eight launches, 35 us so; FP64, F 128, 16 x 64, 63 paths: 572 us with a
// sine and cosine per term, 125 us so.
constexpr int kSynthThreads = 128, kSynthPT = 64;

template <class D>
struct SynthArgs {
    int32_t F, Nr, Nt, Pr;
    const int32_t* nb0;       // reflections of the first path (0: it is the LoS path)
    const double* freqs;
    const float2* g;          // [Pr][F]
    const double* L;
    const D *dt, *dr, *dlos;
    float2* H;
    int32_t p_base;   // first transmit element of this launch
};

template <class M, int RQ, int G>
__global__ void __launch_bounds__(kSynthThreads* G) k_synth(const __grid_constant__ SynthArgs<typename M::D> a) {
    ::sbr::pdl_wait();
    using C = typename M::C;
    constexpr bool kF64 = std::is_same<M, Form64>::value;
    constexpr int QT = 8 * RQ, NC = sizeof(C) == 8 ? 16 : 8, NT = kSynthThreads * G, NCG = NC * G;
    constexpr int kV = NCG * kSynthPT / NT, kA = (NCG * QT + NT - 1) / NT, kW = 128;   // per thread; NCG divides kW
    constexpr int kPhasors = NCG * (QT + kSynthPT), kSums = G > 1 ? QT * kSynthPT : 0;
    __shared__ C s_mem[kPhasors > kSums ? kPhasors : kSums], s_w[kW];
    C* s_a = s_mem;                    // [NCG][QT]
    C* s_v = s_mem + NCG * QT;         // [NCG][kSynthPT]
    const int tid = threadIdx.x, tp = tid & 15, tq = (tid >> 4) & 7, grp = tid / kSynthThreads;
    const int32_t f = blockIdx.x, p0 = a.p_base + blockIdx.y * kSynthPT, q0 = blockIdx.z * QT;
    const double fr = a.freqs[f];
    const typename M::Freq fq = M::freq(fr);
    const int los = a.Pr > 0 && *a.nb0 == 0 ? 1 : 0;
    C acc[RQ][4];
#pragma unroll
    for (int i = 0; i < RQ; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = M::zero();
    float2 dv[kV], da[kA];   // delays of the chunk (FP32)
    const int np = min(kSynthPT, a.Nt - p0), nq = min(QT, a.Nr - q0);   // elements of the tile
    auto request = [&](int n0) {
        if constexpr (!kF64) {
#pragma unroll
            for (int i = 0; i < kV; ++i) {
                const int e = tid + i * NT, n = n0 + e / kSynthPT, x = e % kSynthPT;
                dv[i] = n < a.Pr && x < np ? __ldg(a.dt + (int64_t)n * a.Nt + (p0 + x)) : make_float2(0.f, 0.f);
            }
#pragma unroll
            for (int i = 0; i < kA; ++i) {
                const int e = tid + i * NT, n = n0 + e / QT, x = e % QT;
                da[i] = e < NCG * QT && n < a.Pr && x < nq ? __ldg(a.dr + (int64_t)n * a.Nr + (q0 + x)) : make_float2(0.f, 0.f);
            }
        }
    };
    request(los);
    for (int n0 = los; n0 < a.Pr; n0 += NCG) {
        const int cnt = min(NCG, a.Pr - n0), w0 = (n0 - los) % kW;
        if (w0 == 0) {   // the weights of the next kW paths
            if (n0 > los) __syncthreads();
            if (tid < kW && n0 + tid < a.Pr) s_w[tid] = M::weight(a.g[(int64_t)(n0 + tid) * a.F + f], fq, fr, a.L[n0 + tid]);
        }
        if (n0 == los || w0 == 0) __syncthreads();
        if constexpr (kF64) {   // no lane without a phasor: a sine and cosine of one lane take the pipe for a warp's
            for (int e = tid; e < cnt * (np + nq); e += NT) {
                const bool tx = e < cnt * np;
                const int u = tx ? e : e - cnt * np, k = u / (tx ? np : nq), x = u - k * (tx ? np : nq);
                const C v = M::phasor(fq, tx ? __ldg(a.dt + (int64_t)(n0 + k) * a.Nt + p0 + x) : __ldg(a.dr + (int64_t)(n0 + k) * a.Nr + q0 + x));
                if (tx) s_v[k * kSynthPT + x] = v;
                else s_a[k * QT + x] = M::mul(s_w[w0 + k], v);
            }
        } else {
#pragma unroll
            for (int i = 0; i < kV; ++i)
                if ((tid + i * NT) / kSynthPT < cnt) s_v[tid + i * NT] = M::phasor(fq, dv[i]);
#pragma unroll
            for (int i = 0; i < kA; ++i)
                if ((tid + i * NT) / QT < cnt) s_a[tid + i * NT] = M::mul(s_w[w0 + (tid + i * NT) / QT], M::phasor(fq, da[i]));
        }
        __syncthreads();
        if (n0 + NCG < a.Pr) request(n0 + NCG);
        for (int k = grp * NC; k < min(cnt, grp * NC + NC); ++k) {
            C v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = s_v[k * kSynthPT + tp + 16 * j];
#pragma unroll
            for (int i = 0; i < RQ; ++i) {
                if (kF64 && tq + 8 * i >= nq) continue;
                const C x = s_a[k * QT + tq + 8 * i];
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (!kF64 || 16 * j < np) M::mac(acc[i][j], x, v[j]);
            }
        }
        __syncthreads();
    }
    if (G > 1) {   // the sums of groups 1 .. G - 1 into group 0
        for (int h = 1; h < G; ++h) {
            if (grp == h)
#pragma unroll
                for (int i = 0; i < RQ; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) s_mem[(4 * i + j) * kSynthThreads + tid % kSynthThreads] = acc[i][j];
            __syncthreads();
            if (grp == 0)
#pragma unroll
                for (int i = 0; i < RQ; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = M::add(acc[i][j], s_mem[(4 * i + j) * kSynthThreads + tid]);
            __syncthreads();
        }
        if (grp > 0) return;
    }
    if (los) {
        const C w = M::weight(a.g[f], fq, fr, a.L[0]);
#pragma unroll
        for (int i = 0; i < RQ; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int q = tq + 8 * i, p = tp + 16 * j;
                if (q < nq && p < np)
                    M::mac(acc[i][j], w, M::phasor(fq, __ldg(a.dlos + (int64_t)(q0 + q) * a.Nt + (p0 + p))));
            }
    }
#pragma unroll
    for (int i = 0; i < RQ; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int q = tq + 8 * i, p = tp + 16 * j;
            if (q < nq && p < np) a.H[((int64_t)f * a.Nr + (q0 + q)) * a.Nt + (p0 + p)] = M::out(acc[i][j]);
        }
}

template <class M, int RQ>
sbr_status synth_launch(SynthArgs<typename M::D> a, cudaStream_t s) {
    const int64_t cols = ((int64_t)a.Nt + kSynthPT - 1) / kSynthPT;
    for (int64_t c = 0; c < cols; c += 65535) {   // (a grid's y dimension)
        a.p_base = (int32_t)(c * kSynthPT);
        const dim3 grid((unsigned)a.F, (unsigned)std::min<int64_t>(65535, cols - c), (unsigned)((a.Nr + 8 * RQ - 1) / (8 * RQ)));
        // groups: 32 warps per SM are wanted, a block of one group has four
        const int64_t want = 8 * (int64_t)sm_count() / ((int64_t)grid.x * grid.y * grid.z);
        ::sbr::note_launch();
        if constexpr (RQ <= 2) {   // (48 KB of shared memory)
            if (want >= 4) {
                SBR_TRY_CUDA(::sbr::launch_pdl(k_synth<M, RQ, 4>, grid, dim3(4 * kSynthThreads), 0, s, a));
                continue;
            }
        }
        if (want >= 2) SBR_TRY_CUDA(::sbr::launch_pdl(k_synth<M, RQ, 2>, grid, dim3(2 * kSynthThreads), 0, s, a));
        else SBR_TRY_CUDA(::sbr::launch_pdl(k_synth<M, RQ, 1>, grid, dim3(kSynthThreads), 0, s, a));
    }
    return SBR_OK;
}

// ---------------------------------------------------------------- per-element form
// H[f, q, :] = sum over element q's own paths n of w_n(f) exp(-j 2 pi f dt_np / c):
// nothing is shared between receive elements, so the phasor of every term is
// needed. FP32: a thread holds two transmit elements (so that their phasors
// turn in packed operations: half the issue slots) at kElF consecutive frequencies; the phasor
// at the middle one comes from phasor32, the others by rotating it with
// exp(-j 2 pi df d / c) - 1 (precise for the small step between subcarriers) and that
// of two and four steps, at most three in turn (their roundings add up: eight in turn
// left 1.15e-7 of H from 7 paths, where a sine and cosine per term leaves 8e-8, as
// three do), four operations each instead of a sine and a cosine. That needs equally
// spaced frequencies (to 2^-28 of a cycle over the delay) and a step of at most 1/16
// cycle, tested per path and element; other grids take phasor32
// per term. The paths are summed from the last to the first: they are sorted by
// their reflections, so the strongest come when the sum's rounding matters least.
// Bound by the FP32 pipe, about eleven operations a term: F 512, 64 x 256, 63
// paths per element: 948 us with sincospif per term and an FP64 prologue, 258 us
// so (250 us with eight rotations in turn; with those, 10 us more with one element per
// thread and scalar operations, 21 with every operation packed and the weights doubled
// in shared memory).
// A launch of few warps waits for the chain of one element's paths (0.45 us a path):
// there G groups of 32 threads take a part of the paths each, from the weakest to the
// strongest, and their sums are added at the end.
constexpr int kElF = 16, kElMid = 8, kElPaths = 64, kElMax = 128, kElGroups = 8;

template <class D>
struct ElArgs {
    int32_t F, Nq, Nt;
    const int32_t* rx_off;
    const double* freqs;
    const float2* g;          // [P][F]
    const double* L;
    const D* dt;              // [P][Nt]
    float2* H;
    int32_t p_base;   // first transmit element of this launch
};

// block (elements / 2, G)
template <int G>
__global__ void __launch_bounds__(G > 1 ? 32 * G : kElMax) k_synth_el32(const __grid_constant__ ElArgs<float2> a) {
    ::sbr::pdl_wait();
    __shared__ __align__(16) float2 s_w[kElPaths][kElF];
    __shared__ float s_sum[G > 1 ? G / 2 : 1][4 * kElF][G > 1 ? 32 : 1];
    __shared__ df s_f[kElF], s_foc[kElF], s_t[kElPaths];
    __shared__ float s_step, s_dev;
    __shared__ df s_mid;
    const int grp = G > 1 ? threadIdx.y : 0, tid = grp * blockDim.x + threadIdx.x, threads = G * blockDim.x;
    const int32_t f0 = blockIdx.x * kElF, q = blockIdx.y;
    const uint32_t p0 = a.p_base + blockIdx.z * 2 * blockDim.x + threadIdx.x, p1 = p0 + blockDim.x;   // the two elements (unsigned: past Nt, up to 2^31 and some)
    const int nf = min(kElF, a.F - f0);
    const bool act = p0 < (uint32_t)a.Nt, two = p1 < (uint32_t)a.Nt;
    if (tid < 32) {   // one warp, at least: the block's frequencies
        const double fk = a.freqs[f0 + min(tid, nf - 1)];
        const double first = __shfl_sync(0xffffffffu, fk, 0), last = __shfl_sync(0xffffffffu, fk, nf - 1);
        const double step = nf > 1 ? (last - first) / (nf - 1) : 0.0;
        const double mid = nf > kElMid ? __shfl_sync(0xffffffffu, fk, kElMid) : first + kElMid * step;
        float dev = (float)fabs((fk - mid - (min(tid, nf - 1) - kElMid) * step) * kInvC0);
        if (!(dev == dev)) dev = INFINITY;
        for (int o = 16; o; o >>= 1) dev = fmaxf(dev, __shfl_xor_sync(0xffffffffu, dev, o));
        if (tid < kElF) {
            s_f[tid] = df_split(fk);
            s_foc[tid] = df_split(fk * kInvC0);
        }
        if (tid == 0) {
            s_mid = df_split(mid * kInvC0);
            s_step = (float)(step * kInvC0);
            s_dev = dev;
        }
    }
    const int32_t a0 = a.rx_off[q], a1 = a.rx_off[q + 1];
    float2 re[kElF], im[kElF];   // of the two elements
#pragma unroll
    for (int k = 0; k < kElF; ++k) re[k] = im[k] = make_float2(0.f, 0.f);
    for (int32_t n1 = a1; n1 > a0; n1 -= kElPaths) {   // paths [n0, n1)
        const int cnt = min(kElPaths, n1 - a0);
        const int32_t n0 = n1 - cnt;
        __syncthreads();
        for (int n = tid; n < cnt; n += threads) s_t[n] = df_split(a.L[n0 + n] * kInvC0);
        __syncthreads();
#pragma unroll 4
        for (int e = tid; e < cnt * kElF; e += threads) {
            const int n = e / kElF, k = e % kElF;
            s_w[n][k] = k < nf ? turned(a.g[(int64_t)(n0 + n) * a.F + f0 + k], cycles_mod1(s_f[k], s_t[n])) : make_float2(0.f, 0.f);
        }
        __syncthreads();
        if (!act) continue;
        const float2* dt = a.dt + (int64_t)n0 * a.Nt;
        // this group's paths [c0, c1) of the chunk
        const int part = (cnt + G - 1) / G, c0 = grp * part, c1 = min(cnt, c0 + part);
        if (c0 >= c1) continue;
        // delays two paths ahead
        auto delay = [&](int n, uint32_t p) { return __ldg(dt + (int64_t)max(n, c0) * a.Nt + p); };
        const uint32_t pb = two ? p1 : p0;
        float2 da = delay(c1 - 1, p0), db = delay(c1 - 1, pb), ea = delay(c1 - 2, p0), eb = delay(c1 - 2, pb);
        for (int n = c1 - 1; n >= c0; --n) {
            const float2 d0 = da, d1 = db;
            da = ea, db = eb;
            ea = delay(n - 2, p0), eb = delay(n - 2, pb);
            // scalar operations here: packed ones would need every weight twice, from
            // shared memory (whose loads then bound the loop) or by moves
            const float4* w4 = reinterpret_cast<const float4*>(s_w[n]);   // weights of two frequencies
            auto add = [&](int k, float wx, float wy, float2 vx, float2 vy) {
                re[k].x = fmaf(wx, vx.x, fmaf(-wy, vy.x, re[k].x));
                re[k].y = fmaf(wx, vx.y, fmaf(-wy, vy.y, re[k].y));
                im[k].x = fmaf(wx, vy.x, fmaf(wy, vx.x, im[k].x));
                im[k].y = fmaf(wx, vy.y, fmaf(wy, vx.y, im[k].y));
            };
            auto turn = [&](float2& vx, float2& vy, float2 c, float2 sx, float2 sy) {
                const float2 x = __ffma2_rn(vx, c, __ffma2_rn(vy, sx, vx));
                vy = __ffma2_rn(vx, sy, __ffma2_rn(vy, c, vy));
                vx = x;
            };
            const float dmax = fmaxf(fabsf(d0.x), fabsf(d1.x));
            if (fabsf(s_step) * dmax <= 0.0625f && s_dev * dmax <= 3.7252903e-9f) {
                // rotation by one step: c = cos z - 1, s = -sin z (and the other way round for -z)
                const float2 z = __fmul2_rn(dup2(6.28318531f * s_step), make_float2(d0.x, d1.x)), z2 = __fmul2_rn(z, z);
                float2 c = __ffma2_rn(z2, dup2(2.48015873e-5f), dup2(-1.38888889e-3f));
                c = __ffma2_rn(c, z2, dup2(4.16666667e-2f));
                c = __fmul2_rn(__ffma2_rn(c, z2, dup2(-0.5f)), z2);
                float2 s = __ffma2_rn(z2, dup2(-1.98412698e-4f), dup2(8.33333333e-3f));
                s = __ffma2_rn(s, z2, dup2(-1.66666667e-1f));
                const float2 sp = __ffma2_rn(__fmul2_rn(s, z2), z, z), sn = make_float2(-sp.x, -sp.y);   // sin z, -sin z
                const float2 m0 = phasor32(s_mid, d0), m1 = phasor32(s_mid, d1);
                // by two and four steps: 2 c (2 + c), 2 s (1 + c)
                const float2 c2 = __ffma2_rn(__fadd2_rn(c, c), c, __fmul2_rn(c, dup2(4.f)));
                const float2 sp2 = __ffma2_rn(__fadd2_rn(sp, sp), c, __fadd2_rn(sp, sp)), sn2 = make_float2(-sp2.x, -sp2.y);
                const float2 c4 = __ffma2_rn(__fadd2_rn(c2, c2), c2, __fmul2_rn(c2, dup2(4.f)));
                const float2 sp4 = __ffma2_rn(__fadd2_rn(sp2, sp2), c2, __fadd2_rn(sp2, sp2)), sn4 = make_float2(-sp4.x, -sp4.y);
                float2 bx = make_float2(m0.x, m1.x), by = make_float2(m0.y, m1.y);
                float2 dx = bx, dy = by;
                // upwards from the middle (b, b + 4), then downwards: at most three rotations each
#pragma unroll
                for (int k = 0; k < kElMid; k += 4) {
                    const float4 w0 = w4[(kElMid + k) / 2], w1 = w4[(kElMid + k) / 2 + 1];
                    float2 x1 = bx, y1 = by, x2 = bx, y2 = by;
                    turn(x1, y1, c, sp, sn);
                    turn(x2, y2, c2, sp2, sn2);
                    add(kElMid + k, w0.x, w0.y, bx, by);
                    add(kElMid + k + 1, w0.z, w0.w, x1, y1);
                    add(kElMid + k + 2, w1.x, w1.y, x2, y2);
                    turn(x2, y2, c, sp, sn);
                    if (k + 4 < kElMid) turn(bx, by, c4, sp4, sn4);
                    add(kElMid + k + 3, w1.z, w1.w, x2, y2);
                }
#pragma unroll
                for (int k = kElMid; k > 0; k -= 4) {   // k - 1 ... k - 4
                    const float4 w0 = w4[k / 2 - 1], w1 = w4[k / 2 - 2];
                    float2 x1 = dx, y1 = dy, x2 = dx, y2 = dy;
                    turn(x1, y1, c, sn, sp);
                    turn(x2, y2, c2, sn2, sp2);
                    turn(dx, dy, c4, sn4, sp4);
                    add(k - 1, w0.z, w0.w, x1, y1);
                    add(k - 2, w0.x, w0.y, x2, y2);
                    turn(x2, y2, c, sn, sp);
                    add(k - 4, w1.x, w1.y, dx, dy);
                    add(k - 3, w1.z, w1.w, x2, y2);
                }
            } else {
#pragma unroll
                for (int k = 0; k < kElF; ++k) {
                    const float2 v0 = phasor32(s_foc[k], d0), v1 = phasor32(s_foc[k], d1);
                    add(k, s_w[n][k].x, s_w[n][k].y, make_float2(v0.x, v1.x), make_float2(v0.y, v1.y));
                }
            }
        }
    }
    if constexpr (G > 1) {   // the sums of the groups, pairwise
#pragma unroll 1
        for (int h = G / 2; h >= 1; h /= 2) {
            __syncthreads();
            if (grp >= h && grp < 2 * h)
#pragma unroll
                for (int k = 0; k < kElF; ++k) {
                    float(*o)[32] = &s_sum[grp - h][4 * k];
                    o[0][threadIdx.x] = re[k].x; o[1][threadIdx.x] = re[k].y;
                    o[2][threadIdx.x] = im[k].x; o[3][threadIdx.x] = im[k].y;
                }
            __syncthreads();
            if (grp < h)
#pragma unroll
                for (int k = 0; k < kElF; ++k) {
                    const float(*o)[32] = &s_sum[grp][4 * k];
                    re[k].x += o[0][threadIdx.x]; re[k].y += o[1][threadIdx.x];
                    im[k].x += o[2][threadIdx.x]; im[k].y += o[3][threadIdx.x];
                }
        }
        if (grp > 0) return;
    }
    if (act)
#pragma unroll
        for (int k = 0; k < kElF; ++k)
            if (k < nf) {
                float2* row = a.H + ((int64_t)(f0 + k) * a.Nq + q) * a.Nt;
                row[p0] = make_float2(re[k].x, im[k].x);
                if (two) row[p1] = make_float2(re[k].y, im[k].y);
            }
}

// FP64 form: thread per output, a sine and cosine per term. Blocks no wider than the
// array, as many of them on an SM as fit: the pipe is kept busy by one warp of each.
// F 300, 64 x 64, 63 paths per element: 4860 us with phasors and delays in the same
// arithmetic and the products left to the compiler (six operations), 4645 us with four.
__global__ void __launch_bounds__(kSynthThreads, 16) k_synth_el64(const __grid_constant__ ElArgs<double> a) {
    ::sbr::pdl_wait();
    __shared__ double2 s_w[kSynthThreads];
    const int32_t f = blockIdx.x, q = blockIdx.y;
    const uint32_t p = a.p_base + blockIdx.z * blockDim.x + threadIdx.x;
    const double fr = a.freqs[f];
    const Form64::Freq fq = Form64::freq(fr);
    const int32_t a0 = a.rx_off[q], a1 = a.rx_off[q + 1];
    double2 acc = Form64::zero();
    for (int32_t n0 = a0; n0 < a1; n0 += kSynthThreads) {
        const int cnt = min(kSynthThreads, a1 - n0);
        __syncthreads();
        for (int k = threadIdx.x; k < cnt; k += blockDim.x)
            s_w[k] = Form64::weight(a.g[(int64_t)(n0 + k) * a.F + f], fq, fr, a.L[n0 + k]);
        __syncthreads();
        if (p < (uint32_t)a.Nt)
            for (int k = 0; k < cnt; ++k)
                Form64::mac(acc, s_w[k], Form64::phasor(fq, __ldg(a.dt + (int64_t)(n0 + k) * a.Nt + p)));
    }
    if (p < (uint32_t)a.Nt) a.H[((int64_t)f * a.Nq + q) * a.Nt + p] = Form64::out(acc);
}

template <class D>
sbr_status elements_form(const sbr_path_list* pl, const float2* g, const double* freqs, int32_t F,
                         const double* tx_elem, int32_t Nt, float2* H, cudaStream_t s) {
    constexpr bool fp64 = std::is_same<D, double>::value;
    DelayArgs<D> d{};
    d.P = pl->P;
    d.nb = pl->nb;
    d.pts = pl->pts;
    d.rx = pl->rx;
    d.rx_xyz = pl->rx_xyz;
    d.T0 = mk3(pl->tx[0], pl->tx[1], pl->tx[2]);
    d.tx_elem = tx_elem;
    d.Nt = Nt;
    SBR_TRY(dalloc_n(&d.dt, (size_t)pl->P * Nt, s));
    sbr_status st = delays_run(d, s);
    if (st == SBR_OK) {
        ElArgs<D> a{F, pl->n_rx, Nt, pl->rx_off, freqs, g, pl->L, d.dt, H, 0};
        // FP32: two elements per thread; blocks as wide as the array up to kElMax threads, or of
        // 32 in 2, 4 or 8 groups while the launch has fewer than four warps per scheduler.
        // Whole call, 63 paths per element, warps without groups: 1 to 76 warps 39 us with one
        // group, 24 with two, 16.5 (the host's time) with four or eight (33 to 41 before the
        // rotations, a thread per output then); 304: 39.8, 24.7, 18.5, 17.7; 608: 41.1, 29.7,
        // 26.8, 31.4; 912: 43.7, 37.1, 37.8, 43.8.
        const int64_t warps = ((int64_t)F + kElF - 1) / kElF * pl->n_rx * (((int64_t)Nt + 63) / 64);
        int groups = 1;
        while (!fp64 && groups < kElGroups && warps * groups < 16 * (int64_t)sm_count()) groups *= 2;
        const int width = fp64 ? std::min(kSynthThreads, (Nt + 31) / 32 * 32) : groups > 1 ? 32 : std::min(kElMax, ((Nt + 1) / 2 + 31) / 32 * 32), per = fp64 ? width : 2 * width;
        const int64_t cols = ((int64_t)Nt + per - 1) / per;
        for (int64_t c = 0; c < cols && st == SBR_OK; c += 65535) {   // (a grid's z dimension)
            a.p_base = (int32_t)(c * per);
            const dim3 grid((unsigned)(fp64 ? F : (F + kElF - 1) / kElF), (unsigned)pl->n_rx, (unsigned)std::min<int64_t>(65535, cols - c));
            ::sbr::note_launch();
            cudaError_t e;
            if constexpr (fp64) {
                e = ::sbr::launch_pdl(k_synth_el64, grid, dim3(width), 0, s, a);
            } else {
                const auto kern = groups == 1 ? k_synth_el32<1> : groups == 2 ? k_synth_el32<2> : groups == 4 ? k_synth_el32<4> : k_synth_el32<8>;
                e = ::sbr::launch_pdl(kern, grid, dim3(width, groups), 0, s, a);
            }
            if (e != cudaSuccess) {
                set_error("per-element synthesis: %s", cudaGetErrorString(e));
                st = SBR_ERR_CUDA;
            }
        }
    }
    dfree(d.dt, s);
    return st;
}

template <class D>
sbr_status reference_form(const sbr_path_list* pl, const float2* g, const double* freqs, int32_t F,
                          const double* tx_elem, int32_t Nt, const double* rx_elem, int32_t Nr,
                          int32_t rx_index, float2* H, cudaStream_t s) {
    const int32_t o0 = pl->h_rx_off[rx_index], Pr = pl->h_rx_off[rx_index + 1] - o0;
    DelayArgs<D> d{};
    d.P = Pr;
    d.nb = pl->nb + o0;
    d.pts = pl->pts + (int64_t)o0 * kKmax * 3;
    d.R0 = pl->rx_xyz + 3 * (int64_t)rx_index;
    d.T0 = mk3(pl->tx[0], pl->tx[1], pl->tx[2]);
    d.tx_elem = tx_elem;
    d.rx_elem = rx_elem;
    d.Nt = Nt;
    d.Nr = Nr;
    // the three tables in one allocation
    const size_t nt = (size_t)Pr * Nt, nr = (size_t)Pr * Nr, nl = (size_t)Nr * Nt;
    SBR_TRY(dalloc_n(&d.dt, nt + nr + nl, s));
    d.dr = d.dt + nt;
    d.dlos = d.dr + nr;
    sbr_status st = delays_run(d, s);
    if (st == SBR_OK) {
        // the LoS path (no reflection) sorts first among a receiver's paths; the
        // kernel reads its reflection count on the device
        const SynthArgs<D> a{F, Nr, Nt, Pr, d.nb, freqs, g + (int64_t)o0 * F, pl->L + o0, d.dt, d.dr, d.dlos, H, 0};
        if constexpr (std::is_same<D, double>::value)
            st = Nr <= 8 ? synth_launch<Form64, 1>(a, s) : (Nr <= 16 ? synth_launch<Form64, 2>(a, s) : synth_launch<Form64, 4>(a, s));
        else
            st = Nr <= 8 ? synth_launch<Form32, 1>(a, s)
                         : (Nr <= 16 ? synth_launch<Form32, 2>(a, s)
                                     : (Nr <= 32 ? synth_launch<Form32, 4>(a, s) : synth_launch<Form32, 8>(a, s)));
    }
    dfree(d.dt, s);
    return st;
}

}  // namespace

sbr_status synth_elements_run(const sbr_path_list* pl, const float2* g, const double* freqs, int32_t F,
                              const double* tx_elem, int32_t Nt, bool fp64, float2* H, cudaStream_t s) {
    return fp64 ? elements_form<double>(pl, g, freqs, F, tx_elem, Nt, H, s)
                : elements_form<float2>(pl, g, freqs, F, tx_elem, Nt, H, s);
}

sbr_status synth_simt_run(const sbr_path_list* pl, const float2* g, const double* freqs, int32_t F,
                          const double* tx_elem, int32_t Nt, const double* rx_elem, int32_t Nr,
                          int32_t rx_index, bool fp64, float2* H, cudaStream_t s) {
    return fp64 ? reference_form<double>(pl, g, freqs, F, tx_elem, Nt, rx_elem, Nr, rx_index, H, s)
                : reference_form<float2>(pl, g, freqs, F, tx_elem, Nt, rx_elem, Nr, rx_index, H, s);
}

}  // namespace sbr
