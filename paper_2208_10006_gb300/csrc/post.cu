// Channel statistics (Eq. 2, 4, 5; the Table I quantities) and MIMO capacity
// (Eq. 15-17).
//
// PDP / stats: one block per receiver. tau = L / c, bin floor(tau / bin_s),
// tap = sum |g|^2 (FP64 accumulation), PL_coh from the coherent sum with the
// FP64-reduced delay phase, tau_rms from the power-weighted moments (Eq. 5),
// power-weighted mean AoD/AoA.
//
// Capacity: Eq. 16 multiplies W by Q = sum |h|^2, which read literally drives
// C to zero at realistic path loss; the reading used is the Frobenius
// normalisation W_f = (Nr Nt / Qbar) H_f H_f^H (H_f^H H_f when Nt < Nr),
// Qbar = mean_f ||H_f||_F^2. W_f is formed in FP32 on CUDA cores, then
// log2 det(I + SNR/Nt W_f) from a complex L D L^H factorisation in registers
// (double-float, or FP64 at high SNR); the per-(f, SNR) log-determinants are
// averaged over f in a fixed order.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "dfloat.cuh"
#include "sbr_internal.cuh"

namespace sbr {
namespace {

constexpr int kPdpThreads = 256;

__device__ double block_sum(double v, double* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0) {
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
        sh[32] = t;
    }
    __syncthreads();
    return sh[32];
}

__global__ void __launch_bounds__(kPdpThreads)
k_pdp(const int32_t* __restrict__ rx_off, const double* __restrict__ L, const double* __restrict__ aod,
      const double* __restrict__ aoa, const float2* __restrict__ g, int32_t F, int32_t f_index,
      double fc, double bin_s, int32_t n_bins, float* __restrict__ pdp, double* __restrict__ stats) {
    ::sbr::pdl_wait();
    extern __shared__ double acc[];  // [n_bins]
    const int r = blockIdx.x;
    const int32_t o0 = rx_off[r], o1 = rx_off[r + 1];
    for (int k = threadIdx.x; k < n_bins; k += blockDim.x) acc[k] = 0.0;
    __syncthreads();
    double sp = 0, st = 0, st2 = 0, cr = 0, ci = 0, a1 = 0, a2 = 0, a3 = 0, a4 = 0;
    for (int32_t n = o0 + threadIdx.x; n < o1; n += blockDim.x) {
        float2 gg = g[(int64_t)n * F + f_index];
        double gr = gg.x, gi = gg.y;
        double pw = gr * gr + gi * gi;
        double tau = L[n] / kC0;
        double kb = floor(tau / bin_s);
        if (kb >= 0.0 && kb < (double)n_bins) atomicAdd(&acc[(int)kb], pw);
        sp += pw; st += pw * tau; st2 += pw * tau * tau;
        double cyc = fc * L[n] / kC0;
        double s, c;
        sincospi(-2.0 * (cyc - floor(cyc)), &s, &c);
        cr += gr * c - gi * s;
        ci += gr * s + gi * c;
        a1 += pw * aod[2 * n]; a2 += pw * aod[2 * n + 1];
        a3 += pw * aoa[2 * n]; a4 += pw * aoa[2 * n + 1];
    }
    {
        // the nine block sums at once, each in the order of block_sum (butterfly
        // within each warp, then the warps in order): two barriers instead of 27.
        // A receiver with at most 32 paths has them all in warp 0, whose sums
        // alone are added (the other warps' are exact zeros): the FP64 pipe,
        // this kernel's bound, then carries one warp's butterflies, not eight
        __shared__ double part[kPdpThreads / 32][9];
        __shared__ double tot[9];
        double v[9] = {sp, st, st2, cr, ci, a1, a2, a3, a4};
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const bool one_warp = o1 - o0 <= 32;
        if (!one_warp || warp == 0) {
#pragma unroll
            for (int q = 0; q < 9; ++q)
                for (int o = 16; o; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
            if (lane == 0)
#pragma unroll
                for (int q = 0; q < 9; ++q) part[warp][q] = v[q];
        }
        __syncthreads();
        if (threadIdx.x < 9) {
            double t = 0.0;
            const int nw = one_warp ? 1 : kPdpThreads / 32;
            for (int w = 0; w < nw; ++w) t += part[w][threadIdx.x];
            tot[threadIdx.x] = t;
        }
        __syncthreads();
        sp = tot[0]; st = tot[1]; st2 = tot[2]; cr = tot[3]; ci = tot[4];
        a1 = tot[5]; a2 = tot[6]; a3 = tot[7]; a4 = tot[8];
    }
    // a bin holds a sum of powers (>= 0): its bit pattern is positive exactly when
    // it is non-zero, which keeps the test of the (mostly empty) bins off the FP64 pipe
    for (int k = threadIdx.x; k < n_bins; k += blockDim.x) {
        const double v = acc[k];
        pdp[(int64_t)r * n_bins + k] = __double_as_longlong(v) > 0 ? (float)(10.0 * log10(v)) : -INFINITY;
    }
    if (threadIdx.x == 0) {
        double* o = stats + (int64_t)r * SBR_NSTATS;
        if (o1 == o0 || !(sp > 0.0)) {
            o[0] = INFINITY; o[1] = INFINITY;
            for (int k = 2; k < SBR_NSTATS; ++k) o[k] = NAN;
        } else {
            o[0] = -10.0 * log10(cr * cr + ci * ci);
            o[1] = -10.0 * log10(sp);
            double m1 = st / sp, m2 = st2 / sp, var = m2 - m1 * m1;
            o[2] = sqrt(var > 0.0 ? var : 0.0);
            o[3] = a1 / sp; o[4] = a2 / sp; o[5] = a3 / sp; o[6] = a4 / sp;
        }
    }
}

// ---------------------------------------------------------------- capacity
constexpr int kCapThreads = 256;
constexpr int kMaxSnr = 32;        // SNR values per capacity call
constexpr int kFrobBlocks = 512;   // most partial sums of ||H||^2

// linear SNR values of one capacity call, passed by value in the launch
struct SnrList {
    double lin[kMaxSnr];
};

// sum of |h|^2 over this block's share of H, in double-float: an FP64 addition
// costs some 70 FP32 ones on this GPU, a double-float one about ten, so the
// pass runs at memory speed (H [1024, 64, 256]: 167 us with FP64 sums, 28 us).
// A share with an entry that is not finite, above 2^40 (a thread's sum of 2^47 squares
// stays in the FP32 range), or with none above 2^-40 (where an FP32 product could leave
// the normal range) is summed in FP64.
__global__ void __launch_bounds__(kCapThreads)
k_frob(const float2* __restrict__ H, int64_t n, double* __restrict__ part) {
    ::sbr::pdl_wait();
    __shared__ double sh[33];
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    df s{0.f, 0.f};
    float top = 0.f;
    bool wild = false;
    auto add = [&](float x) {
        const df p = two_prod(x, x);
        const df t = two_sum(s.hi, p.hi);
        s = fast_two_sum(t.hi, __fadd_rn(s.lo, __fadd_rn(t.lo, p.lo)));
        top = fmaxf(top, fabsf(x));
        wild |= !(fabsf(x) < 1.0995116e12f);
    };
    // 16-byte loads of two entries where H starts on 16 bytes
    const bool pairs = (reinterpret_cast<uintptr_t>(H) & 15) == 0;
    const int64_t np = pairs ? n / 2 : 0;
    const float4* H4 = reinterpret_cast<const float4*>(H);
    int64_t i = first;
    for (; i + 3 * step < np; i += 4 * step) {   // four loads in flight
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = __ldg(H4 + i + u * step);
#pragma unroll
        for (int u = 0; u < 4; ++u) { add(v[u].x); add(v[u].y); add(v[u].z); add(v[u].w); }
    }
    for (; i < np; i += step) {
        const float4 v = __ldg(H4 + i);
        add(v.x); add(v.y); add(v.z); add(v.w);
    }
    for (i = 2 * np + first; i < n; i += step) { add(H[i].x); add(H[i].y); }
    const bool plain = !__syncthreads_or(wild) && __syncthreads_or(top > 9.094947e-13f);
    double v = df_to_double(s);
    if (!plain) {
        v = 0.0;
        for (i = first; i < n; i += step) v += (double)H[i].x * H[i].x + (double)H[i].y * H[i].y;
    }
    v = block_sum(v, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = v;
}

// Complex entries of the matrix that is factorised, as double-float pairs
// (.x real, .y imaginary; packed FP32 instructions) or in FP64. Both take 16 bytes.
struct EntryDf {
    cdf2 v;
    struct Row { cdf2 u, ju; };   // -u and its product with the conjugation's sign: acc + u k_re + ju k_im = acc - u conj(k)
    // c w + one
    __device__ __forceinline__ void set(double c, float2 w, float one) {
        const df cd = df_from_double(c);
        v = cdf2_make(df_add(df{one, 0.f}, df_mul_f(cd, w.x)), df_mul_f(cd, w.y));
    }
    // a pivot as kept in shared memory, and its value
    __device__ __forceinline__ double raw() const { return __hiloint2double(__float_as_int(v.h.x), __float_as_int(v.l.x)); }
    static __device__ __forceinline__ double value(double raw) {
        return (double)__int_as_float(__double2hiint(raw)) + (double)__int_as_float(__double2loint(raw));
    }
    struct Inv { df v; };
    __device__ __forceinline__ Inv inverse(unsigned mask, int lane) const {   // that of the given lane's entry
        const df r = df_rcp(df{v.h.x, v.l.x});
        return Inv{df{__shfl_sync(mask, r.hi, lane), __shfl_sync(mask, r.lo, lane)}};
    }
    __device__ __forceinline__ EntryDf scaled(const Inv& inv) const {   // minus the entry over the pivot
        return EntryDf{cdf2_make(df_neg(df_mul(df{v.h.x, v.l.x}, inv.v)), df_neg(df_mul(df{v.h.y, v.l.y}, inv.v)))};
    }
    __device__ __forceinline__ Row row() const { return Row{v, cdf2{make_float2(v.h.y, -v.h.x), make_float2(v.l.y, -v.l.x)}}; }
    __device__ __forceinline__ void update(const Row& u, const EntryDf& k) { cdf2_mac(v, u.u, u.ju, k.v); }
};

struct EntryF64 {
    double re, im;
    struct Row { double re, im; };
    struct Inv { double v; };
    __device__ __forceinline__ void set(double c, float2 w, float one) { re = one + c * w.x; im = c * w.y; }
    __device__ __forceinline__ double raw() const { return re; }
    static __device__ __forceinline__ double value(double raw) { return raw; }
    __device__ __forceinline__ Inv inverse(unsigned mask, int lane) const { return Inv{__shfl_sync(mask, 1.0 / re, lane)}; }
    __device__ __forceinline__ EntryF64 scaled(const Inv& inv) const { return EntryF64{re * inv.v, im * inv.v}; }
    __device__ __forceinline__ Row row() const { return Row{re, im}; }
    __device__ __forceinline__ void update(const Row& u, const EntryF64& k) {
        re -= u.re * k.re + u.im * k.im;
        im -= u.im * k.re - u.re * k.im;
    }
};
static_assert(sizeof(EntryDf) == 16 && sizeof(EntryF64) == 16, "one shared-memory column of 16-byte entries");

__host__ __device__ constexpr int cap_blk(int a, int b) { return a * (a + 1) / 2 + b; }   // block (a, b), a >= b

// column `16 b + (tk = c)` of the block, as its 16 owners (a half warp) publish it for
// the step that eliminates it: the entries, minus the entries over the pivot, the pivot
template <int NB, int b, class E>
__device__ __forceinline__ void ldl_publish(const E (&A)[cap_blk(NB, 0)], int c, E* col, E* row, double* piv) {
    const int ti = threadIdx.x & 15, half = threadIdx.x & 16;
    const typename E::Inv inv = A[cap_blk(b, b)].inverse(0xffffu << half, half | c);
#pragma unroll
    for (int a = b; a < NB; ++a) {
        col[ti + 16 * a] = A[cap_blk(a, b)];
        row[ti + 16 * a] = A[cap_blk(a, b)].scaled(inv);
    }
    if (ti == c) piv[16 * b + c] = A[cap_blk(b, b)].raw();
}

// the columns of block jb (16 jb ...), then those of the blocks after it
template <int NB, int jb, class E>
__device__ __forceinline__ void ldl_block(int n, E (&A)[cap_blk(NB, 0)], E* s_col, double* piv) {
    constexpr int N = 16 * NB;
    const int ti = threadIdx.x & 15, tk = threadIdx.x >> 4;
    for (int jj = 0; jj < 16 && 16 * jb + jj < n; ++jj) {
        const int j = 16 * jb + jj;
        const E *col = s_col + (j & 1) * 2 * N, *row = col + N;
        E* next = s_col + ((j + 1) & 1) * 2 * N;
        typename E::Row u[NB];
#pragma unroll
        for (int a = jb; a < NB; ++a) u[a] = row[ti + 16 * a].row();
#pragma unroll
        for (int b = jb; b < NB; ++b) {
            if (b == jb && (tk | 1) <= jj) continue;   // both columns of this warp are done
            const E k = col[tk + 16 * b];
#pragma unroll
            for (int a = b; a < NB; ++a) A[cap_blk(a, b)].update(u[a], k);
        }
        if (tk == ((jj + 1) & 15)) {
            if (jj < 15) ldl_publish<NB, jb>(A, tk, next, next + N, piv);
            else if constexpr (jb + 1 < NB) ldl_publish<NB, jb + 1>(A, tk, next, next + N, piv);
        }
        __syncthreads();
    }
    if constexpr (jb + 1 < NB) ldl_block<NB, jb + 1, E>(n, A, s_col, piv);
}

// Pivots of the L D L^H factorisation of I + c ws W into piv[0 .. n). Thread
// (ti, tk) of 16 x 16 holds entries (ti + 16 a, tk + 16 b), a >= b, in
// registers; per column one barrier, after which every thread reads the column and
// its scaled form and updates its entries (those above the diagonal and, in a block
// off the column's, left of it are updated too: nothing reads them).
template <int NB, class E>
__device__ __forceinline__ void ldl_pivots(int n, double c, const float2* s_w, float ws, E* s_col, double* piv) {
    constexpr int N = 16 * NB;
    const int ti = threadIdx.x & 15, tk = threadIdx.x >> 4;
    E A[cap_blk(NB, 0)];
#pragma unroll
    for (int a = 0; a < NB; ++a)
#pragma unroll
        for (int b = 0; b <= a; ++b) {
            const float2 w = s_w[cap_blk(a, b) * kCapThreads + threadIdx.x];
            A[cap_blk(a, b)].set(c, make_float2(w.x * ws, w.y * ws), a == b && ti == tk ? 1.f : 0.f);
        }
    if (tk == 0) ldl_publish<NB, 0>(A, 0, s_col, s_col + N, piv);
    __syncthreads();
    ldl_block<NB, 0>(n, A, s_col, piv);
}

// Log-determinants ln det(I + SNR/Nt W_f) of one frequency, n = min(Nr, Nt) <=
// 16 NB <= 64. grid (F, splits): block (f, y) forms W_f and takes the SNRs y,
// y + splits, ...
//
// W[a][b] = sum_p H[a][p] conj(H[b][p])  (Nt >= Nr)  or  sum_q conj(H[q][a]) H[q][b].
// Blocked summation: FP32 partial sums over runs of kCapRun terms, their totals
// in double-float, so the rounding error of an entry grows with the run length
// rather than with the array size (16,384 terms at a 128 x 128 UPA). Each
// thread forms the entries that it later factorises, from a run of H staged in
// shared memory. The factorisation is bound by the FP32 pipe (27 packed
// instructions per entry and column in place of 4 FP64 ones at 1/71 of the FP32
// rate); it runs in double-float while the largest diagonal entry of I + c W is at
// most 2^16: an update rounds 2^-47 of that at most, so that up to 63 of them leave
// 2^-25 of the smallest pivot (>= 1), where the FP32 entries of W carry 2^-9. Above
// (SNRs beyond about 45 dB) it runs in FP64. C from the same W against an FP64
// factorisation: 3e-15 for 0 to 30 dB channels of full rank; of channels of rank one
// and n up to 64, 1e-12 at a diagonal of 2^12, 1e-11 at 2^14, 8e-11 below 2^16 (FP64
// itself, above: 1e-11). The error of C against 64 bits, 1e-10 to 4e-8 from the FP32
// sums of W, is the same as with an FP64 Cholesky.
// H [1024, 64, 256], seven SNRs, the whole call: 15.4 ms with an FP64 Cholesky
// in shared memory (three barriers per column); 1.84 ms with a thread's columns
// across its warp, a reciprocal of the pivot and scaled entries in every thread and
// two blocks an SM; 1.53 with a warp owning two columns, so that it skips the ones
// that are done, and three blocks; 1.35 with the reciprocal by the pivot's owner;
// 1.31 with the scaled column by its owners; 1.29 with four blocks (64 registers).
// The packed instructions left (15 block updates of 64 columns in place of 20) take
// 0.85 ms.
constexpr int kCapRun = 32;

template <int NB>
struct CapShared {
    float2 h[kCapRun][16 * NB + 1];
    float4 col[4 * 16 * NB];
    float2 w[cap_blk(NB, 0) * kCapThreads];
    double piv[16 * NB];
    double scale;
    unsigned top;   // bits of the largest diagonal entry of W
};

// W_f's entries of this thread (rounded to FP32) into sh.w, in the order of ldl_pivots
template <int NB, bool kWide>
__device__ __forceinline__ void gram(const float2* __restrict__ h, int Nt, int n, int len, CapShared<NB>& sh) {
    constexpr int N = 16 * NB, kBlk = cap_blk(NB, 0), kLoad = kCapRun * N / kCapThreads;
    const int tid = threadIdx.x, ti = tid & 15, tk = tid >> 4;
    // entry e of a run is (p, row), consecutive threads along the rows of H
    float2 v[kLoad];
    auto load = [&](int p0) {
#pragma unroll
        for (int k = 0; k < kLoad; ++k) {
            const int e = tid + k * kCapThreads;
            const int r = kWide ? e / kCapRun : e % N, p = p0 + (kWide ? e % kCapRun : e / N);
            v[k] = r < n && p < len ? __ldg(h + (kWide ? (int64_t)r * Nt + p : (int64_t)p * Nt + r)) : make_float2(0.f, 0.f);
        }
    };
    df re[kBlk], im[kBlk];
#pragma unroll
    for (int k = 0; k < kBlk; ++k) re[k] = im[k] = df{0.f, 0.f};
    load(0);
    for (int p0 = 0; p0 < len; p0 += kCapRun) {
#pragma unroll
        for (int k = 0; k < kLoad; ++k) {
            const int e = tid + k * kCapThreads;
            sh.h[kWide ? e % kCapRun : e / N][kWide ? e / kCapRun : e % N] = v[k];
        }
        __syncthreads();
        if (p0 + kCapRun < len) load(p0 + kCapRun);
        float sr[kBlk], si[kBlk];
#pragma unroll
        for (int k = 0; k < kBlk; ++k) sr[k] = si[k] = 0.f;
#pragma unroll 4
        for (int p = 0; p < kCapRun; ++p) {
            float2 x[NB], y[NB];
#pragma unroll
            for (int a = 0; a < NB; ++a) {
                x[a] = sh.h[p][ti + 16 * a];
                y[a] = sh.h[p][tk + 16 * a];
            }
#pragma unroll
            for (int a = 0; a < NB; ++a)
#pragma unroll
                for (int b = 0; b <= a; ++b) {
                    // one fused operation a term, then the sum: with every rounding written out,
                    // since a compiler free to choose the product that is fused chose another
                    // in one of the eight forms (C in the ninth digit of a few antennas)
                    float &r = sr[cap_blk(a, b)], &i = si[cap_blk(a, b)];
                    r = __fadd_rn(r, __fmaf_rn(x[a].x, y[b].x, __fmul_rn(x[a].y, y[b].y)));
                    i = __fadd_rn(i, kWide ? __fmaf_rn(x[a].y, y[b].x, -__fmul_rn(x[a].x, y[b].y))
                                           : __fmaf_rn(x[a].x, y[b].y, -__fmul_rn(x[a].y, y[b].x)));
                }
        }
#pragma unroll
        for (int k = 0; k < kBlk; ++k) {
            re[k] = df_add(re[k], df{sr[k], 0.f});
            im[k] = df_add(im[k], df{si[k], 0.f});
        }
        __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < kBlk; ++k) sh.w[k * kCapThreads + tid] = make_float2(re[k].hi, im[k].hi);
}

template <int NB>
__global__ void __launch_bounds__(kCapThreads, 4)
k_capacity(const float2* __restrict__ H, int32_t Nr, int32_t Nt, const __grid_constant__ SnrList snr, int32_t n_snr,
           const double* __restrict__ part, int32_t n_part, double* __restrict__ ld) {
    ::sbr::pdl_wait();
    extern __shared__ __align__(16) unsigned char smem[];
    CapShared<NB>& sh = *reinterpret_cast<CapShared<NB>*>(smem);
    const int tid = threadIdx.x, ti = tid & 15, tk = tid >> 4;
    const int n = min(Nr, Nt);
    const float2* h = H + (int64_t)blockIdx.x * Nr * Nt;
    if (tid < 32) {   // Qbar = mean over f of ||H_f||^2, from the partial sums of all of H
        double q = 0.0;
        for (int i = tid; i < n_part; i += 32) q += part[i];
        for (int o = 16; o; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
        if (tid == 0) {
            sh.scale = (double)Nr * Nt / (q / gridDim.x);
            sh.top = 0u;
        }
    }
    if (Nt >= Nr) gram<NB, true>(h, Nt, n, Nt, sh);
    else gram<NB, false>(h, Nt, n, Nr, sh);   // at least one barrier in either
    if (ti == tk)
#pragma unroll
        for (int a = 0; a < NB; ++a) atomicMax(&sh.top, __float_as_uint(sh.w[cap_blk(a, a) * kCapThreads + tid].x));
    __syncthreads();
    // W in units of 2^e, its largest entry in [1, 2) (below 1 where it is subnormal), so that
    // neither it nor the factor of an SNR leaves the normal FP32 range whatever the scale of
    // H; as it is where it is zero or not finite
    const int e = (int)((sh.top >> 23) & 0xffu) - 127;
    const float ws = sh.top && e < 128 ? ldexpf(1.f, -e) : 1.f;
    const double scale = sh.scale;
    for (int si = blockIdx.y; si < n_snr; si += gridDim.y) {
        const double c = snr.lin[si] / Nt * scale / ws;
        bool large = false;
        if (ti == tk)
#pragma unroll
            for (int a = 0; a < NB; ++a)
                large |= ti + 16 * a < n && !(1.0 + c * (sh.w[cap_blk(a, a) * kCapThreads + tid].x * ws) <= 65536.0);
        const bool wide = __syncthreads_or(large) != 0;
        if (wide) ldl_pivots<NB>(n, c, sh.w, ws, reinterpret_cast<EntryF64*>(sh.col), sh.piv);
        else ldl_pivots<NB>(n, c, sh.w, ws, reinterpret_cast<EntryDf*>(sh.col), sh.piv);
        // the first warp reads the pivots; the next SNR's are written after a barrier
        // (the first of them by thread 0, of this warp)
        if (tid < 32) {
            double s = 0.0;
            bool bad = false;
            for (int j = tid; j < n; j += 32) {
                const double d = wide ? sh.piv[j] : EntryDf::value(sh.piv[j]);
                bad |= !(d > 0.0);
                s += log(d);
            }
            for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            bad = __any_sync(0xffffffffu, bad);
            if (tid == 0) ld[(int64_t)blockIdx.x * n_snr + si] = bad ? NAN : s;
        }
    }
}

// one block per SNR: the mean over frequencies, in bit/s/Hz
__global__ void __launch_bounds__(kCapThreads)
k_cap_reduce(const double* __restrict__ ld, int32_t F, int32_t n_snr, double* __restrict__ C) {
    ::sbr::pdl_wait();
    __shared__ double sh[33];
    double s = 0.0;
    for (int32_t f = threadIdx.x; f < F; f += blockDim.x) s += ld[(int64_t)f * n_snr + blockIdx.x];
    s = block_sum(s, sh);
    if (threadIdx.x == 0) C[blockIdx.x] = s / F / log(2.0);
}

template <int NB>
sbr_status capacity_launch(const float2* H, int32_t F, int32_t Nr, int32_t Nt, const SnrList& snr, int32_t n_snr,
                           const double* part, int32_t n_part, double* ld, cudaStream_t s) {
    static std::atomic<unsigned long long> attr{0};
    SBR_TRY(set_smem_once((const void*)k_capacity<NB>, (int)sizeof(CapShared<NB>), &attr));
    // one block per frequency while these fill the chip twice over; below, the
    // SNRs of a frequency go to blocks of their own, each of which forms W_f again
    const int splits = std::max(1, std::min<int>(n_snr, 4 * sm_count() / std::max(1, F)));
    ::sbr::note_launch();
    SBR_TRY_CUDA(::sbr::launch_pdl(k_capacity<NB>, dim3((unsigned)F, (unsigned)splits), dim3(kCapThreads),
                                   sizeof(CapShared<NB>), s, H, Nr, Nt, snr, n_snr, part, n_part, ld));
    return SBR_OK;
}

// the three launches of a capacity call: part [kFrobBlocks] and ld [F * n_snr] are scratch
sbr_status capacity_kernels(const float2* H, int32_t F, int32_t Nr, int32_t Nt, const double* snr_db, int32_t n_snr,
                            double* part, double* ld, double* C, cudaStream_t s) {
    // the linear SNR list travels by value in the launch, so the call returns as
    // soon as its work is enqueued (no host table has to outlive it)
    SnrList snr{};
    for (int i = 0; i < n_snr; ++i) snr.lin[i] = std::pow(10.0, snr_db[i] / 10.0);
    const int64_t total = (int64_t)F * Nr * Nt;
    const int n_part = (int)std::min<int64_t>(kFrobBlocks, (total + 2 * kCapThreads - 1) / (2 * kCapThreads));
    ::sbr::note_launch();
    SBR_TRY_CUDA(::sbr::launch_pdl(k_frob, dim3(n_part), dim3(kCapThreads), 0, s, H, total, part));
    const int n = std::min(Nr, Nt);
    if (n <= 16) SBR_TRY(capacity_launch<1>(H, F, Nr, Nt, snr, n_snr, part, n_part, ld, s));
    else if (n <= 32) SBR_TRY(capacity_launch<2>(H, F, Nr, Nt, snr, n_snr, part, n_part, ld, s));
    else if (n <= 48) SBR_TRY(capacity_launch<3>(H, F, Nr, Nt, snr, n_snr, part, n_part, ld, s));
    else SBR_TRY(capacity_launch<4>(H, F, Nr, Nt, snr, n_snr, part, n_part, ld, s));
    ::sbr::note_launch();
    SBR_TRY_CUDA(::sbr::launch_pdl(k_cap_reduce, dim3(n_snr), dim3(kCapThreads), 0, s, ld, F, n_snr, C));
    return SBR_OK;
}

// 10 log10 of a / b for positive normal a and b next to each other (a few percent):
// 20 / ln 10 atanh((a - b) / (a + b)), the difference exact
__device__ __noinline__ float ratio_db_near(double a, double b) {
    const int e = (__double2hiint(b) & 0x7ff00000) - 0x3ff00000;   // b's mantissa in [1, 2)
    const double xa = __hiloint2double(__double2hiint(a) - e, __double2loint(a));
    const double xb = __hiloint2double(__double2hiint(b) - e, __double2loint(b));
    const df s = df_mul(df_split(xa - xb), df_rcp(df_add(df_split(xa), df_split(xb))));
    constexpr double k = 8.685889638065035;   // 20 / ln 10
    const df y = df_mul(s, df{(float)k, (float)(k - (double)(float)k)});
    return __fadd_rn(y.hi, __fmaf_rn(y.hi, __fmul_rn(s.hi, s.hi) * (1.f / 3.f), y.lo));
}
// 10 log10 of a / b for powers (a > 0): in double-float, one FP64 logarithm costs
// some 3000 FP32 slots on this GPU; FP64 where a or b is zero, subnormal or not finite.
// The difference of logarithms is right to 1e-10 dB, next to 0 dB the form above keeps
// the relative precision (the targets of 4096 receivers, 16 taps and 8 frequencies: 43.1 us
// with both, 42.6 us with the difference alone, 46.4 with mantissas divided for every tap).
__device__ __forceinline__ float ratio_db(double a, double b) {
    auto plain = [](double x) { return (unsigned)(__double2hiint(x) - 0x00100000) < 0x7fe00000u; };
    if (!plain(a) || !plain(b)) return (float)(10.0 * log10(a / b));
    const float r = df_mul(df_sub(df_log2(a), df_log2(b)), df{3.01029992f, 3.56040455e-8f}).hi;   // 10 log10 2
    return fabsf(r) < 0.01f ? ratio_db_near(a, b) : r;
}

// surrogate targets of P_n = |g_n(f)|^2, tau_n = L_n / c relative to the first
// arrival: one warp per receiver. Its lanes first compute the delay and the tap
// of one path each (FP64, once for all frequencies), then stand for (slice,
// frequency): nf = the power of two at or above F (at most 32) frequencies and
// 32 / nf slices of the paths, each lane with sums of its own and a column of
// taps in shared memory; the slices are added at the end. Bound by the FP64 pipe
// (nine operations per path and frequency). 4096 receivers x 25 paths x 8
// frequencies: 1436 us with a warp per (receiver, frequency) and butterflies
// over 35 FP64 sums; with the gains of the same paths (2517 us more) the two
// take 103 us now.
constexpr int kTgtWarps = 4;

__global__ void __launch_bounds__(32 * kTgtWarps)
k_surrogate_targets(const int32_t* __restrict__ rx_off, int32_t n_rx, const float2* __restrict__ g,
                    const double* __restrict__ L, int32_t F, int nf, int32_t n_taps, double tap_s, double floor_db,
                    float* __restrict__ out) {
    ::sbr::pdl_wait();
    extern __shared__ double tgt_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double* s_tap = tgt_smem + warp * (32 * n_taps + 48);   // [n_taps][32]
    double* s_t = s_tap + 32 * n_taps;                      // [32]
    int* s_b = reinterpret_cast<int*>(s_t + 32);            // [32]
    const int r = blockIdx.x * kTgtWarps + warp;
    if (r >= n_rx) return;
    const int p0 = rx_off[r], p1 = rx_off[r + 1];
    const int stride = 2 + n_taps;
    float* o = out + (int64_t)r * F * stride;
    if (p1 == p0) {
        for (int64_t k = lane; k < (int64_t)F * stride; k += 32) o[k] = NAN;
        return;
    }
    // lengths are not negative: their bit patterns are ordered as they are
    unsigned long long lmin = ~0ull;
    for (int p = p0 + lane; p < p1; p += 32) lmin = min(lmin, (unsigned long long)__double_as_longlong(L[p]));
    for (int s = 16; s; s >>= 1) lmin = min(lmin, __shfl_xor_sync(0xffffffffu, lmin, s));
    const double tmin = __longlong_as_double((long long)lmin) / kC0;
    const int slices = 32 / nf, fl = lane & (nf - 1), sl = lane / nf;
    for (int f0 = 0; f0 < F; f0 += nf) {
        const int f = f0 + fl;
        for (int k = 0; k < n_taps; ++k) s_tap[32 * k + lane] = 0.0;
        double sp = 0.0, st = 0.0, st2 = 0.0;
        for (int c0 = p0; c0 < p1; c0 += 32) {
            __syncwarp();
            if (c0 + lane < p1) {
                const double t = L[c0 + lane] / kC0 - tmin;
                const double b = floor(t / tap_s);
                s_t[lane] = t;
                s_b[lane] = b >= 0.0 && b < n_taps ? (int)b : -1;
            }
            __syncwarp();
            const int cnt = min(32, p1 - c0);
            if (f < F) {
                for (int k = sl; k < cnt; k += slices) {
                    const float2 gg = __ldg(g + (int64_t)(c0 + k) * F + f);
                    const double pw = (double)gg.x * gg.x + (double)gg.y * gg.y;
                    const double t = s_t[k];
                    const int b = s_b[k];
                    sp += pw;
                    st += pw * t;
                    st2 += pw * t * t;
                    if (b >= 0) s_tap[32 * b + lane] += pw;
                }
            }
        }
        for (int s = nf; s < 32; s <<= 1) {
            sp += __shfl_xor_sync(0xffffffffu, sp, s);
            st += __shfl_xor_sync(0xffffffffu, st, s);
            st2 += __shfl_xor_sync(0xffffffffu, st2, s);
        }
        __syncwarp();
        // slice sl of frequency f: taps sl, sl + slices, ...
        if (f < F) {
            float* of = o + (int64_t)f * stride;
            if (sl == 0) {
                of[0] = -ratio_db(sp, 1.0);
                const double mean = st / sp;
                of[1] = (float)sqrt(fmax(st2 / sp - mean * mean, 0.0));
            }
            for (int k = sl; k < n_taps; k += slices) {
                double v = 0.0;
                for (int q = 0; q < slices; ++q) v += s_tap[32 * k + q * nf + fl];
                of[2 + k] = fmaxf(v > 0.0 ? ratio_db(v, sp) : (float)floor_db, (float)floor_db);
            }
        }
        __syncwarp();
    }
}

}  // namespace

sbr_status pdp_run(const sbr_path_list* pl, const float2* g, int32_t F, int32_t f_index, double fc,
                   double bin_s, int32_t n_bins, float* pdp, double* stats, cudaStream_t s) {
    if (pl->n_rx == 0) return SBR_OK;
    size_t smem = sizeof(double) * (size_t)n_bins;
    if (smem > 48 * 1024)
        SBR_TRY_CUDA(cudaFuncSetAttribute(k_pdp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    ::sbr::note_launch(), (void)::sbr::launch_pdl(k_pdp, dim3(pl->n_rx), dim3(kPdpThreads), smem, s, pl->rx_off, pl->L, pl->aod, pl->aoa, g, F, f_index, fc,
                                               bin_s, n_bins, pdp, stats);
    SBR_TRY_CUDA(cudaGetLastError());
    return SBR_OK;
}

sbr_status surrogate_targets_run(const sbr_path_list* pl, const float2* g, int32_t F, int32_t n_taps,
                                double tap_s, double floor_db, float* out, cudaStream_t s) {
    if (pl->n_rx == 0) return SBR_OK;
    int nf = 1;
    while (nf < F && nf < 32) nf *= 2;
    const size_t smem = sizeof(double) * kTgtWarps * (32 * (size_t)n_taps + 48);   // n_taps <= 32: below 48 KB
    ::sbr::note_launch(), (void)::sbr::launch_pdl(
        k_surrogate_targets, dim3((unsigned)((pl->n_rx + kTgtWarps - 1) / kTgtWarps)), dim3(32 * kTgtWarps), smem, s,
        pl->rx_off, pl->n_rx, g, pl->L, F, nf, n_taps, tap_s, floor_db, out);
    SBR_TRY_CUDA(cudaGetLastError());
    return SBR_OK;
}

sbr_status capacity_run(const float2* H, int32_t F, int32_t Nr, int32_t Nt, const double* snr_db,
                        int32_t n_snr, double* C, cudaStream_t s) {
    double *part, *ld;
    SBR_TRY(dalloc_n(&part, kFrobBlocks, s));
    sbr_status st = dalloc_n(&ld, (size_t)F * n_snr, s);
    if (st == SBR_OK) {
        st = capacity_kernels(H, F, Nr, Nt, snr_db, n_snr, part, ld, C, s);
        dfree(ld, s);
    }
    dfree(part, s);
    return st;
}


// ---------------------------------------------------------------- capacity without allocation
// Some callers cannot allocate device memory once they are running: a host
// framework that owns the whole device memory pool and forbids libraries from
// calling cudaMalloc, or a real-time simulation loop held to a fixed memory
// footprint after start-up. sbr_capacity_noalloc serves them: the same
// kernels as sbr_capacity, with every scratch buffer placed in the fixed
// array below, which each GPU that loads the library holds until the process
// exits (about 1.1 MB).
constexpr int kNoAllocMaxF = 4096;    // frequencies per call
constexpr int kNoAllocMaxSnr = kMaxSnr;  // SNR values per call

struct CapacityScratch {
    double part[kFrobBlocks];                    // partial sums of ||H||_F^2
    double ld[kNoAllocMaxF * kNoAllocMaxSnr];    // ln det per (f, SNR)
};
static __device__ __align__(256) CapacityScratch g_capacity_scratch;

namespace {

std::mutex g_scratch_mu;
CapacityScratch* g_scratch_ptr[256] = {};

// device address of the scratch array on the current device; looked up once
// per device (the first call on a device does it)
sbr_status capacity_scratch(CapacityScratch** out) {
    int dev = 0;
    SBR_TRY_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 256) {
        set_error("device ordinal %d out of range", dev);
        return SBR_ERR_UNSUPPORTED;
    }
    std::lock_guard<std::mutex> lk(g_scratch_mu);
    if (!g_scratch_ptr[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_capacity_scratch);
        if (e != cudaSuccess || p == nullptr) {
            set_error("cudaGetSymbolAddress(capacity scratch) failed: %s", cudaGetErrorString(e));
            return SBR_ERR_CUDA;
        }
        g_scratch_ptr[dev] = static_cast<CapacityScratch*>(p);
    }
    *out = g_scratch_ptr[dev];
    return SBR_OK;
}

}  // namespace

sbr_status capacity_noalloc_run(const float2* H, int32_t F, int32_t Nr, int32_t Nt,
                                const double* snr_db, int32_t n_snr, double* C, cudaStream_t s) {
    if (F > kNoAllocMaxF || n_snr > kNoAllocMaxSnr) {
        set_error("sbr_capacity_noalloc: F = %d and n_snr = %d exceed the fixed scratch (F <= %d, "
                  "n_snr <= %d); use sbr_capacity", F, n_snr, kNoAllocMaxF, kNoAllocMaxSnr);
        return SBR_ERR_INVALID_ARG;
    }
    CapacityScratch* scr = nullptr;
    SBR_TRY(capacity_scratch(&scr));
    // every scratch field read is first written by this call, so nothing has to
    // be cleared
    return capacity_kernels(H, F, Nr, Nt, snr_db, n_snr, scr->part, scr->ld, C, s);
}

}  // namespace sbr
