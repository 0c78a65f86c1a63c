// H(f) synthesis on the 5th-generation tensor cores (tcgen05), Eq. 13-14.
//
// For one frequency and the reflected paths n of one receiver,
//   H[q,p] = sum_n A[q,n] V[p,n],  A[q,n] = w_n exp(-j 2 pi f dr_qn / c),
//   V[p,n] = exp(-j 2 pi f dt_pn / c),
// is the complex contraction U diag(w) V^T. It runs as one real GEMM
//   C (2Nr x Nt) = A' (2Nr x 2P) B' (2P x Nt)
// with rows r(q) / i(q) of C the real / imaginary part of H[q, :] and the
// contraction index k = 2n + {0: real, 1: imaginary}:
//   A'[r(q), 2n] =  Re A,  A'[r(q), 2n+1] = -Im A
//   A'[i(q), 2n] =  Im A,  A'[i(q), 2n+1] =  Re A
//   B'[2n, p]    =  Re V,  B'[2n+1, p]    =  Im V;
// in a tile of 64 receive elements, r(q) = 16 (q / 8) + q % 8 and
// i(q) = r(q) + 8 (acc_row).
// Each operand is split x = hi + lo into two 16-bit values and the product is
// taken as hi*hi + hi*lo + lo*hi, accumulated in FP32 in tensor memory. Two
// forms: BF16 (the lo*lo term, ~2^-16 relative, dropped) and FP16 (~2^-22
// relative, with 5 exponent bits: A' is scaled per frequency by a power of two
// that brings max_n |w_n| into [1/2, 1), and the accumulator is scaled back,
// both exactly). The phasors are generated on chip
// (FP32 phase from the prepared delays) straight into 128-byte-swizzled
// K-major shared-memory tiles; one thread of a warp of its own issues tcgen05.mma (M=128, N=256,
// K=16) and commits to an mbarrier; the epilogue reads TMEM with tcgen05.ld
// in the 16-lane shape that gives each thread the real and the imaginary row
// of one receive element, adds the exact per-element LoS term and stores
// complex64.
//
// Every wait on an mbarrier is bounded; on expiry the CTA records
// ST_TIMEOUT, releases its tensor memory and returns.
#include <algorithm>
#include <type_traits>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "batch.cuh"
#include "dfloat.cuh"
#include "tcgen05.cuh"
#include "sbr_internal.cuh"
#include "synth_ops.cuh"

namespace sbr {
namespace {

using namespace tc;

// One CTA per SM: warps [0, 16) generate the operands, [16, 24) are the epilogue,
// the last one issues the MMAs.
constexpr int kGenWarps = 16, kEpiWarps = 8;
constexpr int kGenThreads = 32 * kGenWarps;
constexpr int kMmaWarp = kGenWarps + kEpiWarps;
constexpr int kTcThreads = 32 * (kMmaWarp + 1);
constexpr int kChunkP = 32;      // paths per K-chunk (K = 64 16-bit values = one 128-byte row)
constexpr int kABytes = kTileM * 128;  // 16 KB: 2 x 64 receive elements

// tile of N transmit elements (N = 64, 128 or 256): shared-memory and TMEM sizes.
// Two operand stages (hi/lo of A' and B' each) and two FP32 accumulators, so
// that the phasors of one K-chunk are generated while the tensor core works on
// the previous one and a tile's epilogue runs while the next tile's MMAs do.
template <int kTileN>
struct TcShape {
    static_assert(kTileN == 64 || kTileN == 128 || kTileN == 256, "tile N");
    static constexpr int kBBytes = kTileN * 128;
    static constexpr int kStage = 2 * kABytes + 2 * kBBytes;        // hi/lo of A and B
    static constexpr int kSmemBytes = 2 * kStage + 1024 + 128;      // + alignment + barriers
    static constexpr int kTmemCols = 2 * kTileN;                    // two accumulators
};

// exp(-j 2 pi c) for two phases of c cycles: reduce to [-1/2, 1/2] exactly, then
// the hardware sine/cosine, whose absolute error on [-pi, pi] (below 1e-6) is
// well under the 2^-16 resolution of the BF16 hi/lo operands. The nearest integer
// comes from adding and taking away 1.5 2^23 (rintf is an instruction of the narrow
// pipe that the sine and cosine need); packed operations up to the sine and cosine.
__device__ __forceinline__ void phasor2(float2 cycles, float2& s, float2& c) {
    const float2 m = __fadd2_rn(cycles, make_float2(12582912.f, 12582912.f));
    const float2 k = __fadd2_rn(m, make_float2(-12582912.f, -12582912.f));
    const float2 z = __fmul2_rn(sub2(cycles, k), make_float2(-6.283185307179586f, -6.283185307179586f));
    __sincosf(z.x, &s.x, &c.x);
    __sincosf(z.y, &s.y, &c.y);
}

// Operands of the tensor-core forms (layouts in synth_ops.cuh): reflected
// paths only, transposed and padded to Pp (a multiple of 8) paths per row, so
// that four paths of one element are one 16-byte load; the LoS weight and the
// FP16 scale per frequency come separately.
struct TcArgs {
    // single receiver of one path list
    int32_t F, Nr, Nt;
    int32_t Pr;                // paths of the receiver (LoS included)
    int32_t Pp;                // padded row length of dtT, drT and w
    const int32_t* nb0;        // reflections of the first path: 0 = it is the LoS path
    const double* freqs;
    const float* dtT;          // [Pp/4][Nt][4]
    const float* drT;          // [Pp/4][Nr][4]
    const float2* w;           // [F][Pp]
    const float2* wl;          // [F]
    const float* sc;           // [F]
    const float* dlos;         // [dl_size(Nr, Nt)]
    float2* H;
    unsigned int* status;
    int inject_timeout;        // test-only: wait on a barrier nothing arrives at
    // batched form: items of all jobs of a wave
    const BatchJobDev* jobs;
    const int64_t* item_off;   // [n_jobs + 1] first item of each job
    int32_t n_jobs;
    int64_t items;
    const int32_t* np;         // [n_jobs] paths of each job
    const int32_t* nb;         // reflections per path slot (batch path store)
    int32_t path_cap;          // padded row length of a job's operands
    const float* dt_all;
    const float* dr_all;
    const float* dl_all;
    const float2* w_all;
    const float2* wl_all;
    const float* sc_all;
};

// one output tile: frequency f, receive elements [q0, q0 + 64), transmit
// elements [p0, p0 + N); the reflected paths [0, nrefl) go through the tensor
// cores, the LoS path (if any) is added exactly in the epilogue
struct TcItem {
    int f, q0, p0, Nr, Nt, nrefl, Pp;
    bool los;
    float foc, sc;
    float2 wl;
    const float* dtT;
    const float* drT;
    const float2* wf;          // reflected-path weights of frequency f
    const float* dlos;
    float2* Hf;                // H of frequency f
};

template <bool kBatch, int kTileN>
__device__ __forceinline__ TcItem tc_item(const TcArgs& a, int64_t it) {
    TcItem x;
    int Pr;
    const int32_t* nb0;
    const double* freqs;
    const float2* w;
    const float2* wl;
    const float* sc;
    float2* H;
    if (kBatch) {
        int lo = 0, hi = a.n_jobs - 1;   // the last job whose first item is <= it
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (__ldg(a.item_off + mid) <= it) lo = mid; else hi = mid - 1;
        }
        const BatchJobDev* J = a.jobs + lo;
        it -= __ldg(a.item_off + lo);
        x.Nr = J->Nr; x.Nt = J->Nt;
        Pr = __ldg(a.np + lo);
        nb0 = a.nb + J->path_base;
        freqs = J->freqs;
        x.dtT = a.dt_all + J->dt_base;
        x.drT = a.dr_all + J->dr_base;
        x.dlos = a.dl_all + J->dl_base;
        w = a.w_all + J->w_base;
        wl = a.wl_all + J->wl_base;
        sc = a.sc_all + J->wl_base;
        x.Pp = a.path_cap;
        H = J->H;
    } else {
        x.Nr = a.Nr; x.Nt = a.Nt;
        Pr = a.Pr;
        nb0 = a.nb0;
        freqs = a.freqs;
        x.dtT = a.dtT; x.drT = a.drT; x.dlos = a.dlos;
        w = a.w;
        wl = a.wl;
        sc = a.sc;
        x.Pp = a.Pp;
        H = a.H;
    }
    // 32-bit decode (a job has F * tiles < 2^31 items); every thread of the
    // CTA repeats it, so it stays cheap
    const uint32_t mtiles = tiles_of(x.Nr, 64), ntiles = tiles_of(x.Nt, kTileN);
    const uint32_t per_f = mtiles * ntiles, itu = (uint32_t)it;
    const uint32_t fq = per_f == 1u ? itu : itu / per_f;
    const uint32_t rem = itu - fq * per_f;
    const uint32_t qt = ntiles == 1u ? rem : rem / ntiles;
    x.f = (int)fq;
    x.q0 = (int)qt * 64;
    x.p0 = (int)(rem - qt * ntiles) * kTileN;
    x.los = Pr > 0 && *nb0 == 0;
    x.nrefl = Pr - (x.los ? 1 : 0);
    // f / c in double-float, rounded once (an FP64 product in every thread costs 20
    // clocks a warp on the narrow pipe)
    x.foc = df_mul(df_split(freqs[x.f]), df{(float)kInvC0, (float)(kInvC0 - (double)(float)kInvC0)}).hi;
    x.wf = w + (int64_t)x.f * x.Pp;
    x.wl = wl[x.f];
    x.sc = sc[x.f];
    x.Hf = H + (int64_t)x.f * x.Nr * x.Nt;
    return x;
}

// x = hi + lo for a pair of values, both BF16 or both FP16: the hi and lo
// halves of two K positions packed as two 32-bit words (lower K index in the
// low 16 bits)
template <bool kF16>
__device__ __forceinline__ void split2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
    if (kF16) {
        __half2 h = __floats2half2_rn(x0, x1);
        float2 hf = __half22float2(h);
        __half2 l = __floats2half2_rn(x0 - hf.x, x1 - hf.y);
        hi = *reinterpret_cast<uint32_t*>(&h);
        lo = *reinterpret_cast<uint32_t*>(&l);
    } else {
        __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
        float2 hf = __bfloat1622float2(h);
        __nv_bfloat162 l = __floats2bfloat162_rn(x0 - hf.x, x1 - hf.y);
        hi = *reinterpret_cast<uint32_t*>(&h);
        lo = *reinterpret_cast<uint32_t*>(&l);
    }
}

// byte offset of the 16-byte chunk c (8 K values) of row r in a 128-byte
// swizzled K-major tile (the layout the matrix descriptors describe)
__device__ __forceinline__ uint32_t chunk_off(int r, int c) {
    return (uint32_t)r * 128u + ((uint32_t)(c ^ (r & 7)) << 4);
}

// shared-memory store without a compiler memory barrier: global loads of later
// work may be hoisted above it (the stores stay ordered among the volatile
// statements, and the tensor core reads them only after a proxy fence and a
// barrier)
__device__ __forceinline__ void sts128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d));
}

// what the epilogue of a tile needs
struct TcEpi {
    int q0, p0, Nr, Nt, acc;
    bool los;
    bool full;                 // whole tile inside H, even Nt, aligned rows: no per-output checks
    bool mma;                  // the tile has reflected paths (an accumulator to read)
    float foc, isc;
    float2 wl;                 // LoS weight (unscaled)
    const float* dlos;
    float2* Hf;
};

// Row of the M = 128 accumulator that holds the real (part 0) or imaginary
// (part 1) part of receive element ql of the tile: receive elements come in
// groups of 8, their real rows followed by their imaginary rows, so that one
// 16-lane tensor-memory load hands each thread both parts of one output
__device__ __forceinline__ int acc_row(int ql, int part) { return 16 * (ql >> 3) + 8 * part + (ql & 7); }

// two outputs, (Re, Im) each, from the accumulator words (re, re, im, im)
template <bool kF16, bool kLos>
__device__ __forceinline__ float4 tc_out(const TcEpi& e, const uint32_t* v, float2 dl) {
    float2 re = make_float2(__uint_as_float(v[0]), __uint_as_float(v[1]));
    float2 im = make_float2(__uint_as_float(v[2]), __uint_as_float(v[3]));
    if (kF16) {
        re = __fmul2_rn(re, dup2(e.isc));
        im = __fmul2_rn(im, dup2(e.isc));
    }
    if (kLos) {
        float2 sn, cs;
        phasor2(__fmul2_rn(dup2(e.foc), dl), sn, cs);
        re = __ffma2_rn(dup2(e.wl.x), cs, __ffma2_rn(dup2(-e.wl.y), sn, re));
        im = __ffma2_rn(dup2(e.wl.x), sn, __ffma2_rn(dup2(e.wl.y), cs, im));
    }
    return make_float4(re.x, im.x, re.y, im.y);
}

// Epilogue of one tile in blocks of 16 lanes (8 receive elements) x 32 columns:
// epilogue warp w reads TMEM lanes [32 (w % 4), + 32) (receive elements
// [16 (w % 4), + 16) of the tile), every second block of them; thread t receives,
// for 8 consecutive columns, (Re, Im) of receive element t / 4 at transmit elements
// 2 (t % 4) and + 1. It scales back (FP16 form), adds the exact per-element
// LoS term and writes them as one 16-byte store (four lanes write 64
// contiguous bytes of a row of H).
template <bool kF16, int kTileN, bool kFull, bool kLos>
__device__ __forceinline__ void tc_epilogue(const TcEpi& e, uint32_t tmem, int warp, int lane) {
    constexpr int kJ = kTileN / 32, kBlocks = 2 * kJ, kBs = kEpiWarps / 4;   // blocks; warps that share a quarter's
    const int lg = warp & 3, b0 = warp >> 2;
    const int qa = lane >> 2, pc = 2 * (lane & 3);
    const uint32_t tacc = tmem + (uint32_t)(e.acc * kTileN) + ((uint32_t)(32 * lg) << 16);
    using Off = typename std::conditional<kFull, int, int64_t>::type;   // a full tile's offsets fit 32 bits
    const Off nt16 = (Off)tiles_of(e.Nt, 16);
    const int nr8 = (int)tiles_of(e.Nr, 8);
    const int rows = e.Nr - e.q0, cols = e.Nt - e.p0;   // of H from the tile's first on
    // LoS delays of a block (dl_index): two 16-byte loads, column pairs 0, 8 and 16, 24
    const float4* dl0 = reinterpret_cast<const float4*>(e.dlos) + ((int64_t)(e.q0 / 8 + 2 * lg) * nt16 + e.p0 / 16) * 32 + lane;
    auto load_dl = [&](int b, float4 (&dl)[2]) {
        const int h = b / kJ, j2 = 2 * (b % kJ);
        const bool in = kFull || e.q0 / 8 + 2 * lg + h < nr8;
#pragma unroll
        for (int k = 0; k < 2; ++k)
            dl[k] = kFull || (in && e.p0 / 16 + j2 + k < nt16) ? __ldg(dl0 + (h * nt16 + j2 + k) * 32) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    float2* out = e.Hf + ((int64_t)e.q0 + 16 * lg + qa) * e.Nt + e.p0 + pc;
    float4 next[2];
    if (kLos) load_dl(b0, next);
#pragma unroll 4
    for (int b = b0; b < kBlocks; b += kBs) {
        const int h = b / kJ, jj = b % kJ;
        // the delays of the next block are requested while this one is processed
        float4 dl[2];
        if (kLos) {
            dl[0] = next[0]; dl[1] = next[1];
            if (b + kBs < kBlocks) load_dl(b + kBs, next);
        }
        if (!kFull && (16 * lg + 8 * h >= rows || 32 * jj >= cols)) continue;   // all outside H
        uint32_t v[16];
        if (e.mma) {
            tmem_ld_16x256b_x4(tacc + ((uint32_t)(16 * h) << 16) + (uint32_t)(32 * jj), v);
        } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = 0u;
        }
        const int q = 16 * lg + 8 * h + qa, p0 = 32 * jj + pc;   // within the tile
        float2* row = out + ((Off)(8 * h) * e.Nt + 32 * jj);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 d4 = dl[k / 2];
            const float4 o = tc_out<kF16, kLos>(e, v + 4 * k, k & 1 ? make_float2(d4.z, d4.w) : make_float2(d4.x, d4.y));
            float2* dst = row + 8 * k;
            if (kFull) {   // whole tile inside H, even Nt, aligned rows: no per-output checks
                *reinterpret_cast<float4*>(dst) = o;
            } else if (q < rows && p0 + 8 * k < cols) {
                const bool two = p0 + 8 * k + 1 < cols;
                if (two && ((((uintptr_t)dst) & 15) == 0)) {
                    *reinterpret_cast<float4*>(dst) = o;
                } else {
                    dst[0] = make_float2(o.x, o.y);
                    if (two) dst[1] = make_float2(o.z, o.w);
                }
            }
        }
    }
}

// The roles meet at mbarriers only: the generating warps fill the two operand
// stages (full), the MMA warp consumes them into one of two accumulators (empty,
// acc_full), the epilogue warps empty those (acc_free), so phasors, MMAs and
// output of different tiles run side by side and each role's latencies (loads,
// sine and cosine, shared memory) are covered by the others' work. With all 16
// warps first generating, then writing out, a block barrier per K-chunk between,
// 42% of the issue slots were used. H [1024, 64, 256] from 45 reflected paths and the
// LoS path, whole call: 68.5 us then, 59 with the roles side by side, 55 with packed
// phasors and the operand prologue in double-float, 50 with the LoS delays in the
// epilogue's order and an epilogue per kind of tile (48 before edge tiles had 64-bit
// offsets, for rows of 2^28 elements and more). It is the epilogue that bounds
// it (32 us without; 47 without the B' phasors; 42 without the stores): 16 + 8 warps
// are the split that leaves it 72 registers (8 + 16: 63 us, 16 + 12 with 64: 50).
// Small arrays at 1024 frequencies, where a tile is mostly outside H: 1 x 1 from 6
// reflected paths 39 us with whole tiles generated and written out (29 before the roles), 24
// with what is outside skipped; 13 x 63 from 128 paths 63 (97), 51.
template <bool kF16, bool kBatch, int kTileN>
__global__ void __launch_bounds__(kTcThreads, 1) k_synth_tc(const __grid_constant__ TcArgs a) {
    using Sh = TcShape<kTileN>;
    static_assert(kGenThreads % kTileN == 0 && 64 * (kChunkP / 4) <= kGenThreads, "generation units");
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* bars = (uint64_t*)(smem + 2 * Sh::kStage);
    enum { kFull = 0, kEmpty = 2, kAccFull = 4, kAccFree = 6, kNever = 8, kDrain = 9, kBars = 10 };
    const uint32_t bar0 = smem_u32(bars);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    uint32_t* tmem_slot = (uint32_t*)(bars + kBars);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(Sh::kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int i = 0; i < kBars; ++i)
            mbar_init(bar(i), i < kEmpty ? kGenWarps : i >= kAccFree && i < kNever ? kEpiWarps : 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    // launched as a programmatic dependent of the operand prologue, the
    // prologue above overlaps its tail; its results are read only after this
    // (a no-op for an ordinary launch)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    bool ok = true;
    // injected fault: the first phase of `never` never completes; the bounded
    // wait gives up and the CTA takes the same exit as a real timeout
    if (a.inject_timeout) ok = __syncthreads_or(!mbar_wait(bar(kNever), 0u, 1u << 12)) == 0;

    const int64_t items = kBatch ? a.items
                                 : (int64_t)a.F * tiles_of(a.Nr, 64) * tiles_of(a.Nt, kTileN);
    auto wait = [&](int i, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait(bar(i), parity)) != 0; };
    uint32_t chunk = 0;   // chunks so far (operand stage and its phase)
    uint32_t tile = 0;    // tiles with MMAs so far (accumulator and its phase)
    if (warp < kGenWarps) {
        for (int64_t it = blockIdx.x; it < items && ok; it += gridDim.x) {
            const TcItem x = tc_item<kBatch, kTileN>(a, it);
            // FP16 form: the power-of-two scale of this frequency's weights (exact)
            const float sc = kF16 ? x.sc : 1.f;
            for (int nb = 0; nb < x.nrefl; nb += kChunkP, ++chunk) {
                const int st = chunk & 1;
                const uint32_t sA_hi = smem_u32(smem) + st * Sh::kStage, sA_lo = sA_hi + kABytes;
                const uint32_t sB_hi = sA_hi + 2 * kABytes, sB_lo = sB_hi + Sh::kBBytes;
                const int cnt = min(kChunkP, x.nrefl - nb);
                const int n16 = 2 * ((cnt + 7) >> 3);   // 16-byte chunks per row (4 paths each), whole MMA K-steps
                // B' (stored N x K): transmit element p, paths nb + 4 c16 .. + 3
                // (padded paths have zero weight, so their phasors are harmless; elements
                // past Nt or Nr are left as they are: their row of an operand reaches only
                // their own row or column of the accumulator, which nothing stores);
                // kGenThreads is a multiple of N, so a thread keeps its element and
                // steps through the chunks. [Pp / 4][Nt] groups of 4 paths:
                // consecutive lanes read consecutive 16-byte groups
                constexpr int kStep = kGenThreads / kTileN, kUnits = 8 / kStep;
                const int pl = tid % kTileN;
                const bool p_in = pl < x.Nt - x.p0;
                const float4* src = reinterpret_cast<const float4*>(x.dtT) + (int64_t)(nb >> 2) * x.Nt + (p_in ? x.p0 + pl : 0);
                // A': receive element q, paths nb + 4 c16 .. + 3 (at most 64 x 8
                // units: one per thread); consecutive lanes take consecutive receive
                // elements (rows r(q) & 7 = q & 7), so that a quarter warp's 16-byte
                // stores land in 8 distinct bank groups of the swizzled rows and a
                // warp shares its weights
                const int ql = tid & 63, qc = tid >> 6, n = nb + 4 * qc;
                const bool q_in = ql < x.Nr - x.q0;
                // every load of the chunk before the wait for its stage
                float4 dt[kUnits], dr = make_float4(0.f, 0.f, 0.f, 0.f), w01 = dr, w23 = dr;
#pragma unroll
                for (int u = 0; u < kUnits; ++u) {
                    const int c16 = tid / kTileN + u * kStep;
                    dt[u] = p_in && c16 < n16 ? __ldg(src + (int64_t)c16 * x.Nt) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
                if (qc < n16 && q_in) {
                    dr = __ldg(reinterpret_cast<const float4*>(x.drT) + (int64_t)(n >> 2) * x.Nr + (x.q0 + ql));
                    w01 = __ldg(reinterpret_cast<const float4*>(x.wf + n));
                    w23 = __ldg(reinterpret_cast<const float4*>(x.wf + n + 2));
                }
                // the stage is free once the MMAs of its previous chunk have completed
                if (chunk >= 2 && !(ok = wait(kEmpty + st, (chunk / 2 - 1) & 1u))) break;
#pragma unroll
                for (int u = 0; u < kUnits; ++u) {
                    const int c16 = tid / kTileN + u * kStep;
                    if (c16 < n16 && p_in) {
                        uint32_t h[4], l[4];
#pragma unroll
                        for (int k = 0; k < 4; k += 2) {
                            float2 sn, cs;
                            phasor2(__fmul2_rn(dup2(x.foc), k ? make_float2(dt[u].z, dt[u].w) : make_float2(dt[u].x, dt[u].y)), sn, cs);
                            split2<kF16>(cs.x, sn.x, h[k], l[k]);
                            split2<kF16>(cs.y, sn.y, h[k + 1], l[k + 1]);
                        }
                        const uint32_t o = chunk_off(pl, c16);
                        sts128(sB_hi + o, h[0], h[1], h[2], h[3]);
                        sts128(sB_lo + o, l[0], l[1], l[2], l[3]);
                    }
                }
                // A' as the two rows r(q) (Re A, -Im A) and i(q) (Im A, Re A)
                if (qc < n16 && q_in) {
                    float sn[4], cs[4];
#pragma unroll
                    for (int k = 0; k < 4; k += 2) {
                        float2 s2, c2;
                        phasor2(__fmul2_rn(dup2(x.foc), k ? make_float2(dr.z, dr.w) : make_float2(dr.x, dr.y)), s2, c2);
                        sn[k] = s2.x; sn[k + 1] = s2.y; cs[k] = c2.x; cs[k + 1] = c2.y;
                    }
                    const float wr[4] = {w01.x, w01.z, w23.x, w23.z};
                    const float wi[4] = {w01.y, w01.w, w23.y, w23.w};
                    uint32_t h0[4], l0[4], h1[4], l1[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float ar = (wr[k] * cs[k] - wi[k] * sn[k]) * sc;
                        const float ai = (wr[k] * sn[k] + wi[k] * cs[k]) * sc;
                        split2<kF16>(ar, -ai, h0[k], l0[k]);
                        // row i(q) holds (Im A, Re A): the same halves swapped, with
                        // the sign of -Im A flipped (rounding to nearest is symmetric,
                        // so these are the bits of a split of (ai, ar))
                        h1[k] = __byte_perm(h0[k], 0u, 0x1032) ^ 0x8000u;
                        l1[k] = __byte_perm(l0[k], 0u, 0x1032) ^ 0x8000u;
                    }
                    const uint32_t o0 = chunk_off(acc_row(ql, 0), qc), o1 = chunk_off(acc_row(ql, 1), qc);
                    sts128(sA_hi + o0, h0[0], h0[1], h0[2], h0[3]);
                    sts128(sA_lo + o0, l0[0], l0[1], l0[2], l0[3]);
                    sts128(sA_hi + o1, h1[0], h1[1], h1[2], h1[3]);
                    sts128(sA_lo + o1, l1[0], l1[1], l1[2], l1[3]);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kFull + st));
            }
        }
    } else if (warp == kMmaWarp) {
        // the whole warp walks the loop, so that descriptors and addresses stay in
        // uniform registers; one elected lane issues
        const bool lead = elect_one();
        const uint64_t dA = make_desc(smem_u32(smem)), dB = make_desc(smem_u32(smem) + 2 * kABytes);
        for (int64_t it = blockIdx.x; it < items && ok; it += gridDim.x) {
            const TcItem x = tc_item<kBatch, kTileN>(a, it);
            if (x.nrefl <= 0) continue;
            const int acc = tile & 1;
            const uint32_t d = tmem + (uint32_t)(acc * kTileN);
            // the accumulator is free once the epilogue of its previous tile has read it
            if (tile >= 2 && !(ok = wait(kAccFree + acc, (tile / 2 - 1) & 1u))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int nb = 0; nb < x.nrefl; nb += kChunkP, ++chunk) {
                const int st = chunk & 1;
                const int nks = (min(kChunkP, x.nrefl - nb) + 7) >> 3;   // MMA K-steps (8 paths each)
                if (!(ok = wait(kFull + st, (chunk / 2) & 1u))) break;
                // the generating warps' stores become visible to the tensor core by one
                // proxy fence here, on the path from them to its reads
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                if (lead) {
                    const uint64_t so = (uint64_t)(st * (Sh::kStage >> 4));
                    for (int ks = 0; ks < nks; ++ks) {
                        const uint64_t o = so + (uint64_t)(2 * ks);   // 16 K values
                        mma_16<kF16, kTileN>(d, dA + o, dB + o, (nb > 0 || ks > 0) ? 1u : 0u);
                        mma_16<kF16, kTileN>(d, dA + o, dB + o + (Sh::kBBytes >> 4), 1u);
                        mma_16<kF16, kTileN>(d, dA + o + (kABytes >> 4), dB + o, 1u);
                    }
                    mma_commit(bar(kEmpty + st));
                    if (nb + kChunkP >= x.nrefl) mma_commit(bar(kAccFull + acc));
                }
                __syncwarp();
            }
            ++tile;
        }
    } else {
        for (int64_t it = blockIdx.x; it < items && ok; it += gridDim.x) {
            const TcItem x = tc_item<kBatch, kTileN>(a, it);
            TcEpi e;
            e.q0 = x.q0; e.p0 = x.p0; e.Nr = x.Nr; e.Nt = x.Nt; e.los = x.los;
            e.acc = tile & 1;
            e.mma = x.nrefl > 0;
            e.foc = x.foc;
            e.isc = kF16 ? 1.f / x.sc : 1.f;   // exact: sc is a power of two
            e.wl = x.wl;
            e.dlos = x.dlos; e.Hf = x.Hf;
            e.full = x.Nr - x.q0 >= 64 && x.Nt - x.p0 >= kTileN && (x.Nt & 1) == 0 && (((uintptr_t)x.Hf) & 15) == 0 &&
                     x.Nt < (1 << 26);   // 32-bit offsets within the tile
            if (e.mma) {
                if (!(ok = wait(kAccFull + e.acc, (tile / 2) & 1u))) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            }
            if (!e.full) {
                if (e.los) tc_epilogue<kF16, kTileN, false, true>(e, tmem, warp - kGenWarps, lane);
                else tc_epilogue<kF16, kTileN, false, false>(e, tmem, warp - kGenWarps, lane);
            } else {
                if (e.los) tc_epilogue<kF16, kTileN, true, true>(e, tmem, warp - kGenWarps, lane);
                else tc_epilogue<kF16, kTileN, true, false>(e, tmem, warp - kGenWarps, lane);
            }
            if (e.mma) {
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kAccFree + e.acc));
                ++tile;
            }
        }
    }
    const bool failed = __syncthreads_or(!ok) != 0;
    // every MMA this CTA issued has completed before its tensor memory is freed
    // (bounded wait; on a normal exit the last epilogue has already seen them)
    if (warp == kMmaWarp) {
        if (elect_one()) mma_commit(bar(kDrain));
        __syncwarp();
        const bool drained = wait(kDrain, 0u);
        if ((failed || !drained) && lane == 0) atomicOr(a.status, (unsigned)ST_TIMEOUT);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Sh::kTmemCols));
    }
}

// Operands of the tensor-core forms in one launch (layouts in synth_ops.cuh):
// blocks [0, nbw) compute the weights, one warp per frequency (the FP16 scale
// is that warp's maximum); the other blocks compute the element delays, one
// thread per path and group of kPrepG elements (per transmit element and
// group of kPrepG receive elements for the LoS delays), the reference
// distance once per thread. Double-float throughout: it is a chain of latencies,
// so blocks of kPrepThreads threads spread it over every SM.
constexpr int kPrepThreads = 128;
constexpr int kPrepG = 2;
struct TcPrep {
    int32_t Pr, Pp, Nt, Nr, F, nbw;
    const int32_t* nb;       // [Pr] reflections of the receiver's paths
    const double* pts;       // [Pr][kKmax][3]
    const double* L;         // [Pr]
    const float2* g;         // [Pr][F]
    const double* freqs;
    const double* tx_elem;
    const double* rx_elem;
    const double* R0;
    d3 T0;
    float* dtT;              // [Pp/4][Nt][4] (synth_ops.cuh)
    float* drT;              // [Pp/4][Nr][4]
    float* dlos;
    float2* w;
    float2* wl;
    float* sc;
};

__global__ void k_tc_prep(const __grid_constant__ TcPrep a) {
    // the synthesis kernel that follows may start its prologue now (it waits
    // for this grid's results before it reads them)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int n0 = (a.Pr > 0 && a.nb[0] == 0) ? 1 : 0;   // the LoS path sorts first
    const int nrefl = a.Pr - n0;
    if ((int)blockIdx.x < a.nbw) {
        const int f = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
        if (f >= a.F) return;
        const double fr = a.freqs[f];
        float m = 0.f;
        // index Pp is the LoS weight, taken by a lane of the last round (often
        // an idle one) instead of after the reduction
        for (int n = lane; n <= a.Pp; n += 32) {
            if (n == a.Pp) {
                a.wl[f] = n0 ? synth_weight(a.g[f], fr, a.L[0]) : make_float2(0.f, 0.f);
                continue;
            }
            float2 ww = make_float2(0.f, 0.f);
            if (n < nrefl) ww = synth_weight(a.g[(int64_t)(n + n0) * a.F + f], fr, a.L[n + n0]);
            a.w[(int64_t)f * a.Pp + n] = ww;
            m = fmaxf(m, fmaxf(fabsf(ww.x), fabsf(ww.y)));
        }
        for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) a.sc[f] = synth_scale(m);
        return;
    }
    // delays; consecutive threads write consecutive words of a row
    const int64_t gt = tiles_of(a.Nt, kPrepG), gr = tiles_of(a.Nr, kPrepG);
    const int64_t n_dt = (int64_t)a.Pp * gt, n_dr = (int64_t)a.Pp * gr, n_dl = (int64_t)a.Nt * gr;
    const int64_t total = n_dt + n_dr + n_dl;
    const int64_t stride = (int64_t)(gridDim.x - a.nbw) * blockDim.x;
    for (int64_t t = (int64_t)(blockIdx.x - a.nbw) * blockDim.x + threadIdx.x; t < total; t += stride) {
        if (t < n_dr + n_dt) {
            const bool tx = t < n_dt;
            const int64_t u = tx ? t : t - n_dt;
            const int n = (int)(u % a.Pp), e0 = (int)(u / a.Pp) * kPrepG;
            const int ne = tx ? a.Nt : a.Nr, left = ne - e0;
            const double* elem = tx ? a.tx_elem : a.rx_elem;
            // element e, path n at [n / 4][e][n % 4]
            float* dst = (tx ? a.dtT : a.drT) + (int64_t)(n >> 2) * ne * 4 + (n & 3);
            if (n < nrefl) {
                const int i = n + n0, m = a.nb[i];
                const df3 P = df3_of(ld3(a.pts + ((int64_t)i * kKmax + (tx ? 0 : m - 1)) * 3));
                const df ref = dist_df(df3_of(tx ? a.T0 : ld3(a.R0)), P);
#pragma unroll
                for (int k = 0; k < kPrepG; ++k)
                    if (k < left) dst[((int64_t)e0 + k) * 4] = el_delay(elem + xyz_at(e0 + k), P, ref);
            } else {
#pragma unroll
                for (int k = 0; k < kPrepG; ++k)
                    if (k < left) dst[((int64_t)e0 + k) * 4] = 0.f;
            }
        } else {
            const int64_t u = t - n_dt - n_dr;
            const int p = (int)(u % a.Nt), q0 = (int)(u / a.Nt) * kPrepG;
            const df ref = dist_df(df3_of(a.T0), df3_of(ld3(a.R0)));
#pragma unroll
            for (int k = 0; k < kPrepG; ++k)
                if (k < a.Nr - q0)
                    a.dlos[dl_index(q0 + k, p, a.Nt)] = el_delay(a.tx_elem + xyz_at(p), df3_of(ld3(a.rx_elem + xyz_at(q0 + k))), ref);
        }
    }
}

inline unsigned blocks_of(int64_t n, int threads) {
    return (unsigned)std::max<int64_t>(1, (n + threads - 1) / threads);
}

}  // namespace

sbr_status synth_tc_run(const sbr_path_list* pl, const float2* g, const double* freqs, int32_t F,
                        const double* tx_elem, int32_t Nt, const double* rx_elem, int32_t Nr,
                        int32_t rx_index, float2* H, bool f16, cudaStream_t s) {
    const int32_t o0 = pl->h_rx_off[rx_index], Pr = pl->h_rx_off[rx_index + 1] - o0;
    const int32_t Pp = (int32_t)std::max<int64_t>(8, ((int64_t)Pr + 7) & ~(int64_t)7);   // reflected paths, padded
    // one buffer for every operand, 16-byte aligned parts: w, wl (8-byte
    // elements) first, then sc, dtT, drT, dlos
    const size_t n_w = (size_t)Pp * F, n_wl = ((size_t)F + 1) & ~(size_t)1;
    const size_t n_sc = ((size_t)F + 3) & ~(size_t)3;
    const size_t n_f = n_sc + (size_t)Pp * Nt + (size_t)Pp * Nr + (size_t)dl_size(Nr, Nt);
    float2* w;
    SBR_TRY(dalloc_n(&w, n_w + n_wl + (n_f + 1) / 2, s));
    float2* wl = w + n_w;
    float* sc = reinterpret_cast<float*>(wl + n_wl);
    float* dtT = sc + n_sc;
    float* drT = dtT + (size_t)Pp * Nt;
    float* dl = drT + (size_t)Pp * Nr;
    TcPrep pp{};
    pp.Pr = Pr; pp.Pp = Pp; pp.Nt = Nt; pp.Nr = Nr; pp.F = F;
    pp.nb = pl->nb + o0;
    pp.pts = pl->pts + (int64_t)o0 * kKmax * 3;
    pp.L = pl->L + o0;
    pp.g = g + (int64_t)o0 * F;
    pp.freqs = freqs; pp.tx_elem = tx_elem; pp.rx_elem = rx_elem;
    pp.R0 = pl->rx_xyz + xyz_at(rx_index);
    pp.T0 = mk3(pl->tx[0], pl->tx[1], pl->tx[2]);
    pp.dtT = dtT; pp.drT = drT; pp.dlos = dl; pp.w = w; pp.wl = wl; pp.sc = sc;
    pp.nbw = (int)blocks_of((int64_t)F * 32, kPrepThreads);
    const int64_t gt = tiles_of(Nt, kPrepG), gr = tiles_of(Nr, kPrepG);
    const int64_t n_del = (int64_t)Pp * (gt + gr) + (int64_t)Nt * gr;
    const unsigned nbd = (unsigned)std::min<int64_t>(blocks_of(n_del, kPrepThreads), 32 * (int64_t)sm_count());
    ::sbr::note_launch(), k_tc_prep<<<(unsigned)pp.nbw + nbd, kPrepThreads, 0, s>>>(pp);
    SBR_TRY_CUDA(cudaGetLastError());
    TcArgs a{};
    a.F = F; a.Nr = Nr; a.Nt = Nt;
    a.Pr = Pr; a.Pp = Pp;
    a.nb0 = pl->nb + o0;
    a.freqs = freqs; a.dtT = dtT; a.drT = drT; a.w = w; a.wl = wl; a.sc = sc; a.dlos = dl; a.H = H;
    a.status = pl->d_status;  // a bounded wait that gave up is reported by sbr_path_query
    a.inject_timeout = fault_mode() == kFaultTimeout ? 1 : 0;
    auto kern = f16 ? k_synth_tc<true, false, 256> : k_synth_tc<false, false, 256>;
    constexpr int kSmemBytes = TcShape<256>::kSmemBytes;
    SBR_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
    int64_t items = (int64_t)F * tiles_of(Nr, 64) * tiles_of(Nt, 256);
    // one persistent CTA per SM (two operand stages and two accumulators each),
    // launched as a programmatic dependent of the prologue
    const int grid = (int)std::min<int64_t>(items, (int64_t)sm_count());
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kTcThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    ::sbr::note_launch();
    SBR_TRY_CUDA(cudaLaunchKernelEx(&cfg, kern, a));
    dfree(w, s);
    return SBR_OK;
}

namespace {
template <bool kF16, int kTileN>
sbr_status batch_tc_launch(const BatchSynthWave& w, cudaStream_t s) {
    TcArgs a{};
    a.jobs = w.jobs;
    a.item_off = w.item_off;
    a.n_jobs = w.n_jobs;
    a.items = w.items;
    a.np = w.np;
    a.nb = w.nb;
    a.path_cap = w.path_cap;
    a.dt_all = w.dt;
    a.dr_all = w.dr;
    a.dl_all = w.dl;
    a.w_all = w.w;
    a.wl_all = w.wl;
    a.sc_all = w.sc;
    a.status = w.status;
    a.inject_timeout = fault_mode() == kFaultTimeout ? 1 : 0;
    if (w.items <= 0) return SBR_OK;
    int grid = (int)std::min<int64_t>(w.items, (int64_t)sm_count());
    ::sbr::note_launch(), k_synth_tc<kF16, true, kTileN><<<grid, kTcThreads, TcShape<kTileN>::kSmemBytes, s>>>(a);
    SBR_TRY_CUDA(cudaGetLastError());
    return SBR_OK;
}

template <bool kF16, int kTileN>
sbr_status batch_tc_attr() {
    SBR_TRY_CUDA(cudaFuncSetAttribute(k_synth_tc<kF16, true, kTileN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      TcShape<kTileN>::kSmemBytes));
    return SBR_OK;
}
}  // namespace

sbr_status batch_synth_prepare(bool f16, int tile_n) {
    switch (tile_n) {
        case 64: return f16 ? batch_tc_attr<true, 64>() : batch_tc_attr<false, 64>();
        case 128: return f16 ? batch_tc_attr<true, 128>() : batch_tc_attr<false, 128>();
        case 256: return f16 ? batch_tc_attr<true, 256>() : batch_tc_attr<false, 256>();
        default: set_error("tile_n %d not in {64, 128, 256}", tile_n); return SBR_ERR_INVALID_ARG;
    }
}

sbr_status batch_synth_tc(const BatchSynthWave& w, bool f16, int tile_n, cudaStream_t s) {
    switch (tile_n) {
        case 64: return f16 ? batch_tc_launch<true, 64>(w, s) : batch_tc_launch<false, 64>(w, s);
        case 128: return f16 ? batch_tc_launch<true, 128>(w, s) : batch_tc_launch<false, 128>(w, s);
        case 256: return f16 ? batch_tc_launch<true, 256>(w, s) : batch_tc_launch<false, 256>(w, s);
        default: set_error("tile_n %d not in {64, 128, 256}", tile_n); return SBR_ERR_INVALID_ARG;
    }
}

}  // namespace sbr
