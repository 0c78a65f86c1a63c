// Learned surrogate of the channel statistics: a BF16 MLP on Fourier features
// of (x, y, z, f) trained on SBR-traced receivers, with full SBR as fallback.
// The paper has no such model; it is a query-time stand-in for the method's
// outputs (path loss, RMS delay spread, PDP; Eq. 2, 4, 5) learned from them.
//
// Network: 4 inputs -> 128 Fourier features -> depth x width ReLU layers ->
// 128 linear outputs (the first n_out used). Training: mean squared error over
// the finite targets with per-output weights, an optional error head learning
// |prediction - target| of one output (stop-gradient), Adam on FP32 master
// weights with BF16 working copies.
//
// Everything the tcgen05 tensor cores read is kept in global memory as "images":
// pieces of [rows][64] BF16 already in the 128-byte-swizzled shared-memory
// layout, so that a piece is staged by one bulk copy without any address work.
//   activations, gradients: [row tile of 128][64-column chunk][128][64]
//   weights W [n_out][n_in]: forward [n_in / 64][n_out][64],
//                            backward (W transposed) [n_out / 64][n_in][64]
// A training step is three launches: k_net (the forward pass, the loss and the
// backward pass of the activations of a 128-row tile in one CTA), k_dw (every
// weight and bias gradient, the images read row-wise as K) and k_adam (sum of
// the partial gradients, Adam, new images). Inference is k_net alone.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include <cuda_bf16.h>

#include "sbr_internal.cuh"
#include "tcgen05.cuh"

struct sbr_mlp;

namespace sbr {
namespace {
using namespace tc;
using bf16 = __nv_bfloat16;

constexpr int kGThreads = 256;
constexpr int kFeat = 128;      // Fourier features: 4 coordinates x 16 octaves x (sin, cos)
constexpr int kOctaves = 16;
constexpr int kOutW = 128;      // output layer width (first n_out used)

constexpr int kChunkBytes = 128 * 128;      // 128 rows x 64 BF16 of an image
constexpr int kMaxLayers = 9;

enum { kEpReluBf16 = 0, kEpBiasF32 = 1 };

struct GemmArgs {
    const unsigned char* A;   // image [M / 128][K / 64][128][64]
    const unsigned char* B;   // forward image [K / 64][N][64] of the weights
    int M, N, K;              // M % 128 == 0, N % tile == 0, K % 64 == 0
    const float* bias;        // [N]
    unsigned char* Cb;        // image [M / 128][N / 64][128][64] out
    float* Cf;                // [M][N] FP32 out
    unsigned int* status;
};

template <int kN>
struct GemmShape {
    static constexpr int kStage = 128 * 128 + kN * 128;   // A and B chunks of 64 BF16 per row
    static constexpr int kSmemTiles = 2 * kStage;          // two stages
    // at least the tiles, and enough that at most 512 / kN CTAs share an SM, so
    // their tensor-memory allocations (kN columns each) always fit
    static constexpr int kTmemReq = 228 * 1024 / (512 / kN + 1) + 1024;
    static constexpr int kSmemReq = kSmemTiles + 1024 + 64 > kTmemReq ? kSmemTiles + 1024 + 64 : kTmemReq;
};

// C = A B^T (FP32 accumulation) of one layer with its bias (and ReLU): the
// layer-by-layer form of the network (sbr_mlp_predict_layered)
template <int kN, int kMode>
__global__ void __launch_bounds__(kGThreads, 1) k_gemm(const __grid_constant__ GemmArgs a) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    using Sh = GemmShape<kN>;
    uint64_t* mbar = (uint64_t*)(smem + Sh::kSmemTiles);
    uint32_t* tmem_slot = (uint32_t*)(smem + Sh::kSmemTiles + 16);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kN));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int k = 0; k < 2; ++k) asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar + k)), "r"(1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    const int m0 = blockIdx.x * 128, n0 = blockIdx.y * kN;
    // K-chunk kc of both operands into stage b with cp.async: chunk kc + 1 is in
    // flight while chunk kc's MMAs run
    auto issue = [&](int kc, int b) {
        unsigned char* sA = smem + b * Sh::kStage;
        unsigned char* sB = sA + 128 * 128;
        const unsigned char* gA = a.A + ((size_t)blockIdx.x * (a.K / 64) + kc) * kChunkBytes;
        const unsigned char* gB = a.B + ((size_t)kc * a.N + n0) * 128;
        for (int e = tid; e < 128 * 8; e += kGThreads) cp_async16(smem_u32(sA + 16 * e), gA + 16 * e);
        for (int e = tid; e < kN * 8; e += kGThreads) cp_async16(smem_u32(sB + 16 * e), gB + 16 * e);
        cp_async_commit();
    };
    uint32_t phase[2] = {0u, 0u};
    bool pending[2] = {false, false};
    bool failed = false;
    const int nchunks = a.K / 64;
    issue(0, 0);
    for (int i = 0; i < nchunks && !failed; ++i) {
        const int bi = i & 1;
        if (i + 1 < nchunks) {
            const int nb = bi ^ 1;
            if (pending[nb]) {   // the MMAs of chunk i - 1 read stage nb
                const bool ok = mbar_wait(smem_u32(mbar + nb), phase[nb]);
                phase[nb] ^= 1u;
                pending[nb] = false;
                if (__syncthreads_or(!ok)) { failed = true; break; }
            }
            issue(i + 1, nb);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            unsigned char* sA = smem + bi * Sh::kStage;
            uint64_t dA = make_desc(smem_u32(sA)), dB = make_desc(smem_u32(sA + 128 * 128));
            for (int ks = 0; ks < 4; ++ks) {
                uint64_t off = (uint64_t)(ks * 32) >> 4;   // 16 BF16 along K
                mma_16<false, kN>(tmem, dA + off, dB + off, (i > 0 || ks > 0) ? 1u : 0u);
            }
            mma_commit(smem_u32(mbar + bi));
        }
        pending[bi] = true;
    }
    cp_async_wait<0>();
    for (int b = 0; b < 2 && !failed; ++b) {   // every MMA of the tile has completed after both
        if (!pending[b]) continue;
        const bool ok = mbar_wait(smem_u32(mbar + b), phase[b]);
        if (__syncthreads_or(!ok)) failed = true;
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (failed && tid == 0) atomicOr(a.status, (unsigned)ST_TIMEOUT);
    if (!failed) {
        const int qw = warp & 3, chalf = warp >> 2;
        const int row = 32 * qw + lane;
        for (int j = 0; j < kN / 64; ++j) {
            const int col0 = (kN / 2) * chalf + 32 * j;
            uint32_t v[32];
            tmem_ld32(tmem + ((uint32_t)(32 * qw) << 16) + (uint32_t)col0, v);
            const int c0 = n0 + col0;
            if (kMode == kEpReluBf16) {
                unsigned char* img = a.Cb + ((size_t)blockIdx.x * (a.N / 64) + c0 / 64) * kChunkBytes;
                for (int k = 0; k < 32; k += 8) {
                    __align__(16) bf16 o[8];
                    for (int u = 0; u < 8; ++u) o[u] = __float2bfloat16_rn(fmaxf(__uint_as_float(v[k + u]) + a.bias[c0 + k + u], 0.f));
                    *reinterpret_cast<uint4*>(img + sw128(row, c0 % 64 + k)) = *reinterpret_cast<const uint4*>(o);
                }
            } else {
                float4* dst = reinterpret_cast<float4*>(a.Cf + (size_t)(m0 + row) * a.N + c0);
                for (int k = 0; k < 8; ++k)
                    dst[k] = make_float4(__uint_as_float(v[4 * k]) + a.bias[c0 + 4 * k],
                                         __uint_as_float(v[4 * k + 1]) + a.bias[c0 + 4 * k + 1],
                                         __uint_as_float(v[4 * k + 2]) + a.bias[c0 + 4 * k + 2],
                                         __uint_as_float(v[4 * k + 3]) + a.bias[c0 + 4 * k + 3]);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kN));
}

// Fourier features of x = (x, y, z, f) mapped to u in [0, 1]^4: for coordinate
// c and octave k, sin and cos of pi 2^(k lmax / 15) u_c; rows >= B are zero
__device__ __forceinline__ float octave(float lmax, int k) { return exp2f(lmax * (float)k / 15.0f); }
__device__ __forceinline__ float unit_coord(float x, int c, float4 lo, float4 inv) {
    const float l = c == 0 ? lo.x : (c == 1 ? lo.y : (c == 2 ? lo.z : lo.w));
    const float i = c == 0 ? inv.x : (c == 1 ? inv.y : (c == 2 ? inv.z : inv.w));
    return (x - l) * i;
}

__global__ void k_features(const float* __restrict__ x, int B, int Mp, float4 lo, float4 inv, float lmax,
                           unsigned char* __restrict__ feat) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= Mp * 4 * kOctaves) return;
    int b = t / (4 * kOctaves), r = t - b * 4 * kOctaves;
    int c = r / kOctaves, k = r - c * kOctaves;
    float s = 0.f, co = 0.f;
    if (b < B) sincospif(octave(lmax, k) * unit_coord(x[4 * (size_t)b + c], c, lo, inv), &s, &co);
    const int col = c * 2 * kOctaves + 2 * k;
    unsigned char* img = feat + ((size_t)(b / 128) * (kFeat / 64) + col / 64) * kChunkBytes;
    *reinterpret_cast<__nv_bfloat162*>(img + sw128(b % 128, col % 64)) = __floats2bfloat162_rn(s, co);
}

// outputs back to target units: y = p scale + shift
__global__ void k_take_outputs(const float* __restrict__ P, int B, int n_out, const float* __restrict__ shift,
                               const float* __restrict__ scale, float* __restrict__ y) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= B * n_out) return;
    int b = t / n_out, o = t - b * n_out;
    y[t] = P[(size_t)b * kOutW + o] * scale[o] + shift[o];
}

inline unsigned nblk(int64_t n, int t = 256) { return (unsigned)std::max<int64_t>(1, (n + t - 1) / t); }

// ---------------------------------------------------------------- fused network
// A 128-row tile goes through every layer in one CTA (and, in training, back).
// Operation o of the tile multiplies the activation tile in shared memory by a
// weight image and turns the FP32 accumulator into the next activations:
//   forward, hidden  bias + ReLU                       -> activations
//   outputs          bias, target units                -> y (inference)
//   loss             bias, loss, its gradient          -> gradient (training)
//   backward         mask of the layer's ReLU          -> gradient (training)
// Warps: sixteen for the epilogues, some for the Fourier features of the next
// tile (all of them for the first), one thread that stages weights by bulk copies kStages chunks ahead and
// one that issues the MMAs. Two accumulators (2 x 256 columns of tensor memory)
// alternate between operations, and the epilogue publishes its result in chunks
// of 64 columns, one barrier each: the MMAs of operation o + 1 on chunk 0 start
// while chunks 1..3 of operation o are still being converted, so the tensor
// core idles for one chunk's conversion per operation only, and the epilogue of
// a tile's outputs overlaps the first layer of the next tile.
// 2^20 queries, 4 x 256: 2.23 ms with one warp set alternating between MMA and
// epilogue, 0.52 ms so (the MMAs alone: 0.28 ms at the measured BF16 rate). Bound
// by shared memory: per chunk the MMAs read 48 KB, 32 KB of weights and 16 KB of
// activations are written, 768 clocks at 128 bytes each against 512 of MMA.
// A training step at 8192 rows, all three launches: 47 us (42 launches: 500 us).
constexpr int kStages = 3;
constexpr int kEpiWarps = 16;
// warps for the features of later tiles: in training most CTAs have one tile, and
// the registers are worth more (local memory spills miss the 20 KB of L1 that the
// shared memory leaves)
template <bool kTrain>
constexpr int kFeatWarps = kTrain ? 2 : 4;
template <bool kTrain>
constexpr int kNetThreads = 32 * (kEpiWarps + kFeatWarps<kTrain> + 2);
constexpr int kActBytes = 4 * kChunkBytes;        // 128 rows x 256
constexpr int kFeatBytes = 2 * kChunkBytes;       // 128 rows x 128
constexpr int kStageBytes = 256 * 128;            // 256 weight rows x 64
constexpr int kBiasFloats = kMaxLayers * 256 + 4 * kOutW;   // every layer's bias, then scale, shift, loss weight and 1 / scale of the outputs
constexpr int kNetSmem = kActBytes + kFeatBytes + kStages * kStageBytes + 1024 + 256 + 4 * kBiasFloats;
constexpr int kMaxOps = 2 * kMaxLayers - 1;

enum { kOpHidden = 0, kOpOutput = 1, kOpLoss = 2, kOpBack = 3 };

struct NetOp {
    const unsigned char* w;   // weight image
    const float* bias;        // [n]; backward: none
    unsigned char* img;       // training: image that receives the result
    int nch, n;               // K / 64 and N
    int kind, layer;          // layer whose ReLU mask is written (hidden) or applied (backward)
};

struct NetArgs {
    const float* x;
    int B;
    float4 lo, inv;
    float lmax;
    int n_ops;
    NetOp op[kMaxOps];
    int n_used;
    const float* shift;
    const float* scale;
    float* y;                 // inference
    const float* Y;           // training: targets
    const float* w;           // loss weights
    int e_ch, e_of;           // error head e_ch of output e_of
    float* loss;
    unsigned char* feat;      // image of the features
    uint32_t* mask;           // [tile][hidden layer][2][512] ReLU masks
    int n_hidden;
    unsigned int* status;
    int inject_timeout;       // test-only: wait on a barrier nothing arrives at
};

struct NetBars {
    uint64_t full[kStages], empty[kStages];
    uint64_t act[4];          // chunk c of the activations has been written
    uint64_t acc[2];          // accumulator complete
    uint64_t feat_full, feat_free;
    uint64_t never, drain;
    float oct[kOctaves];      // 2^(k lmax / 15)
    uint32_t tmem;
};
static_assert(sizeof(NetBars) <= 256, "room between the ring and the biases");

// every wait gives up after 2^26 polls (about a second)
__device__ __forceinline__ bool net_wait(const uint64_t* bar, uint32_t parity) {
    for (uint32_t it = 0; it < kSpin; ++it)
        if (mbar_test(smem_u32(bar), parity)) return true;
    return false;
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&v);
}

// max(v, 0) of two packed BF16 (rounding is monotonic: the same as rounding max(x, 0))
__device__ __forceinline__ uint32_t relu_bf16(uint32_t v) {
    __nv_bfloat162 x = *reinterpret_cast<__nv_bfloat162*>(&v);
    x = __hmax2(x, __floats2bfloat162_rn(0.f, 0.f));
    return *reinterpret_cast<uint32_t*>(&x);
}

// 0xffff in each half whose BF16 is above zero
__device__ __forceinline__ uint32_t positive_mask(uint32_t v) {
    return __hgt2_mask(*reinterpret_cast<__nv_bfloat162*>(&v), __floats2bfloat162_rn(0.f, 0.f));
}

// bits 15 and 31, each over its half (prmt in its sign-replicating mode)
__device__ __forceinline__ uint32_t spread_bits(uint32_t v) {
    uint32_t r;
    asm("prmt.b32 %0, %1, 0, 0xbb99;" : "=r"(r) : "r"(v));
    return r;
}

// sine and cosine of octaves [k0, k1) (multiples of 4) of coordinate c into row r
// of the feature tile
__device__ __forceinline__ void net_features(const NetArgs& a, const float* oct, unsigned char* feat, int r, int row, int c,
                                             int k0, int k1) {
    const bool on = row < a.B;   // rows past the end are zero
    const float u = on ? unit_coord(a.x[4 * (size_t)row + c], c, a.lo, a.inv) : 0.f;
    for (int k = k0; k < k1; k += 4) {
        const float4 f = *reinterpret_cast<const float4*>(oct + k);
        float sn[4], co[4];
        sincospif(f.x * u, sn, co);
        sincospif(f.y * u, sn + 1, co + 1);
        sincospif(f.z * u, sn + 2, co + 2);
        sincospif(f.w * u, sn + 3, co + 3);
        uint32_t w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] = on ? pack_bf16(sn[q], co[q]) : 0u;
        *reinterpret_cast<uint4*>(feat + (c >> 1) * kChunkBytes + sw128(r, 32 * (c & 1) + 2 * k)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Loss and its gradient with respect to the outputs (BF16, into the two chunks
// of the activation tile) for row r (row of the batch) and 16 columns of each chunk:
//   L = (1/B) sum_{b, o finite} w_o (p_bo - y'_bo)^2
//     + (1/B) sum_{b: y_b,c finite} w_e (p_be - |p_bc - y'_bc|)^2   (error head e of output c)
// on the normalised targets y' = (y - shift) / scale. The targets of a chunk are
// requested together; the quotients come from reciprocals taken once and one
// residual correction (forty-eight divisions, each with its branch for special
// operands, took 15 K of the kernel's 60 K clocks).
// a / b from r = 1 / b rounded: correctly rounded in the normal range (Markstein,
// IBM J. Res. Dev. 34, 1990)
__device__ __forceinline__ float quotient(float a, float b, float r) {
    const float q = __fmul_rn(a, r);
    return __fmaf_rn(__fmaf_rn(-q, b, a), r, q);
}

__device__ __forceinline__ void net_loss(const NetArgs& a, uint32_t acc, int r, int row, int qc, unsigned char* act,
                                         const float* bias, const float* s_scale, const float* s_rscale, const float* s_shift,
                                         const float* s_w, float& loss) {
    const float fB = (float)a.B, rB = __frcp_rn(fB);
    float pc = 0.f, yc = NAN;   // prediction and target that the error head learns from
    if (a.e_of >= 0) {
        const float t0 = row < a.B ? __ldg(a.Y + (size_t)row * a.n_used + a.e_of) : NAN;
        yc = quotient(t0 - s_shift[a.e_of], s_scale[a.e_of], s_rscale[a.e_of]);
        pc = __uint_as_float(tmem_ld1(acc - 16u * (uint32_t)qc + (uint32_t)a.e_of)) + bias[a.e_of];
    }
#pragma unroll 1
    for (int c = 0; c < kOutW / 64; ++c) {
        const int col0 = 64 * c + 16 * qc;
        uint32_t h[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
        if (col0 < a.n_used) {
            float yt[16];
#pragma unroll
            for (int k = 0; k < 16; ++k)
                yt[k] = row < a.B && col0 + k < a.n_used ? __ldg(a.Y + (size_t)row * a.n_used + col0 + k) : NAN;
            uint32_t x[16];
            tmem_ld16_start(acc + 64u * (uint32_t)c, x);
            tmem_ld16_wait(x);
#pragma unroll
            for (int k = 0; k < 16; k += 2) {
                float gr[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int q = col0 + k + u;
                    const float pr = __uint_as_float(x[k + u]) + bias[q];
                    const bool head = q == a.e_ch && a.e_of >= 0;
                    const float y = head ? yc : quotient(yt[k + u] - s_shift[q], s_scale[q], s_rscale[q]);
                    const bool on = isfinite(y);   // no row, output or target: NaN
                    const float d = head ? pr - fabsf(pc - y) : pr - y;
                    loss += on ? quotient(s_w[q] * d * d, fB, rB) : 0.f;
                    gr[u] = on ? quotient(2.f * s_w[q] * d, fB, rB) : 0.f;
                }
                h[k / 2] = pack_bf16(gr[0], gr[1]);
            }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k)
            *reinterpret_cast<uint4*>(act + c * kChunkBytes + sw128(r, 16 * qc + 8 * k)) =
                make_uint4(h[4 * k], h[4 * k + 1], h[4 * k + 2], h[4 * k + 3]);
    }
}

template <bool kTrain>
__global__ void __launch_bounds__(kNetThreads<kTrain>, 1) k_net(const __grid_constant__ NetArgs a) {
    constexpr int kFeatWarps = sbr::kFeatWarps<kTrain>, kNetThreads = sbr::kNetThreads<kTrain>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* act = smem;
    unsigned char* feat = act + kActBytes;
    unsigned char* ring = feat + kFeatBytes;
    NetBars& bar = *reinterpret_cast<NetBars*>(ring + kStages * kStageBytes);
    float* s_bias = reinterpret_cast<float*>(ring + kStages * kStageBytes + 256);   // [layer][256]
    float* s_scale = s_bias + kMaxLayers * 256;
    float* s_shift = s_scale + kOutW;
    float* s_w = s_shift + kOutW;
    float* s_rscale = s_w + kOutW;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int kLoadWarp = kEpiWarps + kFeatWarps, kMmaWarp = kLoadWarp + 1;
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bar.tmem)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int k = 0; k < kStages; ++k) mbar_init(smem_u32(bar.full + k), 1), mbar_init(smem_u32(bar.empty + k), 1);
        for (int k = 0; k < 4; ++k) mbar_init(smem_u32(bar.act + k), kEpiWarps);
        for (int k = 0; k < 2; ++k) mbar_init(smem_u32(bar.acc + k), 1);
        mbar_init(smem_u32(&bar.feat_full), kFeatWarps);
        mbar_init(smem_u32(&bar.feat_free), 1);
        mbar_init(smem_u32(&bar.never), 1);
        mbar_init(smem_u32(&bar.drain), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < kOctaves) bar.oct[tid] = octave(a.lmax, tid);
    ::sbr::pdl_wait();
    __syncthreads();
    for (int e = tid; e < 128 * 16; e += kNetThreads) {   // features of the first tile: (coordinate, 4 octaves, row)
        const int r = e & 127, q = e >> 7;
        net_features(a, bar.oct, feat, r, (int)blockIdx.x * 128 + r, q >> 2, 4 * (q & 3), 4 * (q & 3) + 4);
    }
    for (int o = 0; o < a.n_ops; ++o)
        if (a.op[o].kind != kOpBack)
            for (int k = tid; k < a.op[o].n; k += kNetThreads) s_bias[256 * a.op[o].layer + k] = a.op[o].bias[k];
    for (int k = tid; k < kOutW; k += kNetThreads) {
        s_scale[k] = a.scale[k];
        s_shift[k] = a.shift[k];
        if (kTrain) s_w[k] = a.w[k], s_rscale[k] = __frcp_rn(a.scale[k]);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = bar.tmem;
    const int ntiles = (a.B + 127) / 128;
    const int my_tiles = (int)blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    bool ok = true;
    // injected fault: a bounded wait gives up, the CTA takes the exit of a real timeout
    if (a.inject_timeout) ok = __syncthreads_or(!mbar_wait(smem_u32(&bar.never), 0u, 1u << 12)) == 0;
    if (warp == kLoadWarp) {
        if (lane == 0) {
            uint32_t g = 0;   // chunks staged so far
            for (int t = 0; t < my_tiles && ok; ++t)
                for (int o = 0; o < a.n_ops && ok; ++o) {
                    const uint32_t bytes = (uint32_t)a.op[o].n * 128u;
                    for (int kc = 0; kc < a.op[o].nch; ++kc, ++g) {
                        const uint32_t st = g % kStages;
                        if (g >= kStages && !net_wait(bar.empty + st, (g / kStages - 1) & 1u)) { ok = false; break; }
                        mbar_expect(smem_u32(bar.full + st), bytes);
                        bulk_load(smem_u32(ring + st * kStageBytes), a.op[o].w + (size_t)kc * bytes, bytes, smem_u32(bar.full + st));
                    }
                }
            // the copies in flight land before the CTA's shared memory is given up (another
            // role's wait may have run out)
            for (uint32_t k = g > kStages ? g - kStages : 0; k < g; ++k) net_wait(bar.full + k % kStages, (k / kStages) & 1u);
        }
    } else if (warp == kMmaWarp) {
        // the whole warp walks the loop, so that descriptors and addresses stay in
        // uniform registers; one elected lane issues
        const bool lead = elect_one();
        const uint64_t dFeat = make_desc(smem_u32(feat)), dAct = make_desc(smem_u32(act)), dRing = make_desc(smem_u32(ring));
        uint32_t g = 0, ops = 0, act_phase = 0;   // act_phase: parity per chunk
        auto wait = [&](const uint64_t* b, uint32_t parity) { return __all_sync(0xffffffffu, net_wait(b, parity)) != 0; };
        // what other warps wrote to shared memory before they arrived on a barrier
        // becomes visible to the tensor core and the bulk copies by one proxy fence
        // here, on the path from their writes to the reads (a fence in every writing
        // warp costs 60 clocks each, one after the other)
        auto to_async = [] { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); };
        for (int t = 0; t < my_tiles && ok; ++t) {
            const size_t tile = (size_t)blockIdx.x + (size_t)t * gridDim.x;
            for (int o = 0; o < a.n_ops && ok; ++o, ++ops) {
                const int nch = a.op[o].nch;
                const uint32_t acc = tmem + (ops & 1u) * 256u, id = idesc_bf16(a.op[o].n, false, false);
                uint64_t dA = o == 0 ? dFeat : dAct;
                if (o == 0) {
                    ok = t == 0 || wait(&bar.feat_full, (uint32_t)(t - 1) & 1u);
                    to_async();
                    if (kTrain && ok && lead) bulk_store(a.feat + tile * kFeatBytes, smem_u32(feat), kFeatBytes);
                }
                for (int kc = 0; kc < nch && ok; ++kc, ++g, dA += kChunkBytes >> 4) {
                    const uint32_t st = g % kStages;
                    ok = wait(bar.full + st, (g / kStages) & 1u);   // long staged, as a rule
                    if (!ok) break;
                    if (o > 0) {
                        ok = wait(bar.act + kc, (act_phase >> kc) & 1u);
                        act_phase ^= 1u << kc;
                        if (!ok) break;
                        to_async();
                        if (kTrain && lead)
                            bulk_store(a.op[o - 1].img + (tile * nch + kc) * kChunkBytes, smem_u32(act + kc * kChunkBytes), kChunkBytes);
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint64_t dB = dRing + (uint64_t)(st * (kStageBytes >> 4));
                    if (lead) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks) mma_bf16(acc, dA + 2 * ks, dB + 2 * ks, id, (kc > 0 || ks > 0) ? 1u : 0u);
                        mma_commit(smem_u32(bar.empty + st));
                    }
                    __syncwarp();
                }
                if (!ok) break;
                if (lead) {
                    // whatever is written over next has been read by the stores of this tile
                    if (kTrain) bulk_wait_read();
                    mma_commit(smem_u32(bar.acc + (ops & 1u)));
                    if (o == 0) mma_commit(smem_u32(&bar.feat_free));
                }
                __syncwarp();
            }
            if (kTrain && ok) {   // the last gradient: no MMA reads it here
                const int nc = a.op[a.n_ops - 1].n / 64;
                for (int kc = 0; kc < nc && ok; ++kc) {
                    ok = wait(bar.act + kc, (act_phase >> kc) & 1u);
                    act_phase ^= 1u << kc;
                    to_async();
                    if (ok && lead)
                        bulk_store(a.op[a.n_ops - 1].img + (tile * nc + kc) * kChunkBytes, smem_u32(act + kc * kChunkBytes), kChunkBytes);
                }
                if (lead) bulk_wait_read();
            }
        }
        if (kTrain && lead) bulk_wait_done();
        if (!ok) {   // the MMAs issued so far complete before their memory is freed
            if (lead) mma_commit(smem_u32(&bar.drain));
            __syncwarp();
            (void)wait(&bar.drain, 0u);
        }
    } else if (warp >= kEpiWarps) {
        // features of the tiles after the first
        for (int t = 1; t < my_tiles && ok; ++t) {
            ok = __all_sync(0xffffffffu, net_wait(&bar.feat_free, (uint32_t)(t - 1) & 1u));
            if (!ok) break;
            const int r0 = ((int)blockIdx.x + t * (int)gridDim.x) * 128;
#pragma unroll 1
            for (int e = tid - 32 * kEpiWarps; e < 4 * 128; e += 32 * kFeatWarps)
                net_features(a, bar.oct, feat, e & 127, r0 + (e & 127), e >> 7, 0, kOctaves);
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bar.feat_full));
        }
    } else {
        const int lq = warp & 3, qc = warp >> 2;          // TMEM lane quarter, 16-column quarter of a chunk
        const int r = 32 * lq + lane;                     // row of the tile
        const uint32_t tq = tmem + ((uint32_t)(32 * lq) << 16) + 16u * (uint32_t)qc;
        float loss = 0.f;
        uint32_t ops = 0;
        for (int t = 0; t < my_tiles && ok; ++t) {
            const int r0 = ((int)blockIdx.x + t * (int)gridDim.x) * 128, row = r0 + r;
            // ReLU masks of this thread's columns: column 2 k + u of an even (odd)
            // chunk in bit k + 16 u (k + 8 + 16 u) of word [layer][c / 2]
            uint32_t* mask = kTrain ? a.mask + ((size_t)(r0 / 128) * a.n_hidden * 2) * (32 * kEpiWarps) + tid : nullptr;
            for (int o = 0; o < a.n_ops && ok; ++o, ++ops) {
                const int kind = a.op[o].kind, nc = a.op[o].n / 64, layer = a.op[o].layer;
                const float* bias = s_bias + 256 * layer + 16 * qc;
                const uint32_t acc = tq + (ops & 1u) * 256u;
                float b[16];
                auto load_bias = [&](int c) {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        *reinterpret_cast<float4*>(b + 4 * k) = *(reinterpret_cast<const float4*>(bias + 64 * c) + k);
                };
                uint32_t mw[2] = {0u, 0u};   // masks of the two chunk pairs
                if (kTrain && kind == kOpBack) {
                    mw[0] = mask[(2 * layer) * 32 * kEpiWarps];
                    if (nc > 2) mw[1] = mask[(2 * layer + 1) * 32 * kEpiWarps];
                }
                if (kind != kOpBack) load_bias(0);
                ok = __all_sync(0xffffffffu, net_wait(bar.acc + (ops & 1u), (ops >> 1) & 1u));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (kTrain && kind == kOpLoss) {
                    net_loss(a, acc, r, row, qc, act, s_bias + 256 * layer, s_scale, s_rscale, s_shift, s_w, loss);
                    for (int c = 0; c < nc; ++c) {
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(bar.act + c));
                    }
                    continue;
                }
                // the accumulator of the next chunk is on its way while one is converted
                // (two chunks per turn: nc is even)
                uint32_t v[2][16];
                tmem_ld16_start(acc, v[0]);
#pragma unroll 1
                for (int c2 = 0; c2 < nc; c2 += 2)
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const int c = c2 + half;
                    uint32_t(&x)[16] = v[half];
                    tmem_ld16_wait(x);
                    if (c + 1 < nc) tmem_ld16_start(acc + 64u * (uint32_t)(c + 1), v[half ^ 1]);
                    const int col0 = 64 * c + 16 * qc;
                    uint32_t h[8];
                    if (kind == kOpHidden) {
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            h[k] = relu_bf16(pack_bf16(__uint_as_float(x[2 * k]) + b[2 * k], __uint_as_float(x[2 * k + 1]) + b[2 * k + 1]));
                        if (c + 1 < nc) load_bias(c + 1);
                        if (kTrain) {
                            uint32_t m = 0;
#pragma unroll
                            for (int k = 0; k < 8; ++k) m |= positive_mask(h[k]) & (0x00010001u << (k + 8 * half));
                            mw[0] = half ? mw[0] | m : m;
                            if (half) mask[(2 * layer + (c >> 1)) * 32 * kEpiWarps] = mw[0];
                        }
                    } else if (!kTrain) {
                        // outputs in target units, 16-byte stores where every row starts on 16 bytes
                        if (col0 < a.n_used && row < a.B) {
                            float* y = a.y + (size_t)row * a.n_used + col0;
                            const bool vec = (a.n_used & 3) == 0 && (reinterpret_cast<uintptr_t>(a.y) & 15) == 0;
#pragma unroll
                            for (int k = 0; k < 16; k += 4) {
                                const float4 sc = *reinterpret_cast<const float4*>(s_scale + col0 + k);
                                const float4 sh = *reinterpret_cast<const float4*>(s_shift + col0 + k);
                                const float4 o4 = make_float4((__uint_as_float(x[k]) + b[k]) * sc.x + sh.x,
                                                              (__uint_as_float(x[k + 1]) + b[k + 1]) * sc.y + sh.y,
                                                              (__uint_as_float(x[k + 2]) + b[k + 2]) * sc.z + sh.z,
                                                              (__uint_as_float(x[k + 3]) + b[k + 3]) * sc.w + sh.w);
                                const int left = a.n_used - col0 - k;
                                if (vec && left > 0) {
                                    *reinterpret_cast<float4*>(y + k) = o4;
                                } else {
                                    if (left > 0) y[k] = o4.x;
                                    if (left > 1) y[k + 1] = o4.y;
                                    if (left > 2) y[k + 2] = o4.z;
                                    if (left > 3) y[k + 3] = o4.w;
                                }
                            }
                        }
                        if (c + 1 < nc) load_bias(c + 1);
                        continue;
                    } else {
                        const uint32_t m = (c2 ? mw[1] : mw[0]) >> (8 * half);
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            h[k] = pack_bf16(__uint_as_float(x[2 * k]), __uint_as_float(x[2 * k + 1])) & spread_bits(m << (15 - k));
                    }
#pragma unroll
                    for (int k = 0; k < 2; ++k)
                        *reinterpret_cast<uint4*>(act + c * kChunkBytes + sw128(r, 16 * qc + 8 * k)) =
                            make_uint4(h[4 * k], h[4 * k + 1], h[4 * k + 2], h[4 * k + 3]);
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(bar.act + c));
                }
            }
        }
        if (kTrain && a.loss) {
            for (int s = 16; s; s >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, s);
            if (lane == 0 && ok) atomicAdd(a.loss, loss);
        }
    }
    if (!ok) atomicOr(a.status, (unsigned)ST_TIMEOUT);
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == kMmaWarp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// ---------------------------------------------------------------- weight gradients
// dW[o][i] = sum over rows dH[row][o] X[row][i] and db[o] = sum over rows
// dH[row][o], every layer in one launch: CTA (job, part) owns 128 outputs of one
// layer, all its inputs, and a share of the 128-row tiles; both operands are
// images read with the rows as K (MN-major), db a 16-column MMA against ones.
// Each part writes its own sum; k_adam adds the parts in order, so the result
// does not depend on the order of the CTAs and nothing has to be zeroed.
// Bound by reading the images from L2: 37 MB at 8192 rows of the 4 x 256
// network. Five transposing GEMMs with atomics, ten transposes and five column
// sums took 300 us of the step.
constexpr int kDwThreads = 256;
constexpr int kDwStage = 6 * kChunkBytes;   // 2 chunks of dH, up to 4 of X
constexpr int kDwSmem = 2 * kDwStage + 2048 + 1024 + 64;
constexpr int kMaxParts = 32;

struct DwLayer {
    const unsigned char* dH;
    const unsigned char* X;
    int n_in, n_out;
    int64_t off;
    int job0;                 // first job of the layer
};
struct DwArgs {
    DwLayer L[kMaxLayers];
    int n_layers, tiles, parts;
    int64_t n_params;
    float* part;
    unsigned int* status;
};

__global__ void __launch_bounds__(kDwThreads, 1) k_dw(const __grid_constant__ DwArgs a) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* ones = smem + 2 * kDwStage;   // [16][64] BF16
    uint64_t* full = reinterpret_cast<uint64_t*>(ones + 2048);
    uint64_t* empty = full + 2;
    uint64_t* done = full + 4;
    uint32_t* slot = reinterpret_cast<uint32_t*>(full + 5);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    for (int k = tid; k < 512; k += kDwThreads) reinterpret_cast<uint32_t*>(ones)[k] = 0x3f803f80u;
    if (tid == 0) {
        for (int k = 0; k < 5; ++k) mbar_init(smem_u32(full + k), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *slot;
    ::sbr::pdl_wait();
    int l = 0;
    while (l + 1 < a.n_layers && (int)blockIdx.x >= a.L[l + 1].job0) ++l;
    const DwLayer& ly = a.L[l];
    const int mt = (int)blockIdx.x - ly.job0;
    const int nb = ly.n_in / 64, na = ly.n_out / 64;
    const int t0 = (int)((int64_t)blockIdx.y * a.tiles / a.parts), t1 = (int)((int64_t)(blockIdx.y + 1) * a.tiles / a.parts);
    bool ok = true;
    if (tid == 0) {
        int staged = 0;
        for (int t = t0; t < t1; ++t) {
            const int k = t - t0, st = k & 1;
            if (k >= 2 && !net_wait(empty + st, (uint32_t)((k >> 1) - 1) & 1u)) { ok = false; break; }
            staged = k + 1;
            const uint32_t sA = smem_u32(smem + st * kDwStage), f = smem_u32(full + st);
            mbar_expect(f, (uint32_t)((2 + nb) * kChunkBytes));
            bulk_load(sA, ly.dH + ((size_t)t * na + 2 * mt) * kChunkBytes, 2 * kChunkBytes, f);
            bulk_load(sA + 2 * kChunkBytes, ly.X + (size_t)t * nb * kChunkBytes, (uint32_t)(nb * kChunkBytes), f);
        }
        // the copies in flight land before the CTA's shared memory is given up
        for (int j = staged > 2 ? staged - 2 : 0; j < staged; ++j) net_wait(full + (j & 1), (uint32_t)(j >> 1) & 1u);
    } else if (tid == 32) {
        const uint32_t id = idesc_bf16(ly.n_in, true, true), idb = idesc_bf16(16, true, false);
        const uint64_t d1 = make_desc(smem_u32(ones));
        for (int t = t0; t < t1; ++t) {
            const int k = t - t0, st = k & 1;
            if (!net_wait(full + st, (uint32_t)(k >> 1) & 1u)) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t sA = smem_u32(smem + st * kDwStage);
            const uint64_t dA = make_desc_mn(sA, kChunkBytes), dB = make_desc_mn(sA + 2 * kChunkBytes, kChunkBytes);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {   // 16 rows of K: 2048 bytes of every chunk
                const uint32_t accum = (k > 0 || ks > 0) ? 1u : 0u;
                mma_bf16(tmem, dA + 128 * ks, dB + 128 * ks, id, accum);
                mma_bf16(tmem + 256, dA + 128 * ks, d1, idb, accum);
            }
            mma_commit(smem_u32(empty + st));
        }
        mma_commit(smem_u32(done));   // (after a wait that ran out too: what was issued completes before its memory is freed)
    }
    __syncwarp();
    ok = net_wait(done, 0u) && ok;
    ok = !__syncthreads_or(!ok);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok) {
        const int lq = warp & 3, half = warp >> 2, r = 128 * mt + 32 * lq;
        const uint32_t tq = tmem + ((uint32_t)(32 * lq) << 16);
        float* out = a.part + (int64_t)blockIdx.y * a.n_params + ly.off;
        // 32 x 32 blocks through shared memory (rows of 36 floats), so that a
        // store covers whole 128-byte lines
        float* blk = reinterpret_cast<float*>(smem) + warp * (32 * 36);
        for (int c0 = 32 * half; c0 < ly.n_in; c0 += 64) {
            uint32_t v[32];
            tmem_ld32(tq + (uint32_t)c0, v);
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 8; ++k)
                *reinterpret_cast<uint4*>(blk + 36 * lane + 4 * k) = make_uint4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int rr = 4 * k + (lane >> 3), cc = 4 * (lane & 7);
                *reinterpret_cast<float4*>(out + (int64_t)(r + rr) * ly.n_in + c0 + cc) =
                    *reinterpret_cast<const float4*>(blk + 36 * rr + cc);
            }
        }
        if (half == 0) out[(int64_t)ly.n_out * ly.n_in + r + lane] = __uint_as_float(tmem_ld1(tq + 256u));
    } else if (tid == 0) {
        atomicOr(a.status, (unsigned)ST_TIMEOUT);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// ---------------------------------------------------------------- optimiser
struct AdamLayer {
    int64_t off;
    int n_in, n_out;
    unsigned char *Wf, *Wb;
};
struct AdamArgs {
    AdamLayer L[kMaxLayers];
    int n_layers, parts;
    int64_t n;
    float *p, *m, *v, *g;
    const float* part;
    const unsigned int* status;
    float lr, b1, b2, eps, c1, c2;
};

// four consecutive parameters per thread: the gradient (the sum of its parts, in
// order), Adam on the FP32 masters, and the BF16 images of the new weights.
// A step in which a bounded wait gave up changes nothing. kStep false: the images
// alone, from the masters.
template <bool kStep>
__global__ void __launch_bounds__(256) k_adam(const __grid_constant__ AdamArgs a) {
    ::sbr::pdl_wait();
    const int64_t i = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= a.n) return;
    // a wait that gave up in this step's launches or before: read with the rest, nothing stored
    const unsigned failed = kStep ? __ldg(a.status) & ST_TIMEOUT : 0u;
    float p[4];
    *reinterpret_cast<float4*>(p) = *reinterpret_cast<const float4*>(a.p + i);
    if (kStep) {
        float g[4] = {0.f, 0.f, 0.f, 0.f}, m[4], v[4];
#pragma unroll 8
        for (int s = 0; s < a.parts; ++s) {
            const float4 x = __ldg(reinterpret_cast<const float4*>(a.part + s * a.n + i));
            g[0] += x.x; g[1] += x.y; g[2] += x.z; g[3] += x.w;
        }
        *reinterpret_cast<float4*>(m) = *reinterpret_cast<const float4*>(a.m + i);
        *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(a.v + i);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            m[k] = a.b1 * m[k] + (1.f - a.b1) * g[k];
            v[k] = a.b2 * v[k] + (1.f - a.b2) * g[k] * g[k];
            p[k] = p[k] - a.lr * (m[k] / a.c1) / (sqrtf(v[k] / a.c2) + a.eps);
        }
        if (failed) return;
        *reinterpret_cast<float4*>(a.g + i) = *reinterpret_cast<const float4*>(g);
        *reinterpret_cast<float4*>(a.m + i) = *reinterpret_cast<const float4*>(m);
        *reinterpret_cast<float4*>(a.v + i) = *reinterpret_cast<const float4*>(v);
        *reinterpret_cast<float4*>(a.p + i) = *reinterpret_cast<const float4*>(p);
    }
    int l = 0;
    while (l + 1 < a.n_layers && i >= a.L[l + 1].off) ++l;
    const AdamLayer& ly = a.L[l];
    const int64_t j = i - ly.off;
    if (j >= (int64_t)ly.n_in * ly.n_out) return;   // a bias
    const int o = (int)(j / ly.n_in), c = (int)(j - (int64_t)o * ly.n_in);
    *reinterpret_cast<uint2*>(ly.Wf + (size_t)(c >> 6) * ly.n_out * 128 + sw128(o, c & 63)) =
        make_uint2(pack_bf16(p[0], p[1]), pack_bf16(p[2], p[3]));
    unsigned char* wb = ly.Wb + (size_t)(o >> 6) * ly.n_in * 128;
#pragma unroll
    for (int k = 0; k < 4; ++k) *reinterpret_cast<bf16*>(wb + sw128(c + k, o & 63)) = __float2bfloat16_rn(p[k]);
}

template <int kN, int kMode>
sbr_status gemm_launch(const GemmArgs& a, cudaStream_t s) {
    static std::atomic<unsigned long long> attr{0};
    SBR_TRY(set_smem_once((const void*)k_gemm<kN, kMode>, GemmShape<kN>::kSmemReq, &attr));
    dim3 grid(a.M / 128, a.N / kN);
    ::sbr::note_launch(), k_gemm<kN, kMode><<<grid, kGThreads, GemmShape<kN>::kSmemReq, s>>>(a);
    SBR_TRY_CUDA(cudaGetLastError());
    return SBR_OK;
}

// dispatch on the tile width (the whole N, 128 or 256)
template <int kMode>
sbr_status gemm(const GemmArgs& a, cudaStream_t s) {
    return a.N == 256 ? gemm_launch<256, kMode>(a, s) : gemm_launch<128, kMode>(a, s);
}

struct Layer {
    int n_in, n_out;
    int64_t off;                  // of W in the flat parameter order (per layer W, then b)
    unsigned char* Wf = nullptr;  // forward image of the weights
    unsigned char* Wb = nullptr;  // backward image
    unsigned char* H = nullptr;   // image of the activations out (hidden layers)
    unsigned char* dH = nullptr;  // image of the gradient w.r.t. the (pre-activation) output
};

}  // namespace
}  // namespace sbr

struct sbr_mlp {
    int device = 0;
    sbr_mlp_config cfg{};
    int Mp = 0;                        // max_batch rounded up to 128
    std::vector<sbr::Layer> L;         // depth hidden + output
    std::vector<float> loss_w;         // [n_out]
    float* d_loss_w = nullptr;         // [128] loss weights
    float* d_shift = nullptr;          // [128] target normalisation
    float* d_scale = nullptr;
    int64_t n_params = 0;
    float* p = nullptr;                // flat FP32 masters, gradients and Adam moments [n_params]
    float *g = nullptr, *m = nullptr, *v = nullptr;
    float* part = nullptr;             // [n_part][n_params] partial gradients
    int n_part = 0;
    unsigned char* feat = nullptr;     // image of the features
    uint32_t* mask = nullptr;          // ReLU masks of a training step
    float* P = nullptr;                // [Mp][128] outputs (layer-by-layer form)
    unsigned int* status = nullptr;
    int64_t step = 0;
    std::vector<void*> owned;
};

namespace sbr {
namespace {

template <class T>
sbr_status malloc_owned(sbr_mlp* m, T** p, size_t n) {
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(p), std::max<size_t>(n, 1) * sizeof(T));
    if (e != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();
        set_error("mlp allocation of %zu bytes: %s", n * sizeof(T), cudaGetErrorString(e));
        return SBR_ERR_ALLOC;
    }
    m->owned.push_back(*p);
    return SBR_OK;
}

void free_mlp(sbr_mlp* m) {
    if (!m) return;
    cudaDeviceSynchronize();
    for (void* p : m->owned) cudaFree(p);
    delete m;
}

// splitmix64: seeded, platform-independent initial weights
uint64_t splitmix(uint64_t& x) {
    uint64_t z = (x += 0x9e3779b97f4a7c15ull);
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

float4 box_lo(const sbr_mlp_config& c) { return make_float4(c.x_lo[0], c.x_lo[1], c.x_lo[2], c.x_lo[3]); }
float4 box_inv(const sbr_mlp_config& c) {
    return make_float4(1.f / (c.x_hi[0] - c.x_lo[0]), 1.f / (c.x_hi[1] - c.x_lo[1]), 1.f / (c.x_hi[2] - c.x_lo[2]),
                       1.f / (c.x_hi[3] - c.x_lo[3]));
}

// the outputs of every row in m->P, one GEMM per layer
sbr_status forward_layered(const sbr_mlp* m, const float* x, int B, cudaStream_t s) {
    const sbr_mlp_config& c = m->cfg;
    const int Mp = ((B + 127) / 128) * 128;
    ::sbr::note_launch(), k_features<<<nblk((int64_t)Mp * 4 * kOctaves), 256, 0, s>>>(x, B, Mp, box_lo(c), box_inv(c),
                                                                                      c.feat_log2_max, m->feat);
    SBR_TRY_CUDA(cudaGetLastError());
    const unsigned char* in = m->feat;
    for (size_t l = 0; l < m->L.size(); ++l) {
        const Layer& ly = m->L[l];
        GemmArgs a{};
        a.A = in;
        a.B = ly.Wf;
        a.M = Mp;
        a.N = ly.n_out;
        a.K = ly.n_in;
        a.bias = m->p + ly.off + (int64_t)ly.n_out * ly.n_in;
        a.status = m->status;
        if (l + 1 < m->L.size()) {
            a.Cb = ly.H;
            SBR_TRY(gemm<kEpReluBf16>(a, s));
            in = ly.H;
        } else {
            a.Cf = m->P;
            SBR_TRY(gemm<kEpBiasF32>(a, s));
        }
    }
    return SBR_OK;
}

// the operations of the fused kernel: the forward layers, then (training) the
// gradient back through them to the first layer's output
NetArgs net_args(const sbr_mlp* m, const float* x, int B, bool train) {
    const sbr_mlp_config& c = m->cfg;
    NetArgs a{};
    a.x = x;
    a.B = B;
    a.lo = box_lo(c);
    a.inv = box_inv(c);
    a.lmax = c.feat_log2_max;
    const int nl = (int)m->L.size();
    for (int l = 0; l < nl; ++l) {
        const Layer& ly = m->L[l];
        const bool last = l + 1 == nl;
        a.op[a.n_ops++] = NetOp{ly.Wf, m->p + ly.off + (int64_t)ly.n_out * ly.n_in, last ? ly.dH : ly.H, ly.n_in / 64,
                                ly.n_out, last ? (train ? kOpLoss : kOpOutput) : kOpHidden, l};
    }
    if (train)
        for (int l = nl - 1; l >= 1; --l) {
            const Layer& ly = m->L[l];
            a.op[a.n_ops++] = NetOp{ly.Wb, nullptr, m->L[l - 1].dH, ly.n_out / 64, ly.n_in, kOpBack, l - 1};
        }
    a.n_used = c.n_out;
    a.shift = m->d_shift;
    a.scale = m->d_scale;
    a.status = m->status;
    a.inject_timeout = fault_mode() == kFaultTimeout ? 1 : 0;
    return a;
}

template <bool kTrain>
sbr_status net_launch(const NetArgs& a, cudaStream_t s) {
    static std::atomic<unsigned long long> attr{0};
    SBR_TRY(set_smem_once((const void*)k_net<kTrain>, kNetSmem, &attr));
    const int grid = std::min((a.B + 127) / 128, sm_count());
    ::sbr::note_launch();
    SBR_TRY_CUDA(::sbr::launch_pdl(k_net<kTrain>, dim3(grid), dim3(kNetThreads<kTrain>), kNetSmem, s, a));
    return SBR_OK;
}

AdamArgs adam_args(const sbr_mlp* m) {
    AdamArgs a{};
    for (const Layer& ly : m->L) a.L[a.n_layers++] = AdamLayer{ly.off, ly.n_in, ly.n_out, ly.Wf, ly.Wb};
    a.n = m->n_params;
    a.p = m->p;
    a.m = m->m;
    a.v = m->v;
    a.g = m->g;
    a.part = m->part;
    a.status = m->status;
    return a;
}

template <bool kStep>
sbr_status adam_launch(const AdamArgs& a, cudaStream_t s) {
    ::sbr::note_launch();
    SBR_TRY_CUDA(::sbr::launch_pdl(k_adam<kStep>, dim3(nblk(a.n / 4)), dim3(256), 0, s, a));
    return SBR_OK;
}

sbr_status train_step(sbr_mlp* m, const float* x, const float* y, int B, float* loss, cudaStream_t s) {
    const sbr_mlp_config& c = m->cfg;
    NetArgs n = net_args(m, x, B, true);
    n.Y = y;
    n.w = m->d_loss_w;
    n.e_ch = c.err_channel;
    n.e_of = c.err_of;
    n.loss = loss;
    n.feat = m->feat;
    n.mask = m->mask;
    n.n_hidden = (int)m->L.size() - 1;
    SBR_TRY(net_launch<true>(n, s));
    DwArgs d{};
    int jobs = 0;
    for (size_t l = 0; l < m->L.size(); ++l) {
        const Layer& ly = m->L[l];
        d.L[d.n_layers++] = DwLayer{ly.dH, l > 0 ? m->L[l - 1].H : m->feat, ly.n_in, ly.n_out, ly.off, jobs};
        jobs += ly.n_out / 128;
    }
    d.tiles = (B + 127) / 128;
    d.parts = std::min(m->n_part, d.tiles);
    d.n_params = m->n_params;
    d.part = m->part;
    d.status = m->status;
    static std::atomic<unsigned long long> attr{0};
    SBR_TRY(set_smem_once((const void*)k_dw, kDwSmem, &attr));
    ::sbr::note_launch();
    SBR_TRY_CUDA(::sbr::launch_pdl(k_dw, dim3(jobs, d.parts), dim3(kDwThreads), kDwSmem, s, d));
    m->step += 1;
    AdamArgs a = adam_args(m);
    a.parts = d.parts;
    a.lr = c.lr;
    a.b1 = c.beta1;
    a.b2 = c.beta2;
    a.eps = c.eps;
    a.c1 = 1.f - powf(c.beta1, (float)m->step);
    a.c2 = 1.f - powf(c.beta2, (float)m->step);
    return adam_launch<true>(a, s);
}

sbr_status sync_images(sbr_mlp* m, cudaStream_t s) { return adam_launch<false>(adam_args(m), s); }

sbr_status infer_fused(const sbr_mlp* m, const float* x, int B, float* y, cudaStream_t s) {
    NetArgs a = net_args(m, x, B, false);
    a.y = y;
    return net_launch<false>(a, s);
}

}  // namespace
}  // namespace sbr

using namespace sbr;

extern "C" {

sbr_status sbr_mlp_create(const sbr_mlp_config* cfg, const float* loss_w, const float* y_shift,
                          const float* y_scale, sbr_mlp** out, void* stream) {
    clear_error();
    SBR_CHECK_ARG(cfg && out, "config and out");
    *out = nullptr;
    const sbr_mlp_config& c = *cfg;
    SBR_CHECK_ARG(c.n_out >= 1 && c.n_out <= kOutW, "n_out in [1, 128]");
    SBR_CHECK_ARG(c.width == 128 || c.width == 256, "width 128 or 256");
    SBR_CHECK_ARG(c.depth >= 1 && c.depth <= 8, "depth in [1, 8]");
    SBR_CHECK_ARG(c.max_batch >= 1 && c.max_batch <= (1 << 22), "max_batch in [1, 2^22]");
    SBR_CHECK_ARG((c.err_of < 0 && c.err_channel < 0) ||
                      (c.err_of >= 0 && c.err_channel >= 0 && c.err_of < c.n_out && c.err_channel < c.n_out &&
                       c.err_of != c.err_channel),
                  "error head channels: both -1, or two different outputs");
    for (int k = 0; k < 4; ++k) SBR_CHECK_ARG(c.x_hi[k] > c.x_lo[k], "x_hi > x_lo");
    SBR_CHECK_ARG(c.feat_log2_max >= 0.f && c.feat_log2_max <= 20.f, "feat_log2_max in [0, 20]");
    SBR_CHECK_ARG(c.lr > 0.f && c.beta1 >= 0.f && c.beta1 < 1.f && c.beta2 >= 0.f && c.beta2 < 1.f && c.eps > 0.f,
                  "Adam hyper-parameters");
    sbr_mlp* m = new (std::nothrow) sbr_mlp();
    if (!m) { set_error("host allocation"); return SBR_ERR_ALLOC; }
    SBR_TRY_CUDA(cudaGetDevice(&m->device));
    m->cfg = c;
    if (m->cfg.feat_log2_max == 0.f) m->cfg.feat_log2_max = 9.f;
    m->Mp = ((c.max_batch + 127) / 128) * 128;
    m->loss_w.assign(c.n_out, 1.f);
    if (loss_w) for (int k = 0; k < c.n_out; ++k) m->loss_w[k] = loss_w[k];
    auto fail = [&](sbr_status st) { free_mlp(m); return st; };
    sbr_status st;
    const int Mp = m->Mp;
    std::vector<int> widths;
    widths.push_back(kFeat);
    for (int d = 0; d < c.depth; ++d) widths.push_back(c.width);
    widths.push_back(kOutW);
    int jobs = 0;
    for (size_t l = 0; l + 1 < widths.size(); ++l) {
        Layer ly;
        ly.n_in = widths[l];
        ly.n_out = widths[l + 1];
        ly.off = m->n_params;
        const size_t nw = (size_t)ly.n_in * ly.n_out;
        m->n_params += (int64_t)nw + ly.n_out;
        jobs += ly.n_out / 128;
        if ((st = malloc_owned(m, &ly.Wf, 2 * nw)) || (st = malloc_owned(m, &ly.Wb, 2 * nw)) ||
            (l + 2 < widths.size() && (st = malloc_owned(m, &ly.H, 2 * (size_t)Mp * ly.n_out))) ||
            (st = malloc_owned(m, &ly.dH, 2 * (size_t)Mp * ly.n_out)))
            return fail(st);
        m->L.push_back(ly);
    }
    m->n_part = std::max(1, std::min(std::min(kMaxParts, sm_count() / jobs), Mp / 128));
    const size_t np = (size_t)m->n_params;
    if ((st = malloc_owned(m, &m->p, np)) || (st = malloc_owned(m, &m->g, np)) || (st = malloc_owned(m, &m->m, np)) ||
        (st = malloc_owned(m, &m->v, np)) || (st = malloc_owned(m, &m->part, np * m->n_part)) ||
        (st = malloc_owned(m, &m->feat, 2 * (size_t)Mp * kFeat)) || (st = malloc_owned(m, &m->P, (size_t)Mp * kOutW)) ||
        (st = malloc_owned(m, &m->mask, (size_t)(Mp / 128) * c.depth * 2 * 32 * kEpiWarps)) ||
        (st = malloc_owned(m, &m->status, 1)) || (st = malloc_owned(m, &m->d_loss_w, kOutW)) ||
        (st = malloc_owned(m, &m->d_shift, kOutW)) || (st = malloc_owned(m, &m->d_scale, kOutW)))
        return fail(st);
    // He-uniform weights, zero biases
    uint64_t rs = c.seed;
    std::vector<float> host(np, 0.f);
    for (size_t l = 0; l < m->L.size(); ++l) {
        const Layer& ly = m->L[l];
        const size_t nw = (size_t)ly.n_in * ly.n_out;
        const float lim = std::sqrt(6.0f / (float)ly.n_in) * (l + 1 == m->L.size() ? 0.1f : 1.0f);
        for (size_t i = 0; i < nw; ++i)
            host[ly.off + i] = lim * (2.0f * (float)((splitmix(rs) >> 40) * (1.0 / 16777216.0)) - 1.0f);
    }
    if (cudaMemcpy(m->p, host.data(), np * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(m->m, 0, np * 4) != cudaSuccess || cudaMemset(m->v, 0, np * 4) != cudaSuccess) {
        set_error("mlp initialisation copy failed");
        return fail(SBR_ERR_CUDA);
    }
    std::vector<float> lw(kOutW, 0.f), sh(kOutW, 0.f), sc(kOutW, 1.f);
    for (int k = 0; k < c.n_out; ++k) {
        lw[k] = m->loss_w[k];
        if (y_shift) sh[k] = y_shift[k];
        if (y_scale) sc[k] = y_scale[k];
        if (!(sc[k] > 0.f) || !std::isfinite(sh[k])) {
            set_error("y_scale must be > 0 and y_shift finite (output %d)", k);
            return fail(SBR_ERR_INVALID_ARG);
        }
    }
    if (cudaMemcpy(m->d_loss_w, lw.data(), kOutW * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(m->d_shift, sh.data(), kOutW * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(m->d_scale, sc.data(), kOutW * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(m->status, 0, 4) != cudaSuccess) {
        set_error("mlp initialisation copy failed");
        return fail(SBR_ERR_CUDA);
    }
    if ((st = sync_images(m, (cudaStream_t)stream)) != SBR_OK) return fail(st);
    if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return fail(SBR_ERR_CUDA);
    *out = m;
    return SBR_OK;
}

sbr_status sbr_mlp_train_step(sbr_mlp* m, const float* x, const float* y, int32_t B, float* loss, void* stream) {
    clear_error();
    SBR_CHECK_ARG(m && x && y, "mlp, x, y");
    SBR_CHECK_ARG(B >= 1 && B <= m->cfg.max_batch, "1 <= B <= max_batch");
    return train_step(m, x, y, B, loss, (cudaStream_t)stream);
}

sbr_status sbr_mlp_predict(const sbr_mlp* m, const float* x, int32_t B, float* y, void* stream) {
    clear_error();
    SBR_CHECK_ARG(m && x && y, "mlp, x, y");
    SBR_CHECK_ARG(B >= 1 && B <= m->cfg.max_batch, "1 <= B <= max_batch");
    cudaStream_t s = (cudaStream_t)stream;
    return infer_fused(m, x, B, y, s);
}

sbr_status sbr_mlp_predict_layered(const sbr_mlp* m, const float* x, int32_t B, float* y, void* stream) {
    clear_error();
    SBR_CHECK_ARG(m && x && y, "mlp, x, y");
    SBR_CHECK_ARG(B >= 1 && B <= m->cfg.max_batch, "1 <= B <= max_batch");
    cudaStream_t s = (cudaStream_t)stream;
    SBR_TRY(forward_layered(m, x, B, s));
    ::sbr::note_launch(), k_take_outputs<<<nblk((int64_t)B * m->cfg.n_out), 256, 0, s>>>(m->P, B, m->cfg.n_out,
                                                                                      m->d_shift, m->d_scale, y);
    SBR_TRY_CUDA(cudaGetLastError());
    return SBR_OK;
}

int64_t sbr_mlp_param_count(const sbr_mlp* m) { return m ? m->n_params : 0; }

sbr_status sbr_mlp_params(sbr_mlp* m, float* params, int32_t mode, void* stream) {
    clear_error();
    SBR_CHECK_ARG(m && params, "mlp and params");
    SBR_CHECK_ARG(mode >= 0 && mode <= 2, "mode 0, 1 or 2");
    cudaStream_t s = (cudaStream_t)stream;
    const size_t bytes = sizeof(float) * (size_t)m->n_params;
    if (mode == 1) {
        SBR_TRY_CUDA(cudaMemcpyAsync(m->p, params, bytes, cudaMemcpyDeviceToDevice, s));
        return sync_images(m, s);
    }
    SBR_TRY_CUDA(cudaMemcpyAsync(params, mode == 0 ? m->p : m->g, bytes, cudaMemcpyDeviceToDevice, s));
    return SBR_OK;
}

sbr_status sbr_mlp_status(const sbr_mlp* m) {
    clear_error();
    SBR_CHECK_ARG(m != nullptr, "mlp");
    unsigned bits = 0;
    SBR_TRY_CUDA(cudaDeviceSynchronize());
    SBR_TRY_CUDA(cudaMemcpy(&bits, m->status, 4, cudaMemcpyDeviceToHost));
    return status_from_bits(bits);
}

sbr_status sbr_mlp_set_lr(sbr_mlp* m, float lr) {
    clear_error();
    SBR_CHECK_ARG(m != nullptr && lr > 0.f && std::isfinite(lr), "mlp and lr > 0");
    m->cfg.lr = lr;
    return SBR_OK;
}

void sbr_mlp_free(sbr_mlp* m) { free_mlp(m); }

}  // extern "C"
