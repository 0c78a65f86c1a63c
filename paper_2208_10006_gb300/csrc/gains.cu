// Complex path gain g_n(f) (Eq. 1, 3, 6-10), one thread per (path, frequency);
// the arithmetic is path_gain (gains.cuh).
#include <algorithm>

#include "gains.cuh"

namespace sbr {
namespace {

// One thread per (path, frequency), consecutive threads on consecutive
// frequencies of a path. Bound by the FP32 pipe at large P F and by the chain of
// one path at small: small blocks, so that few items reach every SM. Measured
// for 102,400 paths of up to two reflections x 8 frequencies: 2517 us in FP64
// with eight lanes per item (one reflection each; idle lanes of an FP64 warp
// instruction cost as much as busy ones); with the targets of the same receivers
// (1436 us more) the two take 103 us now.
constexpr int kGainThreads = 64;

__global__ void __launch_bounds__(kGainThreads)
k_gains(int64_t P, int32_t F, const int32_t* __restrict__ nb, const int32_t* __restrict__ surf,
        const double* __restrict__ L, const double* __restrict__ jones, const sbr_material* __restrict__ mats,
        int32_t S, const double* __restrict__ freqs, const float* __restrict__ gamma,
        const float* __restrict__ disp, int pol, float2* __restrict__ g) {
    ::sbr::pdl_wait();
    const int64_t item = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= P * F) return;
    const int64_t p = item / F;
    const int32_t fi = (int32_t)(item - p * F);
    g[item] = path_gain(nb[p], surf + p * kKmax, L[p], jones + p * kJones, mats, S, freqs[fi],
                        gamma ? gamma + fi : nullptr, disp ? disp + fi : nullptr, pol);
}

}  // namespace

sbr_status gains_run(const sbr_path_list* pl, const sbr_material* mats, int32_t S,
                     const double* freqs, int32_t F, const float* gamma, const float* disp,
                     int32_t pol, float2* g, cudaStream_t s) {
    int64_t n = pl->P * (int64_t)F;
    if (n == 0) return SBR_OK;
    ::sbr::note_launch(), (void)::sbr::launch_pdl(k_gains, dim3((unsigned)((n + kGainThreads - 1) / kGainThreads)), dim3(kGainThreads), 0, s,
        pl->P, F, pl->nb, pl->surf, pl->L, pl->jones, mats, S, freqs, gamma, disp, pol, g);
    SBR_TRY_CUDA(cudaGetLastError());
    return SBR_OK;
}

}  // namespace sbr
