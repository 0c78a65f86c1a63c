// Index arithmetic of the synthesis that runs past 32 bits for arrays of up to 2^31 - 1
// elements: plain host and device functions.
#pragma once
#include <cstdint>
#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace sbr {

// first of the three coordinates of element e
__host__ __device__ __forceinline__ int64_t xyz_at(int64_t e) { return 3 * e; }

// tiles of t elements that cover n
__host__ __device__ __forceinline__ uint32_t tiles_of(int32_t n, int32_t t) { return ((uint32_t)n + (uint32_t)t - 1u) / (uint32_t)t; }

// LoS delays of the tensor forms, in blocks of 8 receive x 16 transmit elements
__host__ __device__ __forceinline__ int64_t dl_size(int64_t Nr, int64_t Nt) { return ((Nr + 7) / 8) * ((Nt + 15) / 16) * 128; }
// within a block: lane 4 (q % 8) + (p % 8) / 2 holds the pairs of columns p % 16 and p % 16 + 8
__host__ __device__ __forceinline__ int64_t dl_index(int32_t q, int32_t p, int32_t Nt) {
    return ((int64_t)(q >> 3) * tiles_of(Nt, 16) + (p >> 4)) * 128 + ((q & 7) * 4 + ((p & 7) >> 1)) * 4 + ((p >> 3) & 1) * 2 + (p & 1);
}

}  // namespace sbr
