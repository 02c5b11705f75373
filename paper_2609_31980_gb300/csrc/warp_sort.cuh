// warp_sort.cuh — sorting of (d2, index) keys across a warp, shared by the
// selection kernel and the half-cell scan.
#pragma once

#include "frnn_internal.cuh"

namespace frnn {

constexpr uint32_t kFull = 0xffffffffu;

__device__ __forceinline__ uint64_t make_key(float d2, int32_t j) {
    return ((uint64_t)__float_as_uint(d2) << 32) | (uint32_t)j;
}

// Ascending sort of 32 P keys held P a lane (key i = lane * P + p): a bitonic
// network, steps within a lane on registers, across lanes by shuffles.
template <int P>
__device__ __forceinline__ void warp_sort(uint64_t (&k)[P]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int len = 2; len <= 32 * P; len <<= 1) {
#pragma unroll
        for (int j = len >> 1; j > 0; j >>= 1) {
            if (j >= P) {
                const int jl = j / P;   // lanes apart
                // direction from the key's index: the bits at and above P are the lane's
                const bool up = len >= 32 * P || ((lane * P) & len) == 0;
                const bool take_min = ((lane & jl) == 0) == up;
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    const uint64_t o = __shfl_xor_sync(kFull, k[p], jl);
                    k[p] = (take_min == (o < k[p])) ? o : k[p];
                }
            } else {
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    if ((p & j) == 0) {
                        const bool up = len >= P ? ((lane * P) & len) == 0 || len >= 32 * P : (p & len) == 0;
                        const uint64_t x = k[p], y = k[p | j];
                        const bool sw = (x > y) == up;
                        k[p] = sw ? y : x;
                        k[p | j] = sw ? x : y;
                    }
                }
            }
        }
    }
}

}  // namespace frnn
