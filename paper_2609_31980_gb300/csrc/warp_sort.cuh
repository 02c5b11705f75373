// warp_sort.cuh — sorting of (d2, index) keys across a warp and of short lists
// by pairs of lanes, shared by the selection kernel, the half-cell scan and the
// tensor-core path.
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

__device__ __forceinline__ void cswap(uint32_t& a, uint32_t& b) {
    const uint32_t lo = min(a, b), hi = max(a, b);
    a = lo;
    b = hi;
}

// Batcher's odd-even merge sort of P keys in registers.
template <int P>
__device__ __forceinline__ void sort_regs(uint32_t (&k)[P]) {
#pragma unroll
    for (int p = 1; p < P; p <<= 1) {
#pragma unroll
        for (int q = p; q >= 1; q >>= 1) {
#pragma unroll
            for (int i = 0; i < P; ++i) {
                const int j = q % p;   // the step's first key
                if (i >= j && (i - j) % (2 * q) < q && i + q < P && i / (2 * p) == (i + q) / (2 * p))
                    cswap(k[i], k[i + q]);
            }
        }
    }
}

// Sort 2 P 32-bit keys held half each by lanes l and l ^ 16 (the lower lane
// ends with the smaller P): each half by itself, one exchange, one merge.  The
// keys' low five bits are their places; returns whether two neighbouring keys
// of this lane, or the two lanes' edge, agree in all other bits.
template <int P>
__device__ __forceinline__ bool sort_pair(uint32_t (&k)[P]) {
    const int hh = (threadIdx.x & 31) >> 4;
    sort_regs<P>(k);
    // the lower lane keeps the P smallest, the upper the rest (each a bitonic
    // sequence), then one merge in registers
    {
        uint32_t o[P];
#pragma unroll
        for (int i = 0; i < P; ++i) o[i] = __shfl_xor_sync(kFull, k[P - 1 - i], 16);
#pragma unroll
        for (int i = 0; i < P; ++i) k[i] = hh ? max(k[i], o[i]) : min(k[i], o[i]);
    }
#pragma unroll
    for (int j = P / 2; j > 0; j >>= 1)
#pragma unroll
        for (int i = 0; i < P; ++i)
            if ((i & j) == 0) cswap(k[i], k[i | j]);
    uint32_t near = 32u;
#pragma unroll
    for (int i = 0; i + 1 < P; ++i) near = min(near, k[i] ^ k[i + 1]);
    const uint32_t edge = hh ? k[0] : k[P - 1];
    near = min(near, edge ^ __shfl_xor_sync(kFull, edge, 16));
    return near < 32u;
}

}  // namespace frnn
