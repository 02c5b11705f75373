// A kernel that writes the points of a later call and lets the work behind it
// on the stream start long before it has written them, as programmatic
// dependent launch allows: only a kernel that waits for its predecessor
// (griddepcontrol.wait) sees the points.  Every wait is bounded.
#include <cstdint>
#include <cuda_runtime.h>

__device__ __forceinline__ uint64_t now_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

__global__ void k_produce(float* dst, const float* src, int64_t n, uint64_t delay_ns) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint64_t t0 = now_ns();
    for (int i = 0; i < (1 << 22) && now_ns() - t0 < delay_ns; ++i) {}
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[i];
}

extern "C" int produce(float* dst, const float* src, int64_t n, uint64_t delay_ns, void* stream) {
    if (delay_ns > 100000000ull || n < 0) return 1;
    k_produce<<<16, 256, 0, static_cast<cudaStream_t>(stream)>>>(dst, src, n, delay_ns);
    return (int)cudaGetLastError();
}
