// Stand-ins for a few CUDA runtime calls, linked into a copy of the library
// with the linker's --wrap: they count and list what the library calls, and
// refuse launches of large clusters as a device does that cannot place them.
#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>

namespace {
constexpr int kMax = 4096;
struct Call {
    int kind;   // 1 cudaMalloc, 2 cudaMemsetAsync, 3 cudaMemcpyAsync, 4 refused launch, 5 launch
    size_t bytes;
};
Call g_calls[kMax];
std::atomic<int> g_n{0};
std::atomic<int> g_refuse{0};
void note(int kind, size_t bytes) {
    const int i = g_n.fetch_add(1);
    if (i < kMax) g_calls[i] = {kind, bytes};
}
}  // namespace

extern "C" {
cudaError_t __real_cudaMalloc(void**, size_t);
cudaError_t __real_cudaMemsetAsync(void*, int, size_t, cudaStream_t);
cudaError_t __real_cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t);
cudaError_t __real_cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**);

cudaError_t __wrap_cudaMalloc(void** p, size_t n) {
    note(1, n);
    return __real_cudaMalloc(p, n);
}
cudaError_t __wrap_cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) {
    note(2, n);
    return __real_cudaMemsetAsync(p, v, n, s);
}
cudaError_t __wrap_cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
    note(3, n);
    return __real_cudaMemcpyAsync(d, s, n, k, st);
}
cudaError_t __wrap_cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** a) {
    for (unsigned i = 0; g_refuse && i < c->numAttrs; ++i) {
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension && c->attrs[i].val.clusterDim.x > 8) {
            note(4, 0);
            cudaSetDevice(-1);   // (leaves an error behind, as a refused launch does)
            return cudaErrorInvalidClusterSize;
        }
    }
    note(5, 0);
    return __real_cudaLaunchKernelExC(c, f, a);
}

void calls_refuse_clusters(int on) { g_refuse = on; }
void calls_reset() { g_n = 0; }
int calls_count() { return g_n < kMax ? g_n.load() : kMax; }
int calls_kind(int i) { return g_calls[i].kind; }
size_t calls_bytes(int i) { return g_calls[i].bytes; }
}
