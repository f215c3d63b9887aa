// Two pretended GPUs for CPU tests, preloaded in front of the CUDA runtime:
// device memory is host memory, kernels do nothing, and a launch on a stream of
// another device than the current one fails, as it does on hardware (copies and
// waits do not).  FAKE_CUDA_NO_PINNED in the environment: no pinned memory.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>

namespace {
thread_local int t_device = 0;
thread_local cudaStream_t t_stream = nullptr;
struct Stream {
    int device;
};
cudaError_t launch(cudaStream_t s) {
    return reinterpret_cast<Stream*>(s)->device == t_device ? cudaSuccess : cudaErrorInvalidResourceHandle;
}
cudaError_t g_last = cudaSuccess;
}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int* d) { return *d = t_device, cudaSuccess; }
cudaError_t cudaSetDevice(int d) { return d < 0 || d > 1 ? cudaErrorInvalidDevice : (t_device = d, cudaSuccess); }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 227 * 1024;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() {
    cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
cudaError_t cudaMalloc(void** p, size_t n) { return *p = calloc(n ? n : 1, 1), cudaSuccess; }
cudaError_t cudaFree(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
    if (getenv("FAKE_CUDA_NO_PINNED")) return g_last = cudaErrorMemoryAllocation;
    return *p = calloc(n, 1), cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { return memmove(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t) {
    for (size_t i = 0; i < h; i++) memmove(static_cast<char*>(d) + i * dp, static_cast<const char*>(s) + i * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return memset(d, v, n), cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    return *s = reinterpret_cast<cudaStream_t>(new Stream{t_device}), cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { return delete reinterpret_cast<Stream*>(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
// 64 registers a thread, 228 KB of shared memory an SM, 1 KB of it per CTA for the system
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int threads, size_t smem) {
    const size_t by_regs = 65536 / 64 / threads, by_smem = 228 * 1024 / (smem + 1024);
    return *n = int(by_regs < by_smem ? by_regs : by_smem), cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int threads, size_t smem, unsigned) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, f, threads, smem);
}
cudaError_t cudaLibraryLoadData(cudaLibrary_t* l, const void*, cudaJitOption*, void**, unsigned, cudaLibraryOption*, void**, unsigned) {
    return *l = reinterpret_cast<cudaLibrary_t>(&g_last), cudaSuccess;
}
cudaError_t cudaLibraryGetKernel(cudaKernel_t* k, cudaLibrary_t, const char*) { return *k = nullptr, cudaSuccess; }
cudaError_t cudaLibraryUnload(cudaLibrary_t) { return cudaSuccess; }
cudaError_t cudaLaunchCooperativeKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t s) { return g_last = launch(s); }
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t s) { return g_last = launch(s); }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void*) { return *k = nullptr, cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t s) { return g_last = launch(s); }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, CUstream_st* s) { return t_stream = s, 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t* smem, void* s) {
    *smem = 0;
    return *static_cast<cudaStream_t*>(s) = t_stream, cudaSuccess;
}
}
