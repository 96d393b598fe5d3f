// A CUDA runtime on the host: device memory is host memory, kernels are counted and not run, and the n-th call that can
// fail does so, once or from then on.
#pragma once

#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <set>

static std::mutex g_mu;                                    // (layers are planned on threads)
static long g_calls = 0, g_fails = -1;                     // calls so far; the one that fails (< 0: none)
static bool g_onwards = false;                             // and all behind it
static cudaError_t g_error = cudaErrorMemoryAllocation;
static std::set<void*> g_live;
static size_t g_bytes = 0;                                 // allocated so far
static int g_launches = 0;
static cudaError_t g_cooperative = cudaSuccess;            // what launches by cudaLaunchKernelExC return
static bool fails() { const long n = g_calls++; return g_fails >= 0 && (n == g_fails || (g_onwards && n > g_fails)); }

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) {
    std::lock_guard<std::mutex> lk(g_mu);
    *p = nullptr;
    if (fails()) return g_error;
    g_live.insert(*p = std::malloc(n));
    g_bytes += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    std::lock_guard<std::mutex> lk(g_mu);
    if (p && !g_live.erase(p)) { puts("freed what was not allocated"); std::exit(2); }
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) { *d = h; return cudaSuccess; }
static cudaError_t may_fail() { std::lock_guard<std::mutex> lk(g_mu); return fails() ? g_error : cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    const cudaError_t e = may_fail();
    if (e == cudaSuccess) std::memmove(d, s, n);
    return e;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
    const cudaError_t e = may_fail();
    if (e == cudaSuccess) std::memset(d, v, n);
    return e;
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t) {
    for (size_t i = 0; i < h; ++i) std::memmove((char*)d + i * dp, (const char*)s + i * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemset2DAsync(void* d, size_t dp, int v, size_t w, size_t h, cudaStream_t) {
    for (size_t i = 0; i < h; ++i) std::memset((char*)d + i * dp, v, w);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return may_fail(); }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return may_fail(); }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "failed on purpose"; }
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { ++g_launches; return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { ++g_launches; return g_cooperative; }
// what the compiler's own glue calls
void** __cudaRegisterFatBinary(void*) { static void* handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) { *g = *b = dim3(1); *s = 0; *(void**)st = nullptr; return cudaSuccess; }
}
