// fake_cuda.cpp -- a CUDA runtime on host memory, for tests that compile the library's
// host code (xeng_api.cu, no kernels) with the host compiler and make calls of it fail.
// Allocations are counted; a chosen one, or all above a size, fail.
#include <cstdlib>
#include <cstring>
#include <map>

#include "xeng_internal.h"

namespace {
std::map<void *, size_t> g_live;
long g_allocs = 0, g_fail_at = -1;
size_t g_fail_above = ~(size_t)0;
cudaError_t g_last = cudaSuccess;
}  // namespace

extern "C" {

// Count from 0 again; allocation number `at` (-1: none) and those above `bytes` fail.
void fake_allocs(long at, size_t bytes)
{
    g_allocs = 0;
    g_fail_at = at;
    g_fail_above = bytes;
}
long fake_alloc_count() { return g_allocs; }
long fake_live() { return (long)g_live.size(); }
size_t fake_live_bytes()
{
    size_t n = 0;
    for (auto &p : g_live) n += p.second;
    return n;
}

cudaError_t cudaMalloc(void **p, size_t n)
{
    if (g_allocs++ == g_fail_at || n > g_fail_above || !(*p = malloc(n ? n : 1))) return g_last = cudaErrorMemoryAllocation;
    g_live[*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    if (!p) return cudaSuccess;
    if (!g_live.erase(p)) return g_last = cudaErrorInvalidValue;
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind)
{
    if (!d || !s) return g_last = cudaErrorInvalidValue;
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n)
{
    if (!d) return g_last = cudaErrorInvalidValue;
    memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaGetLastError()
{
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
cudaError_t cudaPeekAtLastError() { return g_last; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d)
{
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int)
{
    memset(p, 0, sizeof *p);
    p->major = 10;
    p->minor = 3;
    p->multiProcessorCount = 152;
    return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t *free_b, size_t *total_b)
{
    *free_b = *total_b = (size_t)280 << 30;
    return cudaSuccess;
}

}  // extern "C"

namespace xeng {

cudaError_t status_alloc(int **d_err, int **h_err)
{
    *d_err = (int *)calloc(1, sizeof(StatusBlock));
    *h_err = (int *)calloc(1, sizeof(int));
    return cudaSuccess;
}
void status_free(int *d_err, int *h_err)
{
    free(d_err);
    free(h_err);
}
int single_pass_force_from_env() { return 0; }
void small_scratch_free(SmallScratch *) {}

}  // namespace xeng
