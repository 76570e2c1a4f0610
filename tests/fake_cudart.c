/* A CUDA runtime without a GPU: memory is the host's, kernels do nothing, and
 * the calls that allocate, free or wait are counted (fake_count).  For tests of
 * the library's host side, loaded in front of libcudart. */
#include <stddef.h>
#include <stdlib.h>
#include <string.h>

static int device, counts[3]; /* allocations, frees, waits */
void fake_set_device(int d) { device = d; }
int fake_count(int what) { return counts[what]; }

typedef void *cudaStream_t;
struct cudaFuncAttributes {
    size_t sharedSizeBytes, other[32];
};
int cudaGetDevice(int *d) { *d = device; return 0; }
int cudaMalloc(void **p, size_t n) { ++counts[0]; *p = malloc(n); return *p ? 0 : 2; }
int cudaHostAlloc(void **p, size_t n, unsigned f) { (void)f; *p = malloc(n); return *p ? 0 : 2; }
int cudaFree(void *p) { counts[1] += p != NULL; free(p); return 0; }
int cudaDeviceSynchronize(void) { ++counts[2]; return 0; }
int cudaStreamSynchronize(cudaStream_t s) { (void)s; ++counts[2]; return 0; }
int cudaStreamIsCapturing(cudaStream_t s, int *st) { (void)s; *st = 0; return 0; }
int cudaGetLastError(void) { return 0; }
int cudaMemset(void *p, int v, size_t n) { memset(p, v, n); return 0; }
int cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t s) { (void)s; memset(p, v, n); return 0; }
int cudaMemcpy(void *d, const void *s, size_t n, int k) { (void)k; memcpy(d, s, n); return 0; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int k, cudaStream_t st) { (void)k; (void)st; memcpy(d, s, n); return 0; }
int cudaMemcpyToSymbol(const void *d, const void *s, size_t n, size_t o, int k) { (void)d; (void)s; (void)n; (void)o; (void)k; return 0; }
int cudaDeviceGetAttribute(int *v, int a, int d)
{
    (void)d;
    *v = a == 16 ? 152 : (a == 97 ? 232448 : 0); /* multiprocessors, shared memory per block (opt-in) */
    return 0;
}
int cudaFuncGetAttributes(struct cudaFuncAttributes *a, const void *f) { (void)f; a->sharedSizeBytes = 1024; return 0; }
int cudaFuncSetAttribute(const void *f, int a, int v) { (void)f; (void)a; (void)v; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *f, int t, size_t s) { (void)f; (void)t; (void)s; *n = 1; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int t, size_t s, unsigned fl)
{
    (void)fl;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, f, t, s);
}
int cudaLaunchCooperativeKernel(void) { return 0; }
int __cudaLaunchKernel(void) { return 0; }
int __cudaGetKernel(void **k, const void *f) { *k = (void *)f; return 0; }
