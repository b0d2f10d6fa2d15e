/* A stand-in for the CUDA runtime calls the library makes while it serves
 * requests, loaded before the real one: device memory is host memory, kernels do
 * nothing.  fake_fail_mallocs(skip, n): of the cudaMalloc calls from here on, let
 * `skip` pass and fail the next n. */
#include <stdlib.h>
#include <string.h>

static int skip_left = 0, fail_left = 0;
void fake_fail_mallocs(int skip, int n) {
    __atomic_store_n(&skip_left, skip, __ATOMIC_SEQ_CST);
    __atomic_store_n(&fail_left, n, __ATOMIC_SEQ_CST);
}
int fake_fails_left(void) { return __atomic_load_n(&fail_left, __ATOMIC_SEQ_CST); }

enum { kSuccess = 0, kNoMemory = 2 };
typedef struct { unsigned x, y, z; } dim3_t;

int cudaMalloc(void **p, size_t n) {
    if (fail_left > 0) {
        if (skip_left > 0) {
            skip_left--;
        } else {
            fail_left--;
            return kNoMemory;
        }
    }
    *p = malloc(n ? n : 1);
    return kSuccess;
}
int cudaMallocAsync(void **p, size_t n, void *st) { *p = malloc(n ? n : 1); return kSuccess; }
int cudaHostAlloc(void **p, size_t n, unsigned flags) { *p = malloc(n ? n : 1); return kSuccess; }
int cudaFree(void *p) { free(p); return kSuccess; }
int cudaFreeAsync(void *p, void *st) { free(p); return kSuccess; }
int cudaFreeHost(void *p) { free(p); return kSuccess; }
int cudaMemcpy(void *d, const void *s, size_t n, int kind) { memcpy(d, s, n); return kSuccess; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int kind, void *st) { memcpy(d, s, n); return kSuccess; }
int cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return kSuccess; }
int cudaMemsetAsync(void *d, int v, size_t n, void *st) { memset(d, v, n); return kSuccess; }
int cudaGetDevice(int *d) { *d = 0; return kSuccess; }
int cudaSetDevice(int d) { return kSuccess; }
int cudaGetDeviceCount(int *n) { *n = 1; return kSuccess; }
int cudaDeviceGetAttribute(int *v, int attr, int dev) { *v = 4; return kSuccess; }
int cudaDeviceGetDefaultMemPool(void **pool, int dev) { *pool = 0; return kSuccess; }
int cudaMemPoolSetAttribute(void *pool, int attr, void *v) { return kSuccess; }
int cudaStreamCreateWithFlags(void **st, unsigned flags) { *st = malloc(1); return kSuccess; }
int cudaStreamDestroy(void *st) { free(st); return kSuccess; }
int cudaStreamSynchronize(void *st) { return kSuccess; }
int cudaGetLastError(void) { return kSuccess; }
int cudaFuncSetAttribute(const void *f, int attr, int v) { return kSuccess; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *f, int threads, size_t smem) {
    *n = 2;
    return kSuccess;
}
int cudaLaunchKernelExC(const void *cfg, const void *f, void **args) { return kSuccess; }
int cudaLaunchKernel(const void *f, dim3_t g, dim3_t b, void **args, size_t smem, void *st) { return kSuccess; }
int __cudaLaunchKernel(void *f, dim3_t g, dim3_t b, void **args, size_t smem, void *st) { return kSuccess; }
int __cudaGetKernel(void **k, const void *f) { *k = (void *)f; return kSuccess; }
unsigned __cudaPushCallConfiguration(dim3_t g, dim3_t b, size_t smem, void *st) { return 0; }
int __cudaPopCallConfiguration(dim3_t *g, dim3_t *b, size_t *smem, void *st) {
    g->x = g->y = g->z = b->x = b->y = b->z = 1;
    *smem = 0;
    *(void **)st = 0;
    return kSuccess;
}
