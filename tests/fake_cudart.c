/* The CUDA runtime calls of libflb.so over host memory, to be loaded ahead of
 * libcudart: allocations come from the host heap (and are listed), kernels are not
 * run, and from allocation number fake_fail_from on (1, 2, ..; 0: never) every
 * cudaMalloc fails, as on a device that is full. */
#include <stdlib.h>
#include <string.h>

enum { MAXP = 256 };
int fake_fail_from = 0, fake_allocs = 0, fake_launches = 0;
void* fake_ptr[MAXP];
size_t fake_bytes[MAXP];
int fake_keep_arg = -1; /* argument (a pointer) of the launches to come that is kept */
void* fake_arg = 0;

int cudaMalloc(void** p, size_t n)
{
    ++fake_allocs;
    if (fake_fail_from && fake_allocs >= fake_fail_from) {
        *p = 0;
        return 2; /* cudaErrorMemoryAllocation */
    }
    *p = calloc(n ? n : 1, 1);
    for (int k = 0; k < MAXP; ++k)
        if (!fake_ptr[k]) {
            fake_ptr[k] = *p;
            fake_bytes[k] = n;
            break;
        }
    return 0;
}
int cudaFree(void* p)
{
    for (int k = 0; k < MAXP; ++k)
        if (p && fake_ptr[k] == p) fake_ptr[k] = 0;
    free(p);
    return 0;
}
int cudaMemset(void* p, int v, size_t n) { memset(p, v, n); return 0; }
int cudaMemsetAsync(void* p, int v, size_t n, void* s) { (void)s; memset(p, v, n); return 0; }
int cudaMemcpy(void* d, const void* s, size_t n, int kind) { (void)kind; memcpy(d, s, n); return 0; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int kind, void* st)
{
    (void)kind;
    (void)st;
    memcpy(d, s, n);
    return 0;
}
int cudaLaunchKernel(const void* f, ...) { (void)f; ++fake_launches; return 0; }
int cudaLaunchKernelExC(const void* c, const void* f, void** a)
{
    (void)c;
    (void)f;
    ++fake_launches;
    if (fake_keep_arg >= 0) fake_arg = *(void**)a[fake_keep_arg];
    return 0;
}
int cudaStreamCreateWithFlags(void** s, unsigned f) { (void)f; *s = malloc(1); return 0; }
int cudaStreamDestroy(void* s) { free(s); return 0; }
int cudaStreamSynchronize(void* s) { (void)s; return 0; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaSetDevice(int d) { (void)d; return 0; }
int cudaGetLastError(void) { return 0; }
int cudaDeviceGetAttribute(int* v, int a, int d) { (void)a; (void)d; *v = 152; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int b, size_t s, unsigned fl)
{
    (void)f;
    (void)b;
    (void)s;
    (void)fl;
    *n = 5;
    return 0;
}
int cudaFuncSetAttribute(const void* f, int a, int v) { (void)f; (void)a; (void)v; return 0; }
int cudaEventCreate(void** e) { *e = malloc(1); return 0; }
int cudaEventDestroy(void* e) { free(e); return 0; }
int cudaEventRecord(void* e, void* s) { (void)e; (void)s; return 0; }
int cudaEventSynchronize(void* e) { (void)e; return 0; }
int cudaEventElapsedTime(float* ms, void* a, void* b) { (void)a; (void)b; *ms = 1.0f; return 0; }
