/* A CUDA runtime on the host for the library's own control flow, preloaded in a
 * process without a GPU: allocations are zeroed host memory, copies and memsets
 * are done, kernels are not run.  One allocation or memset of a given size can
 * be made to fail.  Kernels' limits of dynamic shared memory are kept as the runtime
 * keeps them, one for every thread of the process. */
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

enum { MAXBUF = 4096 };
static struct { void* p; size_t n; int zeroed; } buf[MAXBUF];
static int nbuf;
static size_t fail_malloc, fail_memset;
static double fill;
static struct { const void* f; int first, limit; } attr[MAXBUF];
static int nattr, refused, varied;

void fake_fail_malloc(size_t n) { fail_malloc = n; }
void fake_fail_memset(size_t n) { fail_memset = n; }
/* live buffers of n bytes that a memset has cleared */
int fake_cleared(size_t n) {
    int c = 0;
    for (int i = 0; i < nbuf; ++i) c += buf[i].p && buf[i].n == n && buf[i].zeroed;
    return c;
}

/* value of the doubles in new buffers */
void fake_fill(double v) { fill = v; }
/* launches refused for their dynamic shared memory, and limits set to more than one value */
int fake_refused(void) { return refused; }
int fake_varied(void) { return varied; }

int cudaMalloc(void** p, size_t n) {
    if (n == fail_malloc || nbuf == MAXBUF) { fail_malloc = 0; return 2; }
    buf[nbuf].p = *p = calloc(1, n ? n : 1);
    buf[nbuf].n = n;
    if (fill != 0.0)
        for (size_t i = 0; i < n / 8; ++i) ((double*)*p)[i] = fill;
    ++nbuf;
    return 0;
}
int cudaFree(void* p) {
    for (int i = 0; i < nbuf; ++i)
        if (buf[i].p == p) buf[i].p = 0;
    free(p);
    return 0;
}
int cudaMemset(void* p, int v, size_t n) {
    if (n == fail_memset) { fail_memset = 0; return 1; }
    memset(p, v, n);
    for (int i = 0; i < nbuf; ++i)
        if (buf[i].p == p && buf[i].n == n && v == 0) buf[i].zeroed = 1;
    return 0;
}
int cudaMemsetAsync(void* p, int v, size_t n, void* st) { (void)st; return cudaMemset(p, v, n); }
int cudaMemcpy(void* d, const void* s, size_t n, int k) { (void)k; memcpy(d, s, n); return 0; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int k, void* st) { (void)st; return cudaMemcpy(d, s, n, k); }
int cudaStreamSynchronize(void* st) { (void)st; return 0; }
int cudaFuncSetAttribute(const void* f, int a, int v) {
    int i = 0;
    if (a != 8) return 0;                       /* cudaFuncAttributeMaxDynamicSharedMemorySize */
    while (i < nattr && attr[i].f != f) ++i;
    if (i == nattr) { attr[i].f = f; attr[i].first = v; ++nattr; }
    varied += attr[i].first != v;
    attr[i].limit = v;
    return 0;
}
int cudaGetLastError(void) { return 0; }
const char* cudaGetErrorString(int e) { return e ? "failure made by the test" : "no error"; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int* v, int a, int d) { (void)a; (void)d; *v = 152; return 0; }
int __cudaGetKernel(void** k, const void* f) { *k = (void*)(uintptr_t)f; return 0; }
struct dim3 { unsigned x, y, z; };
int __cudaLaunchKernel(void* k, struct dim3 g, struct dim3 b, void** args, size_t smem, void* st) {
    int i = 0;
    (void)g; (void)b; (void)args; (void)st;
    while (i < nattr && attr[i].f != k) ++i;
    refused += smem > (i < nattr ? (size_t)attr[i].limit : 48u * 1024u);
    return 0;
}
