/* A CUDA runtime in which nothing runs: launches are counted, and the k-th one fails
 * the way a real launch does, through the error that cudaGetLastError returns and
 * clears.  Preloaded before liblace in a process without a GPU. */
#include <stddef.h>

typedef struct {
    unsigned x, y, z;
} dim;

static int launched, fail_at, last;

void fake_reset(int k) { launched = 0, fail_at = k, last = 0; }
int fake_launched(void) { return launched; }

int __cudaPushCallConfiguration(dim g, dim b, size_t sm, void* s) { return (void)g, (void)b, (void)sm, (void)s, 0; }
int __cudaPopCallConfiguration(dim* g, dim* b, size_t* sm, void* s) {
    g->x = g->y = g->z = b->x = b->y = b->z = 1;
    *sm = 0;
    *(void**)s = 0;
    return 0;
}
int __cudaGetKernel(void** k, const void* f) { return *k = (void*)f, 0; }
int __cudaLaunchKernel(void* k, dim g, dim b, void** a, size_t sm, void* s) {
    (void)k, (void)g, (void)b, (void)a, (void)sm, (void)s;
    if (++launched == fail_at) last = 701; /* cudaErrorLaunchOutOfResources */
    return launched == fail_at ? 701 : 0;
}
int cudaGetLastError(void) {
    int e = last;
    last = 0;
    return e;
}
int cudaGetDevice(int* d) { return *d = 0, 0; }
int cudaDeviceGetAttribute(int* v, int a, int d) { return (void)a, (void)d, *v = 152, 0; }
int cudaFuncSetAttribute(const void* f, int a, int v) { return (void)f, (void)a, (void)v, 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int t, size_t sm, unsigned fl) {
    return (void)f, (void)t, (void)sm, (void)fl, *n = 2, 0;
}
int cudaMemsetAsync(void* p, int v, size_t n, void* s) { return (void)p, (void)v, (void)n, (void)s, 0; }
int cudaMemcpyAsync(void* d, const void* p, size_t n, int k, void* s) {
    return (void)d, (void)p, (void)n, (void)k, (void)s, 0;
}
int cudaStreamSynchronize(void* s) { return (void)s, 0; }
static int encode(void* m) { return (void)m, 0; } /* any tensor map */
int cudaGetDriverEntryPointByVersion(const char* n, void** f, unsigned v, unsigned long long fl, int* q) {
    return (void)n, (void)v, (void)fl, *f = (void*)encode, *q = 0, 0;
}
