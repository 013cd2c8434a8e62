/* A CUDA runtime without a GPU, to be preloaded before libepic_interp.so:
 * device memory is host memory, kernels are noted and not run, and errors can
 * be ordered.  Copies from pageable memory are done as late as CUDA allows
 * ("may be synchronous with respect to the host", no more): at the next
 * synchronisation of their stream.  A source that has changed by then is
 * counted as stale. */
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>

struct copy { void *dst; const void *src; size_t n; cudaStream_t stream; void *at_call; };
static struct copy pending[256];
static int n_pending, n_stale, n_launch, fail_cooperative, fail_launch;
static struct { const void *function; int cooperative; unsigned grid; } launches[4096];
static struct { const void *function; const char *name; } names[256];
static int n_names;
static struct { char *p; size_t n; } pinned[64];
static int n_pinned;
static cudaError_t last;

static cudaError_t result(int e) {
    if (e) last = (cudaError_t)e;
    return (cudaError_t)e;
}
static int is_pinned(const void *p) {
    for (int i = 0; i < n_pinned; ++i)
        if ((const char *)p >= pinned[i].p && (const char *)p < pinned[i].p + pinned[i].n) return 1;
    return 0;
}

/* ---- what the tests ask ---- */
int fake_pending(void) { return n_pending; }
int fake_stale(void) { return n_stale; }
int fake_launches(void) { return n_launch; }
int fake_cooperative(int i) { return launches[i].cooperative; }
const char *fake_name(int i) {
    for (int j = 0; j < n_names; ++j)
        if (names[j].function == launches[i].function) return names[j].name;
    return "";
}
void fake_reset(void) { n_launch = n_stale = n_pending = 0; }
void fake_fail_cooperative(int e) { fail_cooperative = e; }  /* every cooperative launch fails with e */
void fake_fail_launch(int i, int e) { fail_launch = e ? (i << 16) | e : 0; }  /* launch i fails */

/* ---- memory ---- */
cudaError_t cudaMalloc(void **p, size_t n) {
    *p = aligned_alloc(256, (n + 511) / 256 * 256);
    return result(*p ? 0 : cudaErrorMemoryAllocation);
}
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned f) {
    (void)f;
    *p = calloc(1, n);
    pinned[n_pinned].p = *p;
    pinned[n_pinned++].n = n;
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { (void)p; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *symbol) {
    static void *memory;
    (void)symbol;
    if (!memory) memory = aligned_alloc(256, 64u << 20);
    *p = memory;
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, enum cudaMemcpyKind k) {
    (void)k;
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t s) { (void)s; memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) {
    if (k != cudaMemcpyHostToDevice || is_pinned(s)) {
        memcpy(d, s, n);
        return cudaSuccess;
    }
    struct copy c = {d, s, n, st, malloc(n)};
    memcpy(c.at_call, s, n);
    pending[n_pending++] = c;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    int left = 0;
    for (int i = 0; i < n_pending; ++i) {
        struct copy c = pending[i];
        if (c.stream != s) {
            pending[left++] = c;
            continue;
        }
        if (memcmp(c.src, c.at_call, c.n)) ++n_stale;
        memcpy(c.dst, c.at_call, c.n);
        free(c.at_call);
    }
    n_pending = left;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize(void) { return cudaStreamSynchronize(0); }

/* ---- device, streams, events, errors ---- */
cudaError_t cudaSetDevice(int d) { (void)d; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d) {
    (void)d;
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 232448;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(struct cudaDeviceProp *p, int d) {
    (void)d;
    memset(p, 0, sizeof *p);
    p->multiProcessorCount = 152;
    p->sharedMemPerBlockOptin = 232448;
    p->sharedMemPerMultiprocessor = 233472;
    p->reservedSharedMemPerBlock = 1024;
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *n, void **f, unsigned v, unsigned long long g,
                                             enum cudaDriverEntryPointQueryResult *q) {
    (void)n, (void)v, (void)g, (void)q;
    *f = 0;
    return cudaErrorUnknown;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned f) { (void)f; *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { (void)e, (void)s; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) { (void)s, (void)e, (void)f; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { cudaError_t e = last; last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t e) { (void)e; return "fake"; }

/* ---- kernels ---- */
void **__cudaRegisterFatBinary(void *f) { (void)f; static void *handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterVar(void **h, char *v, char *a, const char *n, int e, size_t s, int c, int g) {
    (void)h, (void)v, (void)a, (void)n, (void)e, (void)s, (void)c, (void)g;
}
void __cudaRegisterFunction(void **h, const char *f, char *df, const char *n, int t, void *a, void *b, void *c, void *d,
                            int *w) {
    (void)h, (void)df, (void)t, (void)a, (void)b, (void)c, (void)d, (void)w;
    names[n_names].function = f;
    names[n_names++].name = n;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
static struct { dim3 g, b; size_t m; cudaStream_t s; } pushed;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, void *s) {
    pushed.g = g, pushed.b = b, pushed.m = m, pushed.s = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *m, void *s) {
    *g = pushed.g, *b = pushed.b, *m = pushed.m, *(cudaStream_t *)s = pushed.s;
    return cudaSuccess;
}
static cudaError_t launch(const void *f, int cooperative, unsigned grid) {
    if (fail_launch && n_launch == fail_launch >> 16) return result(fail_launch & 0xffff);
    if (cooperative && fail_cooperative) return result(fail_cooperative);
    launches[n_launch].function = f;
    launches[n_launch].cooperative = cooperative;
    launches[n_launch++].grid = grid;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void **a, size_t m, cudaStream_t s) {
    (void)b, (void)a, (void)m, (void)s;
    return launch(k, 0, g.x);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **a) {
    (void)a;
    int cooperative = 0;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeCooperative) cooperative = c->attrs[i].val.cooperative;
    return launch(f, cooperative, c->gridDim.x);
}
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v) {
    (void)f, (void)a, (void)v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int t, size_t m, unsigned g) {
    (void)f, (void)t, (void)m, (void)g;
    *n = 2;
    return cudaSuccess;
}
