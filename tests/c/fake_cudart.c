/* A stand-in for the CUDA runtime in which nothing runs: it keeps a log of
 * what the library would have queued, one line each (kernel launches with their
 * grid, block and programmatic attribute, memsets), for the tests of the
 * library's host side on machines without a GPU.  Linked into a copy of the
 * library in place of the runtime. */
#include <cuda_runtime_api.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#define SMS 152
#define PER_SM 4 /* resident CTAs of any kernel */

static char g_log[1 << 16];
static size_t g_len;
static int g_capturing, g_id_queries;
static char g_symbols[1 << 20] __attribute__((aligned(256)));
static struct { const void *host; const char *name; } g_kernel[512];
static int g_kernels;

static void put(const char *line)
{
    const size_t n = strlen(line);
    if (g_len + n + 1 < sizeof(g_log)) {
        memcpy(g_log + g_len, line, n + 1);
        g_len += n;
    }
}

const char *fake_log(void) { return g_log; }
void fake_reset(int capturing) { g_len = 0; g_log[0] = 0; g_capturing = capturing; g_id_queries = 0; }
int fake_id_queries(void) { return g_id_queries; }
int fake_wave(void) { return SMS * PER_SM; }

static const char *kernel_name(const void *f)
{
    for (int i = 0; i < g_kernels; ++i)
        if (g_kernel[i].host == f)
            return g_kernel[i].name;
    return "?";
}

/* -- what the compiler's generated code calls ------------------------------ */
void **__cudaRegisterFatBinary(void *b) { static void *h; (void)b; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void **h, const char *host, char *dev, const char *name, int l, void *t,
                            void *b, void *bd, void *gd, int *w)
{
    (void)h; (void)dev; (void)l; (void)t; (void)b; (void)bd; (void)gd; (void)w;
    if (g_kernels < (int)(sizeof(g_kernel) / sizeof(g_kernel[0]))) {
        g_kernel[g_kernels].host = host;
        g_kernel[g_kernels++].name = name;
    }
}
void __cudaRegisterVar(void **h, char *host, char *dev, const char *name, int e, size_t s, int c, int g)
{
    (void)h; (void)host; (void)dev; (void)name; (void)e; (void)s; (void)c; (void)g;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, void *s)
{
    (void)g; (void)b; (void)m; (void)s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *m, void *s)
{
    g->x = g->y = g->z = b->x = b->y = b->z = 1;
    *m = 0;
    *(void **)s = 0;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(void **k, const void *f) { *k = (void *)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(void *k, dim3 g, dim3 b, void **a, size_t m, void *s)
{
    char line[512];
    (void)a; (void)m; (void)s;
    snprintf(line, sizeof(line), "launch %s grid=%u block=%u programmatic=0\n", kernel_name(k), g.x, b.x);
    put(line);
    return cudaSuccess;
}

cudaError_t cudaLaunchKernel(const void *f, dim3 g, dim3 b, void **a, size_t m, cudaStream_t s)
{
    return __cudaLaunchKernel((void *)f, g, b, a, m, s);
}

/* -- the calls of the single-cover and batched entry points ------------------ */
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **a)
{
    char line[512];
    int pdl = 0;
    (void)a;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization)
            pdl = c->attrs[i].val.programmaticStreamSerializationAllowed;
    snprintf(line, sizeof(line), "launch %s grid=%u block=%u programmatic=%d\n", kernel_name(f),
             c->gridDim.x, c->blockDim.x, pdl);
    put(line);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t s)
{
    char line[64];
    (void)p; (void)v; (void)s;
    snprintf(line, sizeof(line), "memset %zu\n", n);
    put(line);
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d) { (void)a; (void)d; *v = SMS; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *f, int t, size_t m)
{
    (void)f; (void)t; (void)m;
    *n = PER_SM;
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, enum cudaStreamCaptureStatus *st)
{
    (void)s;
    *st = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamGetId(cudaStream_t s, unsigned long long *id)
{
    ++g_id_queries;
    *id = (uintptr_t)s;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *s) { (void)s; *p = g_symbols; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v) { (void)f; (void)a; (void)v; return cudaSuccess; }

static int ctx_get_current(void **c) { *c = &g_len; return 0; }
static int ctx_get_id(void *c, unsigned long long *id) { (void)c; *id = 7; return 0; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *n, void **f, unsigned v, unsigned long long fl,
                                             enum cudaDriverEntryPointQueryResult *q)
{
    (void)v; (void)fl;
    *f = strcmp(n, "cuCtxGetCurrent") == 0 ? (void *)ctx_get_current
         : strcmp(n, "cuCtxGetId") == 0    ? (void *)ctx_get_id
                                           : 0;
    *q = *f ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}

/* -- the pipeline's, the server's and the graph's: not simulated -------------- */
#define NO cudaErrorNotSupported
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned f) { (void)e; (void)f; return NO; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { (void)e; return NO; }
cudaError_t cudaEventQuery(cudaEvent_t e) { (void)e; return NO; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { (void)e; (void)s; return NO; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return NO; }
cudaError_t cudaFreeHost(void *p) { (void)p; return NO; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { (void)g; return NO; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t g) { (void)g; return NO; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long f) { (void)x; (void)g; (void)f; return NO; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t g, cudaStream_t s) { (void)g; (void)s; return NO; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned f) { (void)p; (void)n; (void)f; return NO; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) { (void)d; (void)s; (void)n; (void)k; (void)st; return NO; }
cudaError_t cudaPointerGetAttributes(struct cudaPointerAttributes *a, const void *p) { (void)a; (void)p; return NO; }
cudaError_t cudaSetDevice(int d) { (void)d; return NO; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m) { (void)s; (void)m; return NO; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned f) { (void)s; (void)f; return NO; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { (void)s; return NO; }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g) { (void)s; (void)g; return NO; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { (void)s; return NO; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) { (void)s; (void)e; (void)f; return NO; }
