/* A CUDA runtime that runs no kernel, for host tests of libbvf (preloaded in
 * place of libcudart): device memory is host memory, copies are memcpy, a
 * launch is one line of a log.  Tests arm failures of allocations and of
 * stream or event creation and read the log and the counters. */
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <sys/mman.h>

/* allocations above this are address space only: never touched, never freed */
#define FAKE_LARGE ((size_t)256 << 20)

static int g_fail_malloc, g_fail_object;        /* the n-th from now fails (0: none) */
static long long g_mallocs, g_malloc_bytes, g_instantiated, g_launches, g_last_error_calls;
static size_t g_free_mem = (size_t)200 << 30;
static int g_pending;                           /* error cudaGetLastError would return */
static int g_read_u32 = -1;                     /* value of 4-byte copies to the host */
static struct { const void *fun; char name[256]; } g_fun[2048];
static int g_n_fun;
static char *g_log;
static size_t g_log_len, g_log_cap;

void fake_fail_malloc(int n) { g_fail_malloc = n; }
void fake_fail_object(int n) { g_fail_object = n; }
void fake_free_mem(size_t n) { g_free_mem = n; }
void fake_set_pending(int e) { g_pending = e; }
int fake_pending(void) { return g_pending; }
void fake_read_u32(int v) { g_read_u32 = v; }
long long fake_mallocs(void) { return g_mallocs; }
long long fake_malloc_bytes(void) { return g_malloc_bytes; }
long long fake_instantiated(void) { return g_instantiated; }
long long fake_launches(void) { return g_launches; }
/* "name grid-x grid-y grid-z smem" of every launch since the last clear, one a line */
const char *fake_log(void) { return g_log ? g_log : ""; }
void fake_log_clear(void)
{
    g_log_len = 0;
    if (g_log) g_log[0] = 0;
}

static void launched(const void *fun, struct dim3 g, size_t smem)
{
    const char *name = "?";
    char line[400];
    int i, n;
    for (i = 0; i < g_n_fun; ++i)
        if (g_fun[i].fun == fun) name = g_fun[i].name;
    n = snprintf(line, sizeof line, "%s %u %u %u %zu\n", name, g.x, g.y, g.z, smem);
    if (g_log_len + n + 1 > g_log_cap) {
        g_log_cap = 2 * (g_log_len + n + 1);
        g_log = realloc(g_log, g_log_cap);
    }
    memcpy(g_log + g_log_len, line, n + 1);
    g_log_len += n;
    ++g_launches;
}

static cudaError_t failed(int *countdown, cudaError_t e)
{
    if (*countdown > 0 && --*countdown == 0) {
        g_pending = e;
        return e;
    }
    return cudaSuccess;
}

/* memory */
static void *g_large[256];
static int g_n_large;
static int is_large(const void *p)
{
    int i;
    for (i = 0; i < g_n_large; ++i)
        if (g_large[i] == p) return 1;
    return 0;
}
cudaError_t cudaMalloc(void **p, size_t n)
{
    ++g_mallocs;
    if (failed(&g_fail_malloc, cudaErrorMemoryAllocation)) return cudaErrorMemoryAllocation;
    if (n > FAKE_LARGE)
        *p = mmap(0, n, PROT_NONE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    else
        *p = calloc(1, n ? n : 1);
    if (!*p || *p == MAP_FAILED) return cudaErrorMemoryAllocation;
    if (n > FAKE_LARGE) {
        if (g_n_large == 256) abort();
        g_large[g_n_large++] = *p;
    }
    g_malloc_bytes += n;
    return cudaSuccess;
}
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t s) { (void)s; return cudaMalloc(p, n); }
cudaError_t cudaFree(void *p)
{
    if (!is_large(p)) free(p);
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t s) { (void)s; return cudaFree(p); }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) { *f = g_free_mem; *t = (size_t)280 << 30; return cudaSuccess; }
cudaError_t cudaMemset(void *p, int v, size_t n)
{
    if (!is_large(p)) memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t s) { (void)s; return cudaMemset(p, v, n); }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, enum cudaMemcpyKind k)
{
    memcpy(d, s, n);
    if (k == cudaMemcpyDeviceToHost && n == 4 && g_read_u32 >= 0) memcpy(d, &g_read_u32, 4);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t st)
{
    (void)st;
    return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemcpy2D(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h,
                         enum cudaMemcpyKind k)
{
    size_t r;
    (void)k;
    for (r = 0; r < h; ++r) memcpy((char *)d + r * dp, (const char *)s + r * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h,
                              enum cudaMemcpyKind k, cudaStream_t st)
{
    (void)st;
    return cudaMemcpy2D(d, dp, s, sp, w, h, k);
}
cudaError_t cudaGetSymbolAddress(void **p, const void *sym) { (void)sym; *p = 0; return cudaErrorInvalidSymbol; }

/* streams, events, graphs: small numbered handles */
static void *handle(void)
{
    static size_t n = 16;
    return (void *)(n += 16);
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned f)
{
    (void)f;
    if (failed(&g_fail_object, cudaErrorUnknown)) return cudaErrorUnknown;
    *s = handle();
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned f)
{
    (void)f;
    if (failed(&g_fail_object, cudaErrorUnknown)) return cudaErrorUnknown;
    *e = handle();
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s)
{
    (void)s;
    return e ? cudaSuccess : cudaErrorInvalidResourceHandle;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b) { (void)a; (void)b; *ms = 1.0f; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f)
{
    (void)s; (void)f;
    return e ? cudaSuccess : cudaErrorInvalidResourceHandle;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m) { (void)s; (void)m; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g) { (void)s; *g = handle(); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long f)
{
    (void)g; (void)f;
    ++g_instantiated;
    *x = handle();
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s) { (void)s; return x ? cudaSuccess : cudaErrorInvalidValue; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { (void)g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { (void)x; return cudaSuccess; }

/* device, errors */
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d)
{
    (void)d;
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void)
{
    cudaError_t e = (cudaError_t)g_pending;
    g_pending = 0;
    return e;
}
const char *cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "fake error"; }
static CUresult fake_encode(void) { return CUDA_SUCCESS; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *name, void **f, unsigned v, unsigned long long flags,
                                             enum cudaDriverEntryPointQueryResult *r)
{
    (void)v; (void)flags;
    *f = strcmp(name, "cuTensorMapEncodeTiled") ? 0 : (void *)fake_encode;
    *r = *f ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}

/* kernels: largest shared memory asked for per kernel, and launches */
static struct { const void *fun; int bytes; } g_smem[2048];
static int g_n_smem;
cudaError_t cudaFuncSetAttribute(const void *fun, enum cudaFuncAttribute a, int v)
{
    int i;
    if (a != cudaFuncAttributeMaxDynamicSharedMemorySize) return cudaSuccess;
    for (i = 0; i < g_n_smem && g_smem[i].fun != fun; ++i) {}
    if (i == g_n_smem) ++g_n_smem;
    g_smem[i].fun = fun;
    g_smem[i].bytes = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int b, size_t sm,
                                                                   unsigned fl)
{
    (void)f; (void)b; (void)sm; (void)fl;
    *n = 4;
    return cudaSuccess;
}
/* as the runtime: more than 48 KB only up to the kernel's own limit */
static cudaError_t launch(const void *fun, struct dim3 g, size_t smem)
{
    int i, lim = 48 * 1024;
    for (i = 0; i < g_n_smem; ++i)
        if (g_smem[i].fun == fun && g_smem[i].bytes > lim) lim = g_smem[i].bytes;
    if (smem > (size_t)lim) {
        g_pending = cudaErrorInvalidValue;
        return cudaErrorInvalidValue;
    }
    launched(fun, g, smem);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **a)
{
    (void)a;
    return launch(f, c->gridDim, c->dynamicSmemBytes);
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, struct dim3 g, struct dim3 b, void **a, size_t sm, cudaStream_t s)
{
    (void)b; (void)a; (void)s;
    return launch((const void *)k, g, sm);
}
static struct dim3 c_grid, c_block;
static size_t c_smem;
static void *c_stream;
unsigned __cudaPushCallConfiguration(struct dim3 g, struct dim3 b, size_t sm, void *s)
{
    c_grid = g;
    c_block = b;
    c_smem = sm;
    c_stream = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(struct dim3 *g, struct dim3 *b, size_t *sm, void *s)
{
    *g = c_grid;
    *b = c_block;
    *sm = c_smem;
    *(void **)s = c_stream;
    return cudaSuccess;
}
void **__cudaRegisterFatBinary(void *f) { (void)f; return (void **)handle(); }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterVar(void **h, char *v, char *a, const char *n, int e, size_t s, int c, int g)
{
    (void)h; (void)v; (void)a; (void)n; (void)e; (void)s; (void)c; (void)g;
}
void __cudaRegisterFunction(void **h, const char *fun, char *dev, const char *name, int lim, void *t, void *b,
                            void *bd, void *gd, int *ws)
{
    (void)h; (void)dev; (void)lim; (void)t; (void)b; (void)bd; (void)gd; (void)ws;
    if (g_n_fun == 2048) return;
    g_fun[g_n_fun].fun = fun;
    snprintf(g_fun[g_n_fun].name, sizeof g_fun[0].name, "%s", name);
    ++g_n_fun;
}
