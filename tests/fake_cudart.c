/* A CUDA runtime for tests of the library's host code without a GPU: device
 * memory is zeroed host memory, kernels are noted and not run, streams and
 * events are numbers, and every call that can fail can be made to.  Copies
 * from host memory on a stream read their source when the stream (or the
 * device) is next waited for, as late as a runtime may read memory that is not
 * page-locked; a source that has changed until then is noted. */
#include <stdarg.h>
#include <stddef.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <sys/mman.h>

#include <driver_types.h>

#define MAX 4096

static struct { const void *fun; char name[160]; } g_kernels[MAX];
static struct { char *p; size_t n; } g_blocks[MAX];
static struct { char *dst; const char *src; size_t n; uint64_t sum; } g_copies[MAX];
static int g_nkernels, g_ncopies, g_fail_after, g_capturing, g_events_pending;
static char g_fail_name[64], g_log[1 << 20];
static size_t g_log_len, g_held, g_limit = (size_t)1 << 60;
static uintptr_t g_next = 0x1000;
static cudaError_t g_last;
static struct { dim3 grid, block; size_t smem; void *stream; } g_config;

static void note(const char *fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    const int n = vsnprintf(g_log + g_log_len, sizeof g_log - g_log_len, fmt, ap);
    va_end(ap);
    if (n > 0 && g_log_len + (size_t)n < sizeof g_log) g_log_len += (size_t)n;
}

/* The next call of `name` but `after` fails; device memory is limited to
 * `bytes`; stream captures are on; events recorded have not been reached. */
void fake_fail(const char *name, int after) { snprintf(g_fail_name, sizeof g_fail_name, "%s", name); g_fail_after = after; }
void fake_limit(size_t bytes) { g_limit = bytes; }
void fake_capturing(int on) { g_capturing = on; }
void fake_events_pending(int on) { g_events_pending = on; }
size_t fake_held(void) { return g_held; }
const char *fake_log(void) { return g_log; }
void fake_clear(void) { g_log_len = 0; g_log[0] = 0; }

static cudaError_t result(const char *name, cudaError_t error)
{
    if (strcmp(name, g_fail_name) == 0 && g_fail_after-- == 0) {
        g_fail_name[0] = 0;
        return g_last = error;
    }
    return cudaSuccess;
}

static uint64_t sum_of(const char *p, size_t n)
{
    uint64_t h = 1469598103934665603ull;
    for (size_t i = 0; i < n; ++i) h = (h ^ (uint8_t)p[i]) * 1099511628211ull;
    return h;
}

static void land_copies(void)
{
    for (int i = 0; i < g_ncopies; ++i) {
        if (sum_of(g_copies[i].src, g_copies[i].n) != g_copies[i].sum) note("source changed before its copy: %zu bytes\n", g_copies[i].n);
        memcpy(g_copies[i].dst, g_copies[i].src, g_copies[i].n);
    }
    g_ncopies = 0;
}

static int is_device(const void *p)
{
    for (int i = 0; i < MAX; ++i)
        if (g_blocks[i].p && (const char *)p >= g_blocks[i].p && (const char *)p < g_blocks[i].p + g_blocks[i].n) return 1;
    return 0;
}

static const char *kernel_name(const void *fun)
{
    for (int i = 0; i < g_nkernels; ++i)
        if (g_kernels[i].fun == fun) return g_kernels[i].name;
    return "?";
}

/* registration and launches */
void **__cudaRegisterFatBinary(void *f) { (void)f; static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterVar(void **h, char *v, char *a, const char *n, int e, size_t s, int c, int g)
{ (void)h; (void)v; (void)a; (void)n; (void)e; (void)s; (void)c; (void)g; }
void __cudaRegisterFunction(void **h, const char *fun, char *dev, const char *name, int limit, void *a, void *b, void *c, void *d, int *e)
{
    (void)h; (void)dev; (void)limit; (void)a; (void)b; (void)c; (void)d; (void)e;
    if (g_nkernels == MAX) return;
    g_kernels[g_nkernels].fun = fun;
    snprintf(g_kernels[g_nkernels++].name, sizeof g_kernels[0].name, "%s", name);
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void *stream)
{ g_config.grid = grid; g_config.block = block; g_config.smem = smem; g_config.stream = stream; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream)
{ *grid = g_config.grid; *block = g_config.block; *smem = g_config.smem; *(void **)stream = g_config.stream; return cudaSuccess; }
cudaError_t __cudaGetKernel(void **k, const void *fun) { *k = (void *)fun; return cudaSuccess; }
static cudaError_t launch(const void *fun, dim3 grid, size_t smem, void *stream)
{
    cudaError_t e = result("launch", cudaErrorLaunchFailure);
    if (e == cudaSuccess && (grid.x == 0 || grid.y == 0)) e = g_last = cudaErrorInvalidConfiguration;
    if (e == cudaSuccess) note("launch %s grid %u shared %zu on %zx\n", kernel_name(fun), grid.x, smem, (size_t)stream);
    return e;
}
cudaError_t __cudaLaunchKernel(void *k, dim3 grid, dim3 block, void **args, size_t smem, void *st) { (void)block; (void)args; return launch(k, grid, smem, st); }
cudaError_t cudaLaunchKernel(const void *f, dim3 grid, dim3 block, void **args, size_t smem, void *st) { (void)block; (void)args; return launch(f, grid, smem, st); }
cudaError_t cudaLaunchCooperativeKernel(const void *f, dim3 grid, dim3 block, void **args, size_t smem, void *st) { (void)block; (void)args; return launch(f, grid, smem, st); }
cudaError_t cudaLaunchHostFunc(void *st, void (*fn)(void *), void *arg) { (void)st; fn(arg); return cudaSuccess; }

/* memory */
cudaError_t cudaMalloc(void **p, size_t n)
{
    cudaError_t e = result("cudaMalloc", cudaErrorMemoryAllocation);
    int i = 0;
    while (i < MAX && g_blocks[i].p) ++i;
    if (e == cudaSuccess && (g_held + n > g_limit || i == MAX)) e = g_last = cudaErrorMemoryAllocation;
    if (e != cudaSuccess) {
        note("refused %zu\n", n);
        return e;
    }
    char *q = mmap(NULL, n ? n : 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (q == MAP_FAILED) return g_last = cudaErrorMemoryAllocation;
    g_blocks[i].p = *p = q;
    g_blocks[i].n = n ? n : 1;
    g_held += g_blocks[i].n;
    note("malloc %zu\n", n);
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    for (int i = 0; p && i < MAX; ++i)
        if (g_blocks[i].p == p) {
            munmap(p, g_blocks[i].n);
            g_held -= g_blocks[i].n;
            note("free %zu\n", g_blocks[i].n);
            g_blocks[i].p = NULL;
            return cudaSuccess;
        }
    return p ? (g_last = cudaErrorInvalidValue) : cudaSuccess;
}
cudaError_t cudaMallocAsync(void **p, size_t n, void *st) { (void)st; return cudaMalloc(p, n); }
cudaError_t cudaFreeAsync(void *p, void *st) { (void)st; return cudaFree(p); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned f) { (void)f; *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) { *f = g_limit - g_held; *t = g_limit; return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, enum cudaMemcpyKind k) { (void)k; land_copies(); memcpy(d, s, n); return result("cudaMemcpy", cudaErrorUnknown); }
cudaError_t cudaMemset(void *d, int v, size_t n) { if (v) memset(d, v, n); return result("cudaMemset", cudaErrorUnknown); }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, void *st)
{
    (void)st;
    const cudaError_t e = result("cudaMemcpyAsync", cudaErrorUnknown);
    if (e != cudaSuccess) return e;
    if (k != cudaMemcpyHostToDevice || is_device(s) || g_ncopies == MAX) memcpy(d, s, n);
    else {
        g_copies[g_ncopies].dst = d;
        g_copies[g_ncopies].src = s;
        g_copies[g_ncopies].n = n;
        g_copies[g_ncopies++].sum = sum_of(s, n);
    }
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, void *st)
{
    (void)st;
    const cudaError_t e = result("cudaMemsetAsync", cudaErrorUnknown);
    if (e == cudaSuccess && v) memset(d, v, n);   /* (zeros: device memory starts as zeros here) */
    return e;
}

/* streams, events, graphs */
static void *number(void) { return (void *)(g_next += 0x10); }
cudaError_t cudaStreamCreateWithFlags(void **s, unsigned f) { (void)f; *s = number(); return cudaSuccess; }
cudaError_t cudaStreamDestroy(void *s) { (void)s; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(void *s) { const cudaError_t e = result("cudaStreamSynchronize", cudaErrorUnknown); land_copies(); note("sync %zx\n", (size_t)s); return e; }
cudaError_t cudaDeviceSynchronize(void) { land_copies(); return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(void *s, int *st) { (void)s; *st = g_capturing; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(void *s, int m) { (void)s; (void)m; return cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(int *m) { static int now; const int old = now; now = *m; *m = old; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(void *s, void **g) { (void)s; *g = number(); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(void **e, void *g, unsigned long long f) { (void)g; (void)f; *e = number(); return cudaSuccess; }
cudaError_t cudaGraphLaunch(void *e, void *s) { (void)e; (void)s; return cudaSuccess; }
cudaError_t cudaGraphDestroy(void *g) { (void)g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(void *g) { (void)g; return cudaSuccess; }
cudaError_t cudaEventCreate(void **e) { *e = number(); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(void **e, unsigned f) { (void)f; *e = number(); return cudaSuccess; }
cudaError_t cudaEventDestroy(void *e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventRecord(void *e, void *s) { note("record %zx on %zx\n", (size_t)e, (size_t)s); return cudaSuccess; }
cudaError_t cudaEventSynchronize(void *e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventQuery(void *e) { (void)e; return g_events_pending ? (g_last = cudaErrorNotReady) : cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, void *a, void *b) { (void)a; (void)b; *ms = 1.0f; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(void *s, void *e, unsigned f) { (void)f; note("wait %zx on %zx\n", (size_t)e, (size_t)s); return cudaSuccess; }

/* the device */
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { (void)d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d)
{
    (void)d;
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(struct cudaDeviceProp *p, int d) { (void)d; memset(p, 0, sizeof *p); snprintf(p->name, sizeof p->name, "none"); return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(struct cudaFuncAttributes *a, const void *f) { (void)f; memset(a, 0, sizeof *a); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v) { (void)f; (void)a; (void)v; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int b, size_t s, unsigned fl)
{ (void)f; (void)b; (void)s; (void)fl; *n = 1; return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *n, void **p, unsigned v, unsigned long long f, int *r)
{ (void)n; (void)v; (void)f; *p = NULL; *r = 1; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *s) { (void)s; static char a[64]; *p = a; return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t e) { (void)e; return "fake error"; }
cudaError_t cudaGetLastError(void) { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
