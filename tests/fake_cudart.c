/* A stand-in for the CUDA runtime calls that libvloc.so makes, preloaded into
 * a process without a GPU: memory is addresses only, launches are recorded
 * and never run.  It keeps what a runtime keeps per device (a kernel's
 * dynamic shared-memory limit) and per stream (order by events), so the host
 * side of the library can be run through its C entry points.
 * Build: gcc -shared -fPIC -I$CUDA/include fake_cudart.c
 */
#include <cuda_runtime_api.h>
#include <stdint.h>

#define MAXF 4096
#define MAXL 65536
#define MAXM 4096

static int g_dev = 0;
static size_t g_free = (size_t)270 << 30, g_alloc = 0;
static uintptr_t g_next = (uintptr_t)1 << 40, g_handle = 4096;
static struct { const void* f; int dev; int bytes; } g_lim[MAXF];
static int g_nlim = 0;
static struct { uintptr_t at; size_t bytes; } g_mem[MAXM];
static int g_nmem = 0;
static uintptr_t g_launch[MAXL];   /* stream of each launch */
static int g_nlaunch = 0, g_cap = 0;
static cudaError_t g_last = cudaSuccess;

/* ---- controls of the test */
void fake_set_device(int d) { g_dev = d; }
void fake_set_free(size_t b) { g_free = g_alloc + b; }
size_t fake_allocated(void) { return g_alloc; }
int fake_limits(void) { return g_nlim; }   /* cudaFuncSetAttribute calls that raised a limit */
int fake_captures(void) { return g_cap; }   /* begun and not ended */
int fake_launches(void) { return g_nlaunch; }
uintptr_t fake_launch_stream(int i) { return g_launch[i]; }

static cudaError_t launched(const void* f, size_t smem, cudaStream_t st) {
    size_t limit = 48 * 1024;
    for (int i = 0; i < g_nlim; ++i)
        if (g_lim[i].f == f && g_lim[i].dev == g_dev && (size_t)g_lim[i].bytes > limit) limit = g_lim[i].bytes;
    if (smem > limit) return g_last = cudaErrorInvalidValue;
    if (g_nlaunch < MAXL) g_launch[g_nlaunch++] = (uintptr_t)st;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) {
    (void)d;
    *v = a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) {
    if (a != cudaFuncAttributeMaxDynamicSharedMemorySize) return cudaErrorInvalidValue;
    if (g_nlim == MAXF) return cudaErrorMemoryAllocation;
    g_lim[g_nlim].f = f; g_lim[g_nlim].dev = g_dev; g_lim[g_nlim++].bytes = v;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
    (void)args;
    return launched(f, c->dynamicSmemBytes, c->stream);
}
cudaError_t __cudaGetKernel(const void** k, const void* f) { *k = f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(const void* k, struct dim3 g, struct dim3 b, void** args, size_t smem, cudaStream_t st) {
    (void)g; (void)b; (void)args;
    return launched(k, smem, st);
}
cudaError_t cudaMalloc(void** p, size_t n) {
    if (n > g_free - g_alloc || g_nmem == MAXM) return g_last = cudaErrorMemoryAllocation;
    *p = (void*)g_next;
    g_mem[g_nmem].at = g_next; g_mem[g_nmem++].bytes = n;
    g_next += (n + 511) / 256 * 256;
    g_alloc += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    for (int i = 0; p && i < g_nmem; ++i)
        if (g_mem[i].at == (uintptr_t)p) { g_alloc -= g_mem[i].bytes; g_mem[i] = g_mem[--g_nmem]; return cudaSuccess; }
    return p ? (g_last = cudaErrorInvalidValue) : cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = g_free - g_alloc; *t = g_free; return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind k) { (void)d; (void)s; (void)n; (void)k; return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) {
    (void)d; (void)s; (void)n; (void)k; (void)st;
    return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { (void)d; (void)v; (void)n; return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) { (void)d; (void)v; (void)n; (void)st; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t e) { return e ? "error" : "no error"; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int b, size_t s, unsigned fl) {
    (void)f; (void)b; (void)s; (void)fl;
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* s, void** f, unsigned v, unsigned long long fl,
                                             enum cudaDriverEntryPointQueryResult* q) {
    (void)s; (void)v; (void)fl;
    *f = 0;
    if (q) *q = cudaDriverEntryPointSymbolNotFound;
    return cudaErrorNotSupported;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned fl) { (void)fl; *s = (cudaStream_t)(g_handle += 16); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned fl) { (void)s; (void)e; (void)fl; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)(g_handle += 16); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned fl) { (void)fl; return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { (void)e; (void)s; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) { (void)a; (void)b; *ms = 0.f; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m) { (void)s; (void)m; ++g_cap; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) { (void)s; --g_cap; *g = (cudaGraph_t)(g_handle += 16); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long fl) {
    (void)g; (void)fl;
    *x = (cudaGraphExec_t)(g_handle += 16);
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s) { (void)x; (void)s; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { (void)g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { (void)x; return cudaSuccess; }
