/* A CUDA runtime without a GPU, for host-side tests of the library's own
 * decisions: device memory is zeroed host memory, kernels do nothing but are
 * counted by name, and allocations can be made to fail.  The library's objects
 * are linked against it instead of the CUDA runtime. */
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>

enum { kMaxKernels = 1024 };
static const void* g_fun[kMaxKernels];
static const char* g_name[kMaxKernels];
static long g_count[kMaxKernels];
static unsigned g_grid[kMaxKernels];
static int g_kernels;
static size_t g_limit = (size_t)-1; /* an allocation above this many bytes fails */
static long g_fail_in = -1;         /* the allocation after this many more fails */
static long g_failed, g_live;
static size_t g_largest;
static cudaError_t g_last; /* until cudaGetLastError, as in the runtime */

/* ---- control ---- */
void fake_reset(void)
{
    memset(g_count, 0, sizeof(g_count));
    memset(g_grid, 0, sizeof(g_grid));
    g_limit = (size_t)-1;
    g_fail_in = -1;
    g_failed = 0;
    g_last = cudaSuccess;
}
/* the largest allocation asked for since the last call */
size_t fake_largest(void)
{
    const size_t n = g_largest;
    g_largest = 0;
    return n;
}
void fake_limit(size_t bytes) { g_limit = bytes; }
void fake_fail_in(long n) { g_fail_in = n; }
long fake_failed(void) { return g_failed; }
long fake_live(void) { return g_live; } /* allocations that have not been freed */
/* launches of the kernels whose mangled name contains `part`, and their largest grid.x */
long fake_launches(const char* part)
{
    long n = 0;
    for (int i = 0; i < g_kernels; ++i)
        if (strstr(g_name[i], part)) n += g_count[i];
    return n;
}
unsigned fake_grid(const char* part)
{
    unsigned n = 0;
    for (int i = 0; i < g_kernels; ++i)
        if (strstr(g_name[i], part) && g_grid[i] > n) n = g_grid[i];
    return n;
}

static cudaError_t launched(const void* fun, dim3 grid)
{
    for (int i = 0; i < g_kernels; ++i)
        if (g_fun[i] == fun) {
            ++g_count[i];
            if (grid.x > g_grid[i]) g_grid[i] = grid.x;
        }
    return cudaSuccess;
}

/* ---- memory ---- */
cudaError_t cudaMalloc(void** p, size_t n)
{
    *p = NULL;
    if (n > g_largest) g_largest = n;
    if (n > g_limit || (g_fail_in >= 0 && g_fail_in-- == 0)) {
        ++g_failed;
        return g_last = cudaErrorMemoryAllocation;
    }
    *p = calloc(1, n ? n : 1); /* untouched pages of large ones cost nothing */
    if (!*p) return cudaErrorMemoryAllocation;
    ++g_live;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p)
{
    if (p) --g_live;
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n)
{
    if (n <= (1u << 24)) memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) { (void)s; return cudaMemset(p, v, n); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind k)
{
    (void)k;
    memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t st)
{
    (void)st;
    return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaGetSymbolAddress(void** p, const void* sym) { *p = (void*)sym; return cudaSuccess; }

/* ---- device ---- */
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d)
{
    (void)d;
    switch (a) {
    case cudaDevAttrMultiProcessorCount: *v = 152; break;
    case cudaDevAttrMaxSharedMemoryPerMultiprocessor: *v = 228 * 1024; break;
    case cudaDevAttrMaxSharedMemoryPerBlockOptin: *v = 227 * 1024; break;
    default: *v = 1024; break;
    }
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaGetLastError(void)
{
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t e)
{
    return e == cudaErrorMemoryAllocation ? "out of memory" : e ? "error" : "no error";
}

/* ---- kernels ---- */
static char g_fat;
void** __cudaRegisterFatBinary(void* f) { (void)f; return (void**)&g_fat; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterVar(void** h, char* a, char* b, const char* c, int d, size_t e, int f, int g)
{
    (void)h; (void)a; (void)b; (void)c; (void)d; (void)e; (void)f; (void)g;
}
void __cudaRegisterFunction(void** h, const char* fun, char* dfun, const char* name, int t, void* a,
                            void* b, void* c, void* d, int* w)
{
    (void)h; (void)dfun; (void)t; (void)a; (void)b; (void)c; (void)d; (void)w;
    if (g_kernels == kMaxKernels) abort();
    g_fun[g_kernels] = fun;
    g_name[g_kernels++] = name;
}
static __thread struct {
    dim3 grid, block;
    size_t smem;
    void* st;
} g_cfg;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, void* s)
{
    g_cfg.grid = g; g_cfg.block = b; g_cfg.smem = m; g_cfg.st = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s)
{
    *g = g_cfg.grid; *b = g_cfg.block; *m = g_cfg.smem; *(void**)s = g_cfg.st;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(void** k, const void* fun) { *k = (void*)fun; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(void* k, dim3 g, dim3 b, void** a, size_t m, void* s)
{
    (void)b; (void)a; (void)m; (void)s;
    return launched(k, g);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fun, void** a)
{
    (void)a;
    return launched(fun, c->gridDim);
}
cudaError_t cudaLaunchCooperativeKernel(const void* fun, dim3 g, dim3 b, void** a, size_t m, cudaStream_t s)
{
    (void)b; (void)a; (void)m; (void)s;
    return launched(fun, g);
}
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v)
{
    (void)f; (void)a; (void)v;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(struct cudaFuncAttributes* a, const void* f)
{
    (void)f;
    memset(a, 0, sizeof(*a));
    a->numRegs = 64;
    a->maxThreadsPerBlock = 1024;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int t, size_t m,
                                                                   unsigned fl)
{
    (void)f; (void)fl;
    *n = t > 0 ? 1024 / t : 0;
    if (m && (size_t)*n > 227 * 1024 / m) *n = (int)(227 * 1024 / m);
    if (*n < 1) *n = 1;
    return cudaSuccess;
}

/* ---- streams, events, graphs: nothing runs, so nothing is ordered ---- */
static char g_handle;
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned f) { (void)f; *s = (cudaStream_t)&g_handle; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) { (void)s; (void)e; (void)f; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m) { (void)s; (void)m; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) { (void)s; *g = (cudaGraph_t)&g_handle; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)&g_handle; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned f) { (void)f; return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { (void)e; (void)s; return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t s, unsigned f) { (void)e; (void)s; (void)f; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t a, cudaEvent_t b) { (void)a; (void)b; *t = 1.f; return cudaSuccess; }
cudaError_t cudaGraphGetNodes(cudaGraph_t g, cudaGraphNode_t* nodes, size_t* n) { (void)g; (void)nodes; *n = 0; return cudaSuccess; }
cudaError_t cudaGraphNodeGetType(cudaGraphNode_t n, enum cudaGraphNodeType* t) { (void)n; *t = cudaGraphNodeTypeEmpty; return cudaSuccess; }
cudaError_t cudaGraphEventRecordNodeGetEvent(cudaGraphNode_t n, cudaEvent_t* e) { (void)n; *e = NULL; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long f) { (void)g; (void)f; *x = (cudaGraphExec_t)&g_handle; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s) { (void)x; (void)s; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { (void)x; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { (void)g; return cudaSuccess; }
cudaError_t cudaGraphExecEventRecordNodeSetEvent(cudaGraphExec_t x, cudaGraphNode_t n, cudaEvent_t e) { (void)x; (void)n; (void)e; return cudaSuccess; }
