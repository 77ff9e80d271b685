/* A CUDA runtime without a GPU, for tests of the library's host code: device
 * memory is host memory, kernels do not run, and one launch can be refused
 * (fake_refuse) the way the runtime does it: an error from the launch, which
 * cudaGetLastError reports once. */
#include <stdlib.h>
#include <string.h>

enum { kRefused = 701 /* cudaErrorLaunchOutOfResources */, kDeviceToHost = 2 };

static int g_launches, g_refuse = -1, g_error, g_memsets;
static unsigned g_dups;

/* the launch refused next (0: the next one; -1: none) */
void fake_refuse(int n) { g_launches = 0, g_refuse = n, g_error = 0; }
int fake_launches(void) { return g_launches; }
int fake_memsets(void) { return g_memsets; }
/* the tile duplicates that a read of the status words {flags, duplicates} finds */
void fake_dups(unsigned n) { g_dups = n; }

static int launch(void)
{
    if (g_launches++ == g_refuse)
        return g_error = kRefused;
    return 0;
}
int cudaLaunchKernelExC() { return launch(); }
int __cudaLaunchKernel() { return launch(); }
int cudaGetLastError(void)
{
    const int e = g_error;
    g_error = 0;
    return e;
}
int cudaPeekAtLastError(void) { return g_error; }
const char *cudaGetErrorString() { return "refused"; }

static int take(void **p, size_t n) { return (*p = calloc(n ? n : 1, 1)) ? 0 : 2; }
int cudaMalloc(void **p, size_t n) { return take(p, n); }
int cudaMallocHost(void **p, size_t n) { return take(p, n); }
int cudaFree(void *p) { return free(p), 0; }
int cudaFreeHost(void *p) { return free(p), 0; }

/* stream-ordered blocks, their bytes counted */
static size_t g_pool;
size_t fake_pool_bytes(void) { return g_pool; }
int cudaMallocAsync(void **p, size_t n)
{
    size_t *b = calloc(n + 64, 1);
    if (!b)
        return 2;
    *b = n;
    g_pool += n;
    return *p = (char *)b + 64, 0;
}
int cudaFreeAsync(void *p)
{
    size_t *b = (size_t *)((char *)p - 64);
    return g_pool -= *b, free(b), 0;
}
int cudaMemcpyAsync(void *dst, const void *src, size_t n, int kind)
{
    memcpy(dst, src, n);
    if (kind == kDeviceToHost && n == 8)
        ((unsigned *)dst)[1] = g_dups;
    return 0;
}
int cudaMemsetAsync(void *p, int v, size_t n) { return memset(p, v, n), ++g_memsets, 0; }

static int handle(void **h) { return *h = (void *)&g_launches, 0; }
int cudaStreamCreateWithFlags(void **h) { return handle(h); }
int cudaEventCreate(void **h) { return handle(h); }
int cudaStreamEndCapture(void *s, void **h) { return handle(h); }
int cudaGraphInstantiate(void **h) { return handle(h); }
int __cudaGetKernel(void **h) { return handle(h); }
void **__cudaRegisterFatBinary() { return (void **)&g_launches; }
int cudaGraphGetNodes(void *g, void *nodes, size_t *n) { return *n = 0, 0; }
int cudaGetDeviceCount(int *n) { return *n = 1, 0; }
int cudaGetDevice(int *d) { return *d = 0; }
int cudaDeviceGetAttribute(int *v) { return *v = 152, 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n) { return *n = 8, 0; }

#define OK(name) int name() { return 0; }
OK(__cudaPopCallConfiguration) OK(__cudaPushCallConfiguration) OK(__cudaRegisterFatBinaryEnd)
OK(__cudaRegisterFunction) OK(__cudaRegisterVar) OK(__cudaUnregisterFatBinary) OK(cudaDeviceSynchronize)
OK(cudaEventDestroy) OK(cudaEventElapsedTime) OK(cudaEventRecord) OK(cudaEventRecordWithFlags)
OK(cudaEventSynchronize) OK(cudaFuncSetAttribute) OK(cudaGetDriverEntryPointByVersion) OK(cudaGetSymbolAddress)
OK(cudaGraphDestroy) OK(cudaGraphEventRecordNodeGetEvent) OK(cudaGraphExecDestroy)
OK(cudaGraphExecEventRecordNodeSetEvent) OK(cudaGraphLaunch) OK(cudaGraphNodeGetType) OK(cudaSetDevice)
OK(cudaStreamBeginCapture) OK(cudaStreamDestroy) OK(cudaStreamSynchronize)
