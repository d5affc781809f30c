/* A stand-in for the CUDA runtime, enough for the receiver's host code to run without a GPU:
 * device memory is host memory, kernels are counted and not run, and one chosen call can be
 * made to fail with an error code, which is also left for cudaGetLastError as the runtime does. */
#include <stdlib.h>
#include <string.h>

static char g_name[64];
static int g_nth, g_code, g_last;
static long g_launches;

void fake_fail(const char *name, int nth, int code)
{
    strncpy(g_name, name, sizeof g_name - 1);
    g_nth = nth;
    g_code = code;
}
int fake_pending(void) { return g_nth > 0; }
long fake_launches(void) { return g_launches; }

static int call(const char *name)
{
    if (g_nth > 0 && !strcmp(name, g_name) && --g_nth == 0) return g_last = g_code;
    return 0;
}
int cudaGetLastError(void)
{
    int e = g_last;
    g_last = 0;
    return e;
}
const char *cudaGetErrorName(int e) { return e ? "injected" : "success"; }

int cudaMalloc(void **p, size_t n) { *p = aligned_alloc(256, (n + 255) / 256 * 256); return call("cudaMalloc"); }
int cudaFree(void *p) { free(p); return 0; }
int cudaMemset(void *p, int v, size_t n) { memset(p, v, n); return call("cudaMemset"); }
int cudaMemsetAsync(void *p, int v, size_t n, void *s) { (void)s; memset(p, v, n); return call("cudaMemsetAsync"); }
int cudaMemcpy(void *d, const void *s, size_t n, int k) { (void)k; memcpy(d, s, n); return call("cudaMemcpy"); }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int k, void *st)
{
    (void)k;
    (void)st;
    int e = call("cudaMemcpyAsync");
    if (!e) memcpy(d, s, n);
    return e;
}
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int *v, int a, int d) { (void)a; (void)d; *v = 152; return 0; }
int cudaGetSymbolAddress(void **p, const void *s) { (void)p; (void)s; return 1; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n) { *n = 1; return 0; }

#define HANDLE(name) int name(void **h) { *h = malloc(1); return call(#name); }
HANDLE(cudaEventCreate)
HANDLE(cudaEventCreateWithFlags)
HANDLE(cudaStreamCreateWithFlags)
int cudaEventDestroy(void *h) { free(h); return 0; }
int cudaStreamDestroy(void *h) { free(h); return 0; }
int cudaEventElapsedTime(float *ms) { *ms = 0.f; return 0; }

#define PLAIN(name) int name(void) { return call(#name); }
PLAIN(cudaDeviceSynchronize)
PLAIN(cudaEventRecord)
PLAIN(cudaEventSynchronize)
PLAIN(cudaFuncSetAttribute)
PLAIN(cudaGraphDestroy)
PLAIN(cudaGraphExecDestroy)
PLAIN(cudaGraphExecUpdate)
PLAIN(cudaGraphInstantiate)
PLAIN(cudaGraphLaunch)
PLAIN(cudaStreamBeginCapture)
PLAIN(cudaStreamEndCapture)
PLAIN(cudaStreamSynchronize)
PLAIN(cudaStreamWaitEvent)

int cudaLaunchKernelExC(void) { g_launches++; return call("launch"); }
int __cudaLaunchKernel(void) { g_launches++; return call("launch"); }
int __cudaGetKernel(void) { return 0; }
unsigned __cudaPushCallConfiguration(void) { return 0; }
int __cudaPopCallConfiguration(void) { return 0; }
void **__cudaRegisterFatBinary(void) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void) {}
void __cudaUnregisterFatBinary(void) {}
void __cudaRegisterFunction(void) {}
void __cudaRegisterVar(void) {}
