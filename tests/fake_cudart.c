/* A CUDA runtime with no device behind it, for the library's host code on the CPU: device
 * memory is addresses alone, kernels are launched by name only, copies to the host give
 * zeros.  It keeps what the host code has to get right and a real device would refuse:
 * the shared memory of a launch against what the kernel was allowed on the current device,
 * and the memory a device has.  Linked with the library's objects in place of cudart. */
#include <cuda_runtime_api.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#define MAXF 4096
#define MAXDEV 4
static struct { const void *fun; char name[200]; int smem[MAXDEV]; } funcs[MAXF];
static int nfuncs, device;
static cudaError_t last;
static size_t capacity = (size_t)280 << 30, used, peak;
#define MAXP 65536
static struct { void *p; size_t n; } mem[MAXP];
static int nmem;
static char *next_addr = (char *)0x100000000000ull;
static char *text;
static size_t text_len, text_cap;

static cudaError_t fail(cudaError_t e) { last = e; return e; }
static int find(const void *f)
{
    for (int i = 0; i < nfuncs; ++i)
        if (funcs[i].fun == f) return i;
    return -1;
}
/* what the tests set and read */
void fake_device(int d) { device = d; }
void fake_capacity(size_t bytes) { capacity = bytes; }
size_t fake_used(void) { return used; }
size_t fake_peak(void) { size_t p = peak; peak = used; return p; }
/* one line per launch through the extended interface: device, shared memory, a number
 * (k_nd_level: the entries of a staged tile; others: the share of the L1 that the launch asks
 * for, 0 if none), threads, kernel ("-" where refused) */
const char *fake_log(void) { return text ? text : ""; }
void fake_clear(void) { text_len = 0; if (text) text[0] = 0; }
static void say(int d, size_t smem, int arg, long threads, const char *name)
{
    if (text_cap - text_len < 400) text = realloc(text, text_cap = 2 * text_cap + 4096);
    text_len += (size_t)sprintf(text + text_len, "%d %zu %d %ld %s\n", d, smem, arg, threads, name);
}

void **__cudaRegisterFatBinary(void *b) { return (void **)b; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterVar(void **h, char *a, char *b, const char *c, int d, size_t e, int f, int g)
{ (void)h; (void)a; (void)b; (void)c; (void)d; (void)e; (void)f; (void)g; }
void __cudaRegisterFunction(void **h, const char *fun, char *dev, const char *name, int lim, void *t, void *b, void *bd, void *gd, int *w)
{
    (void)h; (void)dev; (void)lim; (void)t; (void)b; (void)bd; (void)gd; (void)w;
    if (nfuncs == MAXF) abort();
    funcs[nfuncs].fun = fun;
    snprintf(funcs[nfuncs].name, sizeof funcs[0].name, "%s", name);
    for (int d = 0; d < MAXDEV; ++d) funcs[nfuncs].smem[d] = 48 * 1024;
    ++nfuncs;
}
static struct { dim3 g, b; size_t smem; cudaStream_t s; } call;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s)
{ call.g = g; call.b = b; call.smem = smem; call.s = s; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s)
{ *g = call.g; *b = call.b; *smem = call.smem; *(cudaStream_t *)s = call.s; return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
static cudaError_t launch(const void *f, dim3 g, dim3 b, size_t smem, void **args, int shared, int log)
{
    const int i = find(f);
    const long threads = (long)g.x * g.y * g.z * b.x * b.y * b.z;
    if (i < 0) return fail(cudaErrorInvalidDeviceFunction);
    const int arg = strstr(funcs[i].name, "k_nd_level") ? *(int *)args[7] : shared;
    if (smem > (size_t)funcs[i].smem[device]) { say(device, smem, arg, threads, "-"); return fail(cudaErrorInvalidValue); }
    if (log) say(device, smem, arg, threads, funcs[i].name);
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void **args, size_t smem, cudaStream_t s)
{ (void)s; return launch((const void *)k, g, b, smem, args, 0, 0); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args)
{
    int shared = 0;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributePreferredSharedMemoryCarveout) shared = (int)c->attrs[i].val.sharedMemCarveout;
    return launch(f, c->gridDim, c->blockDim, c->dynamicSmemBytes, args, shared, 1);
}
cudaError_t cudaLaunchCooperativeKernel(const void *f, dim3 g, dim3 b, void **args, size_t smem, cudaStream_t s)
{ (void)s; return launch(f, g, b, smem, args, 0, 0); }
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v)
{
    const int i = find(f);
    if (i < 0) return fail(cudaErrorInvalidDeviceFunction);
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) funcs[i].smem[device] = v;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(struct cudaFuncAttributes *a, const void *f) { (void)f; memset(a, 0, sizeof *a); return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int t, size_t s, unsigned fl)
{ (void)f; (void)s; (void)fl; *n = 2048 / t < 32 ? 2048 / t : 32; return cudaSuccess; }

cudaError_t cudaGetLastError(void) { cudaError_t e = last; last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "fake error"; }
cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d)
{
    (void)d;
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerMultiprocessor ? 233472
       : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 1;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(struct cudaDeviceProp *p, int d) { (void)d; memset(p, 0, sizeof *p); p->multiProcessorCount = 152; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *s) { (void)s; *p = next_addr; return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *s, void **p, unsigned v, unsigned long long f, enum cudaDriverEntryPointQueryResult *r)
{ (void)s; (void)v; (void)f; *p = 0; if (r) *r = cudaDriverEntryPointSymbolNotFound; return cudaSuccess; }

cudaError_t cudaMalloc(void **p, size_t n)
{
    if (nmem == MAXP || used + n > capacity) return fail(cudaErrorMemoryAllocation);
    *p = mem[nmem].p = next_addr;
    mem[nmem++].n = n;
    next_addr += (n + 511) / 256 * 256;
    used += n;
    if (used > peak) peak = used;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    for (int i = 0; i < nmem; ++i)
        if (mem[i].p == p) { used -= mem[i].n; mem[i] = mem[--nmem]; return cudaSuccess; }
    return p ? fail(cudaErrorInvalidValue) : cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t st)
{ (void)s; (void)st; if (k == cudaMemcpyDeviceToHost) memset(d, 0, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, enum cudaMemcpyKind k) { return cudaMemcpyAsync(d, s, n, k, 0); }
cudaError_t cudaMemset(void *p, int v, size_t n) { (void)p; (void)v; (void)n; return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t s) { (void)p; (void)v; (void)n; (void)s; return cudaSuccess; }

cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = 0; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned f) { (void)f; *e = 0; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b) { (void)a; (void)b; *ms = 1; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { (void)e; (void)s; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned f) { (void)f; *s = 0; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { (void)s; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) { (void)s; (void)e; (void)f; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, enum cudaStreamCaptureStatus *c) { (void)s; *c = cudaStreamCaptureStatusNone; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m) { (void)s; (void)m; return fail(cudaErrorNotSupported); }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g) { (void)s; *g = 0; return fail(cudaErrorNotSupported); }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { (void)g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t g) { (void)g; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t g, unsigned long long f) { (void)g; (void)f; *e = 0; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s) { (void)e; (void)s; return cudaSuccess; }
int cufftDestroy(int p) { (void)p; return 1; }
int cufftExecC2C(int p, void *a, void *b, int d) { (void)p; (void)a; (void)b; (void)d; return 1; }
int cufftExecZ2Z(int p, void *a, void *b, int d) { (void)p; (void)a; (void)b; (void)d; return 1; }
int cufftPlanMany(int *p) { (void)p; return 1; }
int cufftSetStream(int p, void *s) { (void)p; (void)s; return 1; }
