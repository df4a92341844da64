/* A CUDA runtime that launches nothing, for tests of the library's host side
 * without a GPU: it keeps what a device would check at a launch (each
 * function's shared-memory limit and cluster attribute per device, the block
 * size) and records the launches.  Linked with the library's objects in the
 * place of the CUDA runtime. */
#include <cuda_runtime_api.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#define MAXF 1024
#define MAXL 65536
#define DEVS 4

typedef struct {
    const void *fn;
    char name[256];
    int smem[DEVS], wide[DEVS]; /* 0: never set */
} Func;
typedef struct {
    int f, grid[3], block, smem, cluster;
} Launch;

static Func funcs[MAXF];
static Launch launches[MAXL];
static int nfuncs, nlaunch, device, lowered;
static struct { struct dim3 g, b; size_t s; cudaStream_t st; } pushed;
static const int kOptin = 227 * 1024;

void fake_device(int d) { device = d; }
void fake_reset(void) { nlaunch = lowered = 0; }
int fake_launches(void) { return nlaunch; }
int fake_lowered(void) { return lowered; } /* times a function's limit was set below an earlier one */
const char *fake_launch(int i, int out[6])
{
    const Launch *l = &launches[i];
    out[0] = l->grid[0]; out[1] = l->grid[1]; out[2] = l->grid[2];
    out[3] = l->block; out[4] = l->smem; out[5] = l->cluster;
    return funcs[l->f].name;
}

static Func *find(const void *fn)
{
    for (int i = 0; i < nfuncs; ++i)
        if (funcs[i].fn == fn) return &funcs[i];
    return NULL;
}
static cudaError_t launch(const void *fn, struct dim3 g, struct dim3 b, size_t smem, int cluster)
{
    Func *f = find(fn);
    if (!f) return cudaErrorInvalidDeviceFunction;
    const long long th = (long long)b.x * b.y * b.z;
    const int limit = f->smem[device] ? f->smem[device] : 48 * 1024;
    if (!g.x || !g.y || !g.z || g.y > 65535 || g.z > 65535 || !th || th > 1024) return cudaErrorInvalidConfiguration;
    if ((long long)smem > limit || (cluster > 8 && !f->wide[device])) return cudaErrorInvalidValue;
    if (nlaunch == MAXL) return cudaErrorUnknown;
    Launch *l = &launches[nlaunch++];
    l->f = (int)(f - funcs);
    l->grid[0] = (int)g.x; l->grid[1] = (int)g.y; l->grid[2] = (int)g.z;
    l->block = (int)th; l->smem = (int)smem; l->cluster = cluster;
    return cudaSuccess;
}

/* registration and launch of compiled code */
static void *fat;
void **__cudaRegisterFatBinary(void *p) { (void)p; return &fat; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void **h, const char *host, char *dev, const char *name, int lim, void *a, void *b, void *c, void *d, int *w)
{
    (void)h; (void)dev; (void)lim; (void)a; (void)b; (void)c; (void)d; (void)w;
    if (nfuncs == MAXF) abort();
    funcs[nfuncs].fn = host;
    snprintf(funcs[nfuncs++].name, sizeof funcs[0].name, "%s", name);
}
void __cudaRegisterVar(void **h, char *host, char *dev, const char *name, int ext, size_t size, int c, int g)
{
    (void)h; (void)host; (void)dev; (void)name; (void)ext; (void)size; (void)c; (void)g;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fn) { *k = (cudaKernel_t)fn; return cudaSuccess; }
unsigned __cudaPushCallConfiguration(struct dim3 g, struct dim3 b, size_t s, cudaStream_t st)
{
    pushed.g = g; pushed.b = b; pushed.s = s; pushed.st = st;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(struct dim3 *g, struct dim3 *b, size_t *s, void *st)
{
    *g = pushed.g; *b = pushed.b; *s = pushed.s; *(cudaStream_t *)st = pushed.st;
    return cudaSuccess;
}
static cudaError_t last;
static cudaError_t keep(cudaError_t e) { if (e) last = e; return e; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, struct dim3 g, struct dim3 b, void **a, size_t s, cudaStream_t st)
{
    (void)a; (void)st;
    return keep(launch((const void *)k, g, b, s, 1));
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fn, void **a)
{
    (void)a;
    int cluster = 1;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = (int)c->attrs[i].val.clusterDim.x;
    return keep(launch(fn, c->gridDim, c->blockDim, c->dynamicSmemBytes, cluster));
}
cudaError_t cudaFuncSetAttribute(const void *fn, enum cudaFuncAttribute at, int v)
{
    Func *f = find(fn);
    if (!f) return keep(cudaErrorInvalidDeviceFunction);
    if (at == cudaFuncAttributeMaxDynamicSharedMemorySize) {
        if (v > kOptin) return keep(cudaErrorInvalidValue);
        if (v < f->smem[device]) ++lowered;
        f->smem[device] = v;
    } else if (at == cudaFuncAttributeNonPortableClusterSizeAllowed) {
        f->wide[device] = v;
    }
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *fn, const cudaLaunchConfig_t *c)
{
    const int cs = (int)c->attrs[0].val.clusterDim.x;
    Func *f = find(fn);
    const int limit = f->smem[device] ? f->smem[device] : 48 * 1024;
    if ((long long)c->dynamicSmemBytes > limit || (cs > 8 && !f->wide[device])) return keep(cudaErrorInvalidValue);
    *n = cs == 16 ? 7 : 152 / cs; /* of 16 CTAs seven fit a GB300 at one CTA per SM */
    return cudaSuccess;
}

/* everything else succeeds */
#define OK(name, ...) cudaError_t name(__VA_ARGS__) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { cudaError_t e = last; last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t e) { (void)e; return "fake"; }
cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d) { (void)a; (void)d; *v = 152; return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { (void)n; *p = (void *)(uintptr_t)(1ull << 40); return cudaSuccess; }
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t s) { (void)s; return cudaMalloc(p, n); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned f) { (void)f; *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *s) { (void)s; return cudaMalloc(p, 0); }
static int encode(void) { return 0; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *s, void **p, unsigned v, unsigned long long f, enum cudaDriverEntryPointQueryResult *r)
{
    (void)s; (void)v; (void)f;
    *p = (void *)encode;
    if (r) *r = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned f) { (void)f; return cudaEventCreate(e); }
cudaError_t cudaEventElapsedTime(float *t, cudaEvent_t a, cudaEvent_t b) { (void)a; (void)b; *t = 1.f; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned f) { (void)f; *s = (cudaStream_t)1; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g) { (void)s; *g = (cudaGraph_t)1; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t g, unsigned long long f) { (void)g; (void)f; *e = (cudaGraphExec_t)1; return cudaSuccess; }
OK(cudaEventDestroy, cudaEvent_t e)
OK(cudaEventRecord, cudaEvent_t e, cudaStream_t s)
OK(cudaEventRecordWithFlags, cudaEvent_t e, cudaStream_t s, unsigned f)
OK(cudaEventSynchronize, cudaEvent_t e)
OK(cudaFree, void *p)
OK(cudaFreeAsync, void *p, cudaStream_t s)
OK(cudaGraphDestroy, cudaGraph_t g)
OK(cudaGraphExecDestroy, cudaGraphExec_t e)
OK(cudaGraphLaunch, cudaGraphExec_t e, cudaStream_t s)
OK(cudaMemcpy, void *d, const void *s, size_t n, enum cudaMemcpyKind k)
OK(cudaMemcpyAsync, void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t st)
OK(cudaMemsetAsync, void *d, int v, size_t n, cudaStream_t s)
OK(cudaStreamBeginCapture, cudaStream_t s, enum cudaStreamCaptureMode m)
OK(cudaStreamDestroy, cudaStream_t s)
OK(cudaStreamSynchronize, cudaStream_t s)
OK(cudaStreamWaitEvent, cudaStream_t s, cudaEvent_t e, unsigned f)
