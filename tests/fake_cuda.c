/* A CUDA runtime of several devices that runs nothing, for the library's host
 * code: device memory is host memory, copies copy, and a launch is refused, as
 * the real runtime refuses it, when it wants more dynamic shared memory than
 * the kernel has been allowed on the current device.  Linked with the
 * library's own objects in place of the runtime. */
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>

#define API __attribute__((visibility("default")))

static int device, launches, refused, copies;
static cudaError_t last;
static struct { const void *f; int dev, bytes; } allowed[1024];
static int n_allowed;

API void fake_set_device(int d) { device = d; }
API int fake_launches(void) { return launches; }
API int fake_refused(void) { return refused; }
API int fake_copies(void) { return copies; }

/* The one range of pinned host memory, for the pointer query. */
static CUdeviceptr pinned;
static size_t pinned_bytes;
API void fake_pin(void *p, size_t n) { pinned = (CUdeviceptr)p; pinned_bytes = n; }
static CUresult query(unsigned n, CUpointer_attribute *what, void **to, CUdeviceptr p)
{
    if (p < pinned || p >= pinned + pinned_bytes) return CUDA_ERROR_INVALID_VALUE;
    for (unsigned i = 0; i < n; ++i) switch (what[i]) {
        case CU_POINTER_ATTRIBUTE_MEMORY_TYPE: *(unsigned *)to[i] = CU_MEMORYTYPE_HOST; break;
        case CU_POINTER_ATTRIBUTE_DEVICE_ORDINAL: *(int *)to[i] = 0; break;
        case CU_POINTER_ATTRIBUTE_DEVICE_POINTER: *(CUdeviceptr *)to[i] = p; break;
        case CU_POINTER_ATTRIBUTE_RANGE_START_ADDR: *(CUdeviceptr *)to[i] = pinned; break;
        case CU_POINTER_ATTRIBUTE_RANGE_SIZE: *(size_t *)to[i] = pinned_bytes; break;
        default: return CUDA_ERROR_INVALID_VALUE;
    }
    return CUDA_SUCCESS;
}

static cudaError_t err(cudaError_t e) { if (e) last = e; return e; }

static cudaError_t launch(const void *f, size_t smem)
{
    size_t limit = 48 * 1024;
    for (int i = 0; i < n_allowed; ++i)
        if (allowed[i].f == f && allowed[i].dev == device) limit = (size_t)allowed[i].bytes;
    ++launches;
    if (smem <= limit) return cudaSuccess;
    ++refused;
    return err(cudaErrorInvalidValue);
}

cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v)
{
    if (a != cudaFuncAttributeMaxDynamicSharedMemorySize || v > 227 * 1024 || n_allowed == 1024)
        return err(cudaErrorInvalidValue);
    allowed[n_allowed].f = f;
    allowed[n_allowed].dev = device;
    allowed[n_allowed++].bytes = v;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args)
{
    (void)args;
    return launch(f, c->dynamicSmemBytes);
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, struct dim3 g, struct dim3 b, void **args, size_t smem, cudaStream_t s)
{
    (void)g; (void)b; (void)args; (void)s;
    return launch(k, smem);
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }

static struct dim3 cg, cb;
static size_t csm;
static void *cst;
unsigned __cudaPushCallConfiguration(struct dim3 g, struct dim3 b, size_t smem, struct CUstream_st *s)
{
    cg = g; cb = b; csm = smem; cst = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(struct dim3 *g, struct dim3 *b, size_t *smem, void *s)
{
    *g = cg; *b = cb; *smem = csm; *(void **)s = cst;
    return cudaSuccess;
}
void **__cudaRegisterFatBinary(void *p) { return (void **)p; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void **h, const char *f, char *df, const char *n, int t, void *a, void *b, void *c, void *d,
                            int *w)
{
    (void)h; (void)f; (void)df; (void)n; (void)t; (void)a; (void)b; (void)c; (void)d; (void)w;
}
void __cudaRegisterVar(void **h, char *v, char *a, const char *n, int e, size_t s, int c, int g)
{
    (void)h; (void)v; (void)a; (void)n; (void)e; (void)s; (void)c; (void)g;
}

cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d) { (void)a; (void)d; *v = 152; return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { *p = aligned_alloc(256, (n + 255) / 256 * 256); return cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, enum cudaMemcpyKind k) { (void)k; memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t st)
{
    (void)st;
    return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, enum cudaMemcpyKind k,
                              cudaStream_t st)
{
    (void)k; (void)st;
    ++copies;
    for (size_t y = 0; y < h; ++y) memcpy((char *)d + y * dp, (const char *)s + y * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t s) { (void)s; memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *s) { *p = (void *)s; return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *n, void **f, unsigned v, unsigned long long fl,
                                             enum cudaDriverEntryPointQueryResult *r)
{
    (void)v; (void)fl;
    if (strcmp(n, "cuPointerGetAttributes")) return err(cudaErrorNotSupported);
    *f = (void *)query;
    *r = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *f, int b, size_t s)
{
    (void)f; (void)b; (void)s;
    *n = 2;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int b, size_t s, unsigned fl)
{
    (void)fl;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, f, b, s);
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned f) { (void)f; *e = (cudaEvent_t)malloc(1); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned f) { (void)f; *s = (cudaStream_t)malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m) { (void)s; (void)m; return err(cudaErrorNotSupported); }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g) { (void)s; *g = NULL; return err(cudaErrorNotSupported); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t g, unsigned long long f) { (void)e; (void)g; (void)f; return err(cudaErrorNotSupported); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s) { (void)e; (void)s; return err(cudaErrorNotSupported); }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { (void)g; return cudaSuccess; }

/* The last events recorded (oldest first), for tests of what a call records. */
static cudaEvent_t recorded[64];
static int n_recorded;
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s)
{
    (void)s;
    if (n_recorded < 64) recorded[n_recorded++] = e;
    return cudaSuccess;
}
API int fake_recorded(void **out)
{
    const int n = n_recorded;
    for (int i = 0; i < n; ++i) out[i] = recorded[i];
    n_recorded = 0;
    return n;
}
