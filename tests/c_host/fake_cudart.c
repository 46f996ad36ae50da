/* A stand-in for the CUDA runtime, for tests of the library's host code without a GPU: linked with
 * the library's objects in place of cudart. Kernels do not run; every launch is recorded by name,
 * and the calls whose failures the host code must survive can be made to fail. */
#include <string.h>

#include <cuda_runtime_api.h>

/* STATIC: what every kernel is taken to declare, the most that one in the library does */
enum { MAX_KERNELS = 4096, MAX_LAUNCHES = 64, OPTIN = 227 * 1024, STATIC = 1024 };

static struct { const void *fn; const char *name; int smem[2]; } kernels[MAX_KERNELS];
static int n_kernels, context, fail_queries, fail_opt_ins, launches;
static const char *launched[MAX_LAUNCHES];

/* ------------------------------------------------------------ for the tests */
void fake_use_context(int c) { context = c; }
void fake_device_reset(void) {
    for (int i = 0; i < n_kernels; ++i) kernels[i].smem[context] = 0;
}
void fake_fail_queries(int n) { fail_queries = n; }
void fake_fail_opt_ins(int n) { fail_opt_ins = n; }
int fake_launches(void) { return launches; }
const char *fake_launched(int i) { return launched[i % MAX_LAUNCHES]; }

static int find(const void *fn) {
    for (int i = 0; i < n_kernels; ++i)
        if (kernels[i].fn == fn) return i;
    return -1;
}
static int allowed(int k, size_t bytes) {
    const int most = kernels[k].smem[context];
    return bytes <= (size_t)most || bytes + STATIC <= 48 * 1024;
}

/* ------------------------------------------------------------ the runtime */
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? OPTIN : 0;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(struct cudaFuncAttributes *a, const void *fn) {
    memset(a, 0, sizeof *a);
    a->sharedSizeBytes = STATIC;
    return find(fn) < 0 ? cudaErrorInvalidDeviceFunction : cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *fn, enum cudaFuncAttribute a, int v) {
    const int k = find(fn);
    if (fail_opt_ins > 0) { --fail_opt_ins; return cudaErrorMemoryAllocation; }
    if (k < 0 || a != cudaFuncAttributeMaxDynamicSharedMemorySize || v + STATIC > OPTIN) return cudaErrorInvalidValue;
    kernels[k].smem[context] = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *fn, int threads, size_t bytes) {
    const int k = find(fn);
    if (fail_queries > 0) { --fail_queries; return cudaErrorMemoryAllocation; }
    if (k < 0) return cudaErrorInvalidDeviceFunction;
    *n = allowed(k, bytes) ? (int)(OPTIN / (bytes + 1024)) < 2048 / threads / 4 ? (int)(OPTIN / (bytes + 1024))
                                                                              : 2048 / threads / 4 : 0;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fn, void **args) {
    const int k = find(fn);
    if (k < 0) return cudaErrorInvalidDeviceFunction;
    if (!allowed(k, c->dynamicSmemBytes)) return cudaErrorInvalidValue;
    launched[launches++ % MAX_LAUNCHES] = kernels[k].name;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t e) { return "an error of the stand-in runtime"; }
cudaError_t cudaGetSymbolAddress(void **p, const void *symbol) { *p = (void *)symbol; return cudaSuccess; }

/* ------------------------------------------------------------ what compiled host code registers */
void **__cudaRegisterFatBinary(void *bin) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) {}
void __cudaUnregisterFatBinary(void **h) {}
void __cudaRegisterVar(void **h, char *host, char *dev, const char *name, int ext, size_t n, int cst, int global) {}
void __cudaRegisterFunction(void **h, const char *fn, char *dev, const char *name, int limit, void *tid, void *bid,
                            void *bdim, void *gdim, int *wsize) {
    if (n_kernels < MAX_KERNELS) {
        kernels[n_kernels].fn = fn;
        kernels[n_kernels++].name = name;
    }
}
cudaError_t __cudaGetKernel(void **k, const void *fn) { *k = (void *)fn; return cudaSuccess; }
unsigned __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) { return 1; }
cudaError_t __cudaLaunchKernel(void *k, dim3 g, dim3 b, void **args, size_t smem, void *s) { return cudaErrorInvalidValue; }
