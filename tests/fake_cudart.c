/* A CUDA runtime of two devices that runs nothing: the library's host code linked against it
 * shows which kernel it would launch, how, and on which device.  A launch that asks for more
 * dynamic shared memory than its kernel was granted on the current device is refused, as the real
 * runtime does. */
#include <cuda_runtime_api.h>
#include <string.h>

enum { kDevices = 2, kFunctions = 4096, kSms = 152, kSmemOptin = 232448, kSmemDefault = 48 * 1024 };

static struct {
    const void *host;
    const char *name;
    size_t granted[kDevices];
} g_fn[kFunctions];
static int g_functions, g_device, g_launches;
static struct {
    int fn, grid[3], block, cluster;
    size_t smem;
} g_last;

static int find(const void *host) {
    for (int i = 0; i < g_functions; ++i)
        if (g_fn[i].host == host) return i;
    return -1;
}

void fake_set_device(int d) { g_device = d; }
int fake_launches(void) { return g_launches; }
const char *fake_last_kernel(void) { return g_launches ? g_fn[g_last.fn].name : ""; }
/* grid x, y, z, threads, cluster size (0: none), dynamic shared memory of the last launch */
void fake_last_shape(long long out[6]) {
    for (int i = 0; i < 3; ++i) out[i] = g_last.grid[i];
    out[3] = g_last.block;
    out[4] = g_last.cluster;
    out[5] = (long long)g_last.smem;
}

cudaError_t cudaGetDevice(int *d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d) {
    *v = a == cudaDevAttrMultiProcessorCount ? kSms
         : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? kSmemOptin : 0;
    return d < kDevices ? cudaSuccess : cudaErrorInvalidDevice;
}
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v) {
    const int i = find(f);
    if (i < 0) return cudaErrorInvalidDeviceFunction;
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_fn[i].granted[g_device] = (size_t)v;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args) {
    (void)args;
    const int i = find(f);
    if (i < 0) return cudaErrorInvalidDeviceFunction;
    const size_t have = g_fn[i].granted[g_device] > kSmemDefault ? g_fn[i].granted[g_device]
                                                                 : kSmemDefault;
    if (c->dynamicSmemBytes > have) return cudaErrorInvalidValue;
    g_last.fn = i;
    g_last.grid[0] = (int)c->gridDim.x;
    g_last.grid[1] = (int)c->gridDim.y;
    g_last.grid[2] = (int)c->gridDim.z;
    g_last.block = (int)c->blockDim.x;
    g_last.cluster = 0;
    g_last.smem = c->dynamicSmemBytes;
    for (unsigned k = 0; k < c->numAttrs; ++k)
        if (c->attrs[k].id == cudaLaunchAttributeClusterDimension) {
            const cudaLaunchAttributeValue *v = &c->attrs[k].val;
            g_last.cluster = (int)(v->clusterDim.x * v->clusterDim.y * v->clusterDim.z);
        }
    ++g_launches;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *c) {
    (void)f, (void)c;
    *n = 8;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *f, int b, size_t s) {
    (void)f, (void)b, (void)s;
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k,
                            cudaStream_t t) {
    (void)d, (void)s, (void)n, (void)k, (void)t;
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t t) {
    (void)d, (void)v, (void)n, (void)t;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *s) {
    (void)p, (void)s;
    return cudaErrorInvalidSymbol;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *s, void **p, unsigned v,
                                             unsigned long long f,
                                             enum cudaDriverEntryPointQueryResult *q) {
    (void)s, (void)p, (void)v, (void)f, (void)q;
    return cudaErrorInvalidValue;
}

/* registration of the objects' kernels, and the triple-chevron launches (not used by the tests) */
void **__cudaRegisterFatBinary(void *f) { static void *h; (void)f; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void **h, const char *host, char *dev, const char *name, int t,
                            void *a, void *b, void *c, void *d, int *w) {
    (void)h, (void)dev, (void)t, (void)a, (void)b, (void)c, (void)d, (void)w;
    if (g_functions < kFunctions) {
        g_fn[g_functions].host = host;
        g_fn[g_functions++].name = name;
    }
}
void __cudaRegisterVar(void **h, char *host, char *dev, const char *name, int e, size_t s, int c,
                       int g) {
    (void)h, (void)host, (void)dev, (void)name, (void)e, (void)s, (void)c, (void)g;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, void *t) {
    (void)g, (void)b, (void)s, (void)t;
    return 1;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *s, void *t) {
    (void)g, (void)b, (void)s, (void)t;
    return cudaErrorNotSupported;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
    (void)k, (void)f;
    return cudaErrorNotSupported;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void **a, size_t s,
                               cudaStream_t t) {
    (void)k, (void)g, (void)b, (void)a, (void)s, (void)t;
    return cudaErrorNotSupported;
}
