// A stand-in for the CUDA runtime that runs no kernel, for tests of the
// library's host code without a GPU.  Two devices; device memory is host
// memory; a launch is checked against what was set for its kernel on the
// current device and logged.
#include <cuda_runtime.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

namespace {

int g_device = 0, g_max_cluster = 16, g_max_coop = 1 << 30;
std::map<const void *, std::string> g_names;
std::map<std::pair<int, const void *>, std::map<int, int>> g_attr;
std::map<uintptr_t, std::pair<size_t, int>> g_mem;
std::string g_log;
float g_clock = 0.f;
struct { dim3 grid, block; size_t smem; cudaStream_t stream; } g_cfg;

int attr(const void *f, cudaFuncAttribute a) {
    auto it = g_attr.find({g_device, f});
    return it == g_attr.end() || !it->second.count(a) ? 0 : it->second[a];
}

cudaError_t fits(const void *f, size_t smem, unsigned cluster) {
    if (smem > 48 * 1024 && (size_t)attr(f, cudaFuncAttributeMaxDynamicSharedMemorySize) < smem) return cudaErrorInvalidValue;
    if (cluster > 8 && !attr(f, cudaFuncAttributeNonPortableClusterSizeAllowed)) return cudaErrorInvalidClusterSize;
    return cudaSuccess;
}

cudaError_t launch(const void *f, dim3 grid, size_t smem, unsigned cluster, bool coop) {
    if (cudaError_t e = fits(f, smem, cluster)) return e;
    if (cluster > (unsigned)g_max_cluster) return cudaErrorLaunchOutOfResources;
    if (coop && grid.x > (unsigned)g_max_coop) return cudaErrorCooperativeLaunchTooLarge;
    g_log += std::to_string(g_device) + " " + g_names[f] + " " + std::to_string(grid.x) + " " + std::to_string(cluster) + "\n";
    return cudaSuccess;
}

}  // namespace

extern "C" {

void fake_limits(int max_cluster, int max_coop) {
    g_max_cluster = max_cluster;
    g_max_coop = max_coop;
}
const char *fake_log() { return g_log.c_str(); }
void fake_clear() { g_log.clear(); }

void **__cudaRegisterFatBinary(void *) {
    static void *handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {
    g_names[host] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
    g_cfg = {grid, block, smem, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *s) {
    *grid = g_cfg.grid;
    *block = g_cfg.block;
    *smem = g_cfg.smem;
    *static_cast<cudaStream_t *>(s) = g_cfg.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void **, size_t smem, cudaStream_t) {
    return launch((const void *)k, grid, smem, 1, false);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
    unsigned cluster = 1;
    bool coop = false;
    for (unsigned k = 0; k < c->numAttrs; ++k) {
        if (c->attrs[k].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[k].val.clusterDim.x;
        if (c->attrs[k].id == cudaLaunchAttributeCooperative) coop = c->attrs[k].val.cooperative != 0;
    }
    return launch(f, c->gridDim, c->dynamicSmemBytes, cluster, coop);
}

cudaError_t cudaGetDeviceCount(int *n) { *n = 2; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_device = d; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake runtime error"; }
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) {
    g_attr[{g_device, f}][a] = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    *n = 4;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *c) {
    *n = 0;
    const unsigned cluster = c->numAttrs ? c->attrs[0].val.clusterDim.x : 1;
    if (cudaError_t e = fits(f, c->dynamicSmemBytes, cluster)) return e;
    *n = cluster <= (unsigned)g_max_cluster ? 1 : 0;
    return cudaSuccess;
}

cudaError_t cudaMalloc(void **p, size_t n) {
    *p = calloc(1, (n + 511) & ~size_t(255));
    *p = (void *)(((uintptr_t)*p + 255) & ~uintptr_t(255));   // never given back: a test is one short process
    g_mem[(uintptr_t)*p] = {n, g_device};
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    g_mem.erase((uintptr_t)p);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void **p, size_t n) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
    memset(a, 0, sizeof(*a));
    auto it = g_mem.upper_bound((uintptr_t)p);
    if (it != g_mem.begin() && (--it, (uintptr_t)p < it->first + it->second.first)) {
        a->type = cudaMemoryTypeDevice;
        a->device = it->second.second;
    }
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) { return cudaMalloc(p, 8 << 20); }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
    memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) {
    memset(d, v, n);
    return cudaSuccess;
}

cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)8; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { *g = (cudaGraph_t)8; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) { *e = (cudaGraphExec_t)8; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) {
    g_log += std::to_string(g_device) + " graph 1 1\n";
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)8; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = g_clock += 1.f; return cudaSuccess; }

}  // extern "C"
