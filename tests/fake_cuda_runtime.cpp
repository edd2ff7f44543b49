// A CUDA runtime of two devices without a GPU, for what the library asks of the runtime: device memory
// is host memory, copies copy, kernels do nothing.  A launch is refused as the real one refuses it: with
// more than 48 KB of dynamic shared memory where the kernel's limit has not been raised on the current
// device (cudaFuncSetAttribute holds for one device), or cooperatively on more CTAs than the device has
// SMs.  Conditional nodes are refused while the devices are shared through MPS (fake_set_mps).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <utility>
#include <vector>

#define API extern "C" __attribute__((visibility("default")))
#define FAKE extern "C"

namespace {
constexpr int kDevices = 2, kSms[kDevices] = {152, 100};
int g_dev = 0, g_mps = 0, g_cond = 0, g_launches[kDevices] = {};
std::map<std::pair<int, const void *>, size_t> g_limit;
std::map<const void *, std::string> g_name;
std::string g_refused;
struct Launch {
    std::string name;
    int grid, cluster;
};
std::vector<Launch> g_log;
std::set<cudaStream_t> g_capturing;
std::set<cudaEvent_t> g_forked;
cudaError_t g_last = cudaSuccess;
struct Pending {
    dim3 grid, block;
    size_t smem;
    cudaStream_t st;
} g_pending;
char *handle()
{
    static char *next = (char *)0x1000;
    return next += 16;
}
cudaError_t keep(cudaError_t e)
{
    if (e != cudaSuccess) g_last = e;
    return e;
}
cudaError_t launch(const void *fn, dim3 grid, size_t smem, bool cooperative, int cluster = 1)
{
    const auto it = g_limit.find({g_dev, fn});
    const size_t limit = it == g_limit.end() ? 48 * 1024 : std::max<size_t>(it->second, 48 * 1024);
    if (smem > limit || (cooperative && (int)grid.x > kSms[g_dev])) {
        if (g_refused.empty()) g_refused = g_name[fn];
        return keep(cudaErrorInvalidValue);
    }
    ++g_launches[g_dev];
    g_log.push_back({g_name[fn], (int)grid.x, cluster});
    return cudaSuccess;
}
}  // namespace

API void fake_set_mps(int on) { g_mps = on; }
API int fake_conditional_nodes() { return g_cond; }
API int fake_launches(int dev) { return g_launches[dev]; }
API const char *fake_refused() { return g_refused.c_str(); }
// launches since fake_forget_launches of kernels whose (mangled) name holds `name`: their number, and the grid
// and cluster of the first
API int fake_launches_of(const char *name, int *grid, int *cluster)
{
    int n = 0;
    for (const Launch &l : g_log)
        if (l.name.find(name) != std::string::npos && n++ == 0) {
            *grid = l.grid;
            *cluster = l.cluster;
        }
    return n;
}
API void fake_forget_launches() { g_log.clear(); }

FAKE cudaError_t cudaGetDeviceCount(int *n) { *n = kDevices; return cudaSuccess; }
FAKE cudaError_t cudaGetDevice(int *d) { *d = g_dev; return cudaSuccess; }
FAKE cudaError_t cudaSetDevice(int d) { if (d < 0 || d >= kDevices) return keep(cudaErrorInvalidDevice); g_dev = d; return cudaSuccess; }
FAKE cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int d)
{
    *v = a == cudaDevAttrMultiProcessorCount ? kSms[d] : a == cudaDevAttrMpsEnabled ? g_mps : 0;
    return cudaSuccess;
}
FAKE cudaError_t cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
FAKE const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "refused by the fake runtime"; }
FAKE cudaError_t cudaMallocHost(void **p, size_t n) { *p = calloc(1, n); return cudaSuccess; }
FAKE cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
FAKE cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { memmove(d, s, n); return cudaSuccess; }
FAKE cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t)
{
    for (size_t i = 0; i < h; ++i) memmove((char *)d + i * dp, (const char *)s + i * sp, w);
    return cudaSuccess;
}
FAKE cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
FAKE cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *) { memset(a, 0, sizeof *a); a->type = cudaMemoryTypeDevice; a->device = g_dev; return cudaSuccess; }
FAKE cudaError_t cudaGetSymbolAddress(void **p, const void *) { *p = calloc(1, 1 << 16); return cudaSuccess; }
FAKE cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)handle(); return cudaSuccess; }
FAKE cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
FAKE cudaError_t cudaStreamSynchronize(cudaStream_t s) { return g_capturing.count(s) ? keep(cudaErrorStreamCaptureUnsupported) : cudaSuccess; }
FAKE cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)handle(); return cudaSuccess; }
FAKE cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
FAKE cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
FAKE cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
FAKE cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
FAKE cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { if (g_capturing.count(s)) g_forked.insert(e); else g_forked.erase(e); return cudaSuccess; }
FAKE cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { if (g_forked.count(e)) g_capturing.insert(s); return cudaSuccess; }

// capture: the graphs are not kept
FAKE cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus *st)
{
    *st = g_capturing.count(s) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
FAKE cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) { g_capturing.insert(s); return cudaSuccess; }
FAKE cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t s, cudaGraph_t, const cudaGraphNode_t *, const cudaGraphEdgeData *, size_t, cudaStreamCaptureMode)
{
    g_capturing.insert(s);
    return cudaSuccess;
}
FAKE cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g)
{
    // streams that joined through an event leave with the one that began
    if (!g_forked.empty()) {
        g_forked.clear();
        g_capturing.clear();
    }
    g_capturing.erase(s);
    *g = (cudaGraph_t)handle();
    return cudaSuccess;
}
FAKE cudaError_t cudaStreamGetCaptureInfo(cudaStream_t s, cudaStreamCaptureStatus *st, unsigned long long *id, cudaGraph_t *g, const cudaGraphNode_t **deps, const cudaGraphEdgeData **edges, size_t *n)
{
    cudaStreamIsCapturing(s, st);
    *id = 1; *g = (cudaGraph_t)0x10; *deps = nullptr; *edges = nullptr; *n = 0;
    return cudaSuccess;
}
FAKE cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle *h, cudaGraph_t, unsigned, unsigned)
{
    if (g_mps) return keep(cudaErrorNotSupported);
    ++g_cond;
    *h = 1;
    return cudaSuccess;
}
FAKE cudaError_t cudaGraphAddNode(cudaGraphNode_t *node, cudaGraph_t, const cudaGraphNode_t *, const cudaGraphEdgeData *, size_t, cudaGraphNodeParams *p)
{
    static cudaGraph_t body = (cudaGraph_t)0x20;
    *node = (cudaGraphNode_t)handle();
    p->conditional.phGraph_out = &body;
    return cudaSuccess;
}
FAKE cudaError_t cudaStreamUpdateCaptureDependencies(cudaStream_t, cudaGraphNode_t *, const cudaGraphEdgeData *, size_t, unsigned) { return cudaSuccess; }
FAKE cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { *x = (cudaGraphExec_t)handle(); return cudaSuccess; }
FAKE cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
FAKE cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
FAKE cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

// kernels
FAKE cudaError_t cudaFuncSetAttribute(const void *fn, cudaFuncAttribute a, int v)
{
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_limit[{g_dev, fn}] = (size_t)v;
    return cudaSuccess;
}
FAKE cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *c)
{
    int cs = 1;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cs = c->attrs[i].val.clusterDim.x;
    *n = kSms[g_dev] / cs;
    return cudaSuccess;
}
FAKE cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fn, void **)
{
    bool coop = false;
    int cluster = 1;
    for (unsigned i = 0; i < c->numAttrs; ++i) {
        coop |= c->attrs[i].id == cudaLaunchAttributeCooperative && c->attrs[i].val.cooperative;
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[i].val.clusterDim.x;
    }
    return launch(fn, c->gridDim, c->dynamicSmemBytes, coop, cluster);
}
FAKE cudaError_t cudaLaunchCooperativeKernel(const void *fn, dim3 grid, dim3, void **, size_t smem, cudaStream_t) { return launch(fn, grid, smem, true); }
FAKE unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st *st) { g_pending = {grid, block, smem, st}; return 0; }
FAKE cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *st)
{
    *grid = g_pending.grid; *block = g_pending.block; *smem = g_pending.smem; *(cudaStream_t *)st = g_pending.st;
    return cudaSuccess;
}
FAKE cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fn) { *k = (cudaKernel_t)fn; return cudaSuccess; }
FAKE cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void **, size_t smem, cudaStream_t) { return launch((const void *)k, grid, smem, false); }

// registration at load time
FAKE void **__cudaRegisterFatBinary(void *p) { return (void **)p; }
FAKE void __cudaRegisterFatBinaryEnd(void **) {}
FAKE void __cudaUnregisterFatBinary(void **) {}
FAKE void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
FAKE void __cudaRegisterFunction(void **, const char *fn, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) { g_name[fn] = name; }
FAKE void fake_linked_binary(void (*)(void **), void *, void *, void (*)(void *)) {}   // of relocatable device code

// the tensor maps' encoder
static int encode_nothing(...) { return 0; }
FAKE cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **fn, unsigned, unsigned long long, cudaDriverEntryPointQueryResult *q)
{
    *fn = (void *)encode_nothing;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
