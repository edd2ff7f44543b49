// IF nodes of captured steps: work that a device flag may skip (the FP64 route, Krylov iterations past
// convergence) becomes the body of a conditional node, so that a skipped part costs one node instead
// of one early-exiting launch per kernel.  Compiled as relocatable device code: the device side of
// conditional nodes is in the CUDA device runtime.
#include <cuda_runtime.h>

#include "xk_internal.cuh"

namespace xk {

namespace {

__global__ void k_set_if(cudaGraphConditionalHandle h, const int *flag, int when)
{
    cudaGraphSetConditional(h, ((*flag != 0) == (when != 0)) ? 1u : 0u);
}

}  // namespace

bool capturing(cudaStream_t st)
{
    cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(st, &s) == cudaSuccess && s == cudaStreamCaptureStatusActive;
}

cudaError_t cond_open(cudaStream_t st, cudaStream_t inner, const int *flag, int when, cudaGraphNode_t *node)
{
    cudaStreamCaptureStatus s;
    unsigned long long id;
    cudaGraph_t graph;
    const cudaGraphNode_t *deps;
    const cudaGraphEdgeData *edges;
    size_t n = 0;
    cudaError_t e = cudaStreamGetCaptureInfo(st, &s, &id, &graph, &deps, &edges, &n);
    if (e != cudaSuccess) return e;
    cudaGraphConditionalHandle h;
    e = cudaGraphConditionalHandleCreate(&h, graph, 0, cudaGraphCondAssignDefault);
    if (e != cudaSuccess) return e;
    count_launches(1);
    k_set_if<<<1, 1, 0, st>>>(h, flag, when);
    e = cudaStreamGetCaptureInfo(st, &s, &id, &graph, &deps, &edges, &n);
    if (e != cudaSuccess) return e;
    cudaGraphNodeParams p = {};
    p.type = cudaGraphNodeTypeConditional;
    p.conditional.handle = h;
    p.conditional.type = cudaGraphCondTypeIf;
    p.conditional.size = 1;
    e = cudaGraphAddNode(node, graph, deps, edges, n, &p);
    if (e != cudaSuccess) return e;
    return cudaStreamBeginCaptureToGraph(inner, p.conditional.phGraph_out[0], nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed);
}

cudaError_t cond_close(cudaStream_t st, cudaStream_t inner, cudaGraphNode_t node)
{
    cudaGraph_t body;
    cudaError_t e = cudaStreamEndCapture(inner, &body);
    if (e != cudaSuccess) return e;
    return cudaStreamUpdateCaptureDependencies(st, &node, nullptr, 1, cudaStreamSetCaptureDependencies);
}

}  // namespace xk
