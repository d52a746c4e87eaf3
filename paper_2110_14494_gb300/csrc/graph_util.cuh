// Helpers for recording device-driven loops into CUDA graphs (conditional
// nodes added at the capture point of a stream), and for launches that overlap
// the end of the kernel before them.
#pragma once
#include <cuda_runtime.h>

namespace pic {

// Kernels of the solvers' cycles are launched with programmatic dependent
// launch: their blocks may be scheduled while the previous kernel's last
// blocks still run, and each waits here for that grid (and its memory) before
// its first access.  Without the launch attribute the wait returns at once.
__device__ __forceinline__ void pdl_wait() { cudaGridDependencySynchronize(); }

// A launch's error is its return value: a later call that succeeds can reset
// the last error, so callers keep what this returns.
template <class... P, class... A>
cudaError_t launch_pdl(void (*k)(P...), dim3 g, dim3 b, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = g;
    cfg.blockDim = b;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

// First error of a sequence of launches; launched() reports and clears it.  A
// solve clears it at its start: one that gave up earlier may have left one.
struct LaunchStatus {
    cudaError_t launch_err = cudaSuccess;
    void note(cudaError_t e) {
        if (launch_err == cudaSuccess) launch_err = e;
    }
    bool launched() {
        const bool ok = launch_err == cudaSuccess;
        if (!ok) cudaGetLastError();
        launch_err = cudaSuccess;
        return ok;
    }
};

__device__ __forceinline__ void bar_named(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Adds a conditional node with handle h at the capture point of stream cs
// (which must be capturing) and makes it the stream's only dependency;
// bodies receives its body graphs (owned by the node).
inline cudaError_t add_conditional(cudaStream_t cs, cudaGraphConditionalHandle h, cudaGraphConditionalNodeType type,
                                   unsigned size, cudaGraph_t* bodies) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    cudaGraph_t g = nullptr;
    const cudaGraphNode_t* deps = nullptr;
    const cudaGraphEdgeData* ed = nullptr;
    size_t nd = 0;
    cudaError_t e = cudaStreamGetCaptureInfo(cs, &st, nullptr, &g, &deps, &ed, &nd);
    if (e != cudaSuccess) return e;
    if (st != cudaStreamCaptureStatusActive) return cudaErrorStreamCaptureInvalidated;
    cudaGraphNodeParams p = {};
    p.type = cudaGraphNodeTypeConditional;
    p.conditional.handle = h;
    p.conditional.type = type;
    p.conditional.size = size;
    cudaGraphNode_t node = nullptr;
    e = cudaGraphAddNode(&node, g, deps, ed, nd, &p);
    if (e != cudaSuccess) return e;
    for (unsigned q = 0; q < size; ++q) bodies[q] = p.conditional.phGraph_out[q];
    return cudaStreamUpdateCaptureDependencies(cs, &node, nullptr, 1, cudaStreamSetCaptureDependencies);
}

// Ends a capture into a body graph (the graph stays owned by its node).
inline cudaError_t end_body_capture(cudaStream_t s) {
    cudaGraph_t g = nullptr;
    return cudaStreamEndCapture(s, &g);
}

// The graph a capturing stream records into (null if it is not capturing).
inline cudaGraph_t capturing_graph(cudaStream_t cs) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    cudaGraph_t g = nullptr;
    if (cudaStreamGetCaptureInfo(cs, &st, nullptr, &g) != cudaSuccess || st != cudaStreamCaptureStatusActive)
        return nullptr;
    return g;
}

}  // namespace pic
