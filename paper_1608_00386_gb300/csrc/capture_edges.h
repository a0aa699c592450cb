// Types of the dependencies between captured launches.  A launch with the programmatic stream
// serialization attribute is given a programmatic edge from every kernel that it depends on, those joined
// through events included, and such an edge orders no memory before the launch's griddepcontrol.wait
// (CUDA 13.0).  A launch that reads one kernel's results at once and may overlap another names the one
// that it may overlap here instead, and is launched without the attribute.
#pragma once

#include <cuda_runtime.h>

#include <vector>

namespace mcao {

// the kernel that a capturing stream's next launch depends on, if it is the only node (null otherwise)
inline cudaError_t captured_kernel(cudaStream_t st, cudaGraphNode_t* node) {
    *node = nullptr;
    cudaStreamCaptureStatus status;
    const cudaGraphNode_t* deps = nullptr;
    const cudaGraphEdgeData* data = nullptr;
    size_t n = 0;
    cudaError_t e = cudaStreamGetCaptureInfo(st, &status, nullptr, nullptr, &deps, &data, &n);
    if (e != cudaSuccess || status != cudaStreamCaptureStatusActive || n != 1) return e;
    cudaGraphNodeType type;
    if ((e = cudaGraphNodeGetType(deps[0], &type)) == cudaSuccess && type == cudaGraphNodeTypeKernel) *node = deps[0];
    return e;
}

// The stream's next launch may start once every block of `kernel` has let its dependents go or left; all
// else that it depends on has to be complete.  Nothing changes where it does not depend on `kernel` itself.
inline cudaError_t overlap_captured(cudaStream_t st, cudaGraphNode_t kernel) {
    cudaStreamCaptureStatus status;
    const cudaGraphNode_t* deps = nullptr;
    const cudaGraphEdgeData* data = nullptr;
    size_t n = 0;
    cudaError_t e = cudaStreamGetCaptureInfo(st, &status, nullptr, nullptr, &deps, &data, &n);
    if (e != cudaSuccess || status != cudaStreamCaptureStatusActive || !kernel || n == 0) return e;
    std::vector<cudaGraphNode_t> nodes(deps, deps + n);
    std::vector<cudaGraphEdgeData> edges(n, cudaGraphEdgeData{});
    for (size_t i = 0; i < n; ++i)
        if (nodes[i] == kernel) {
            edges[i].from_port = cudaGraphKernelNodePortProgrammatic;
            edges[i].type = cudaGraphDependencyTypeProgrammatic;
        }
    return cudaStreamUpdateCaptureDependencies(st, nodes.data(), edges.data(), n, cudaStreamSetCaptureDependencies);
}

}  // namespace mcao
