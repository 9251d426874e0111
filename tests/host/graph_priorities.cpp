// Preloaded: prints the priority of every kernel node of a graph that is
// instantiated.
#include <cuda_runtime.h>
#include <dlfcn.h>
#include <stdio.h>

#include <vector>

extern "C" cudaError_t cudaGraphInstantiate(cudaGraphExec_t *exec, cudaGraph_t graph, unsigned long long flags) {
    size_t n = 0;
    cudaGraphGetNodes(graph, nullptr, &n);
    std::vector<cudaGraphNode_t> nodes(n);
    cudaGraphGetNodes(graph, nodes.data(), &n);
    for (cudaGraphNode_t node : nodes) {
        cudaGraphNodeType type;
        cudaLaunchAttributeValue v;
        if (cudaGraphNodeGetType(node, &type) == cudaSuccess && type == cudaGraphNodeTypeKernel &&
            cudaGraphKernelNodeGetAttribute(node, cudaLaunchAttributePriority, &v) == cudaSuccess)
            printf("kernel priority %d\n", v.priority);
    }
    fflush(stdout);
    auto real = (cudaError_t(*)(cudaGraphExec_t *, cudaGraph_t, unsigned long long))dlsym(RTLD_NEXT, "cudaGraphInstantiate");
    return real(exec, graph, flags);
}
