// join.cu -- the graph surgery of the joined ensemble launches (join.cuh).
#include "join.cuh"

#include <algorithm>

namespace pt {

static cudaError_t kernel_nodes(cudaGraph_t g, std::vector<cudaGraphNode_t>& out) {
    size_t nn = 0;
    cudaError_t e = cudaGraphGetNodes(g, nullptr, &nn);
    if (e != cudaSuccess || nn == 0) return e;
    std::vector<cudaGraphNode_t> nodes(nn);
    if ((e = cudaGraphGetNodes(g, nodes.data(), &nn)) != cudaSuccess) return e;
    for (cudaGraphNode_t x : nodes) {
        cudaGraphNodeType t;
        if ((e = cudaGraphNodeGetType(x, &t)) != cudaSuccess) return e;
        if (t == cudaGraphNodeTypeKernel) out.push_back(x);
    }
    return cudaSuccess;
}

cudaError_t join_table_bytes(cudaGraph_t g, size_t* bytes) {
    std::vector<cudaGraphNode_t> nodes;
    cudaError_t e = kernel_nodes(g, nodes);
    *bytes = 64 * 1024;
    for (cudaGraphNode_t x : nodes) {
        cudaKernelNodeParams kp{};
        if (e == cudaSuccess) e = cudaGraphKernelNodeGetParams(x, &kp);
        // arguments are at most 4 KB by the launch limit; ours stay below 1 KB
        *bytes += 1024 + 32 + sizeof(JoinBlock) * (size_t)kp.gridDim.x * kp.gridDim.y * kp.gridDim.z;
    }
    return e;
}

cudaError_t join_smem_limit(const void* joined) {
    cudaFuncAttributes fa{};
    int dev = 0, most = 0;
    cudaError_t e = cudaFuncGetAttributes(&fa, joined);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(joined, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 most - (int)fa.sharedSizeBytes);
    return e;
}

cudaError_t join_find(const JoinCtx& c, const void* fn, std::vector<cudaGraphNode_t>& found,
                      std::vector<cudaKernelNodeParams>& kps) {
    std::vector<cudaGraphNode_t> nodes;
    cudaError_t e = kernel_nodes(c.g, nodes);
    if (e != cudaSuccess) return e;
    for (cudaGraphNode_t x : nodes) {
        cudaKernelNodeParams kp{};
        if ((e = cudaGraphKernelNodeGetParams(x, &kp)) != cudaSuccess) return e;
        if (kp.func != fn) continue;
        found.push_back(x);
        kps.push_back(kp);
    }
    return cudaSuccess;
}

cudaError_t join_replace(JoinCtx& c, const std::vector<cudaGraphNode_t>& found,
                         const cudaKernelNodeParams& jp, unsigned cluster) {
    cudaError_t e;
    std::vector<cudaGraphNode_t> preds, succs;
    for (cudaGraphNode_t x : found) {
        size_t np = 0, ns = 0;
        if ((e = cudaGraphNodeGetDependencies(x, nullptr, nullptr, &np)) != cudaSuccess ||
            (e = cudaGraphNodeGetDependentNodes(x, nullptr, nullptr, &ns)) != cudaSuccess)
            return e;
        std::vector<cudaGraphNode_t> a(np), b(ns);
        std::vector<cudaGraphEdgeData> ea(np), eb(ns);
        if (np && (e = cudaGraphNodeGetDependencies(x, a.data(), ea.data(), &np)) != cudaSuccess)
            return e;
        if (ns && (e = cudaGraphNodeGetDependentNodes(x, b.data(), eb.data(), &ns)) != cudaSuccess)
            return e;
        preds.insert(preds.end(), a.begin(), a.end());
        succs.insert(succs.end(), b.begin(), b.end());
    }
    for (std::vector<cudaGraphNode_t>* v : {&preds, &succs}) {
        std::sort(v->begin(), v->end());
        v->erase(std::unique(v->begin(), v->end()), v->end());
    }
    cudaGraphNode_t node;
    if ((e = cudaGraphAddKernelNode(&node, c.g, preds.data(), preds.size(), &jp)) != cudaSuccess)
        return e;
    if (cluster > 1) {
        cudaKernelNodeAttrValue v{};
        v.clusterDim.x = cluster;
        v.clusterDim.y = v.clusterDim.z = 1;
        if ((e = cudaGraphKernelNodeSetAttribute(node, cudaLaunchAttributeClusterDimension, &v)) !=
            cudaSuccess)
            return e;
    }
    for (cudaGraphNode_t s : succs)
        if ((e = cudaGraphAddDependencies(c.g, &node, &s, nullptr, 1)) != cudaSuccess) return e;
    for (cudaGraphNode_t x : found)
        if ((e = cudaGraphDestroyNode(x)) != cudaSuccess) return e;
    ++c.joined;
    return cudaSuccess;
}

}  // namespace pt
