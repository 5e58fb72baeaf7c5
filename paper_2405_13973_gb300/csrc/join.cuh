// join.cuh -- one launch for the same kernel of many ensemble members.
//
// An ensemble's step is captured member by member; a kernel that runs for a
// few microseconds on a few dozen blocks then costs more to launch than to
// run (256 crystals: 3,640 kernel nodes, about 3 us each whatever they do).
// After the capture every such kernel's nodes are replaced by one node over
// all of them: a table of the members' arguments and, per block, the member
// it works for and its place in that member's grid.  A kernel that can be
// joined keeps its work in a device function of (BlockId, arguments); the
// members' results do not depend on the join.
#pragma once
#include <cuda/std/tuple>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <utility>
#include <vector>

namespace pt {

// a block's place in its (member's) grid
struct BlockId {
    unsigned x, y, z, nx, ny, nz;
};
#ifdef __CUDACC__
__device__ __forceinline__ BlockId solo_block() {
    return {blockIdx.x, blockIdx.y, blockIdx.z, gridDim.x, gridDim.y, gridDim.z};
}
#endif

// per block of a joined launch
struct alignas(8) JoinBlock {
    int member, block;
};

struct JoinCtx {
    cudaGraph_t g = nullptr;
    unsigned char* dev = nullptr;       // tables on the device
    std::vector<unsigned char> host;    // and staged here (copied once all joins are made)
    size_t cap = 0;
    int joined = 0;                     // nodes made
};
// room for the tables of a captured graph
cudaError_t join_table_bytes(cudaGraph_t g, size_t* bytes);
// the kernel nodes of fn in the graph
cudaError_t join_find(const JoinCtx& c, const void* fn, std::vector<cudaGraphNode_t>& found,
                      std::vector<cudaKernelNodeParams>& kp);
// one node (kernel jp) in the place of the found ones: after every
// predecessor, before every successor of any of them
cudaError_t join_replace(JoinCtx& c, const std::vector<cudaGraphNode_t>& found,
                         const cudaKernelNodeParams& jp, unsigned cluster);
// as much dynamic shared memory as the device allows: one limit whatever the
// ensemble, so that none lowers what another's graph was made with
cudaError_t join_smem_limit(const void* joined);
// joins of each translation unit's kernels
cudaError_t join_push(JoinCtx& c);
cudaError_t join_tree(JoinCtx& c);
cudaError_t join_fmm(JoinCtx& c);
cudaError_t join_pairs(JoinCtx& c);

#ifdef __CUDACC__
template <class Body, int THREADS, class... A>
__global__ void __launch_bounds__(THREADS) k_joined(const cuda::std::tuple<A...>* args,
                                                    const uint4* dims, const JoinBlock* blocks) {
    const JoinBlock u = blocks[blockIdx.x];
    const uint4 d = dims[u.member];
    BlockId b;
    b.nx = d.x;
    b.ny = d.y;
    b.nz = d.z;
    b.x = (unsigned)u.block % d.x;
    b.y = (unsigned)u.block / d.x % d.y;
    b.z = (unsigned)u.block / d.x / d.y;
    cuda::std::apply([&](const A&... a) { Body{}(b, a...); }, args[u.member]);
}

template <class Tuple, size_t... I>
Tuple join_args(void** p, std::index_sequence<I...>) {
    return Tuple(*static_cast<const typename cuda::std::tuple_element<I, Tuple>::type*>(p[I])...);
}

// Joins the nodes of `solo`; KEY: the index of an argument (a pointer) that
// differs from member to member: should one member launch the kernel twice
// in a step, its launches depend on one another and nothing is joined.
template <class Body, int THREADS, int KEY, class... A>
cudaError_t join_kernel(JoinCtx& c, void (*solo)(A...), unsigned cluster = 1) {
    using Tuple = cuda::std::tuple<A...>;
    std::vector<cudaGraphNode_t> found;
    std::vector<cudaKernelNodeParams> kp;
    cudaError_t e = join_find(c, (const void*)solo, found, kp);
    const size_t n = found.size();
    if (e != cudaSuccess || n < 2) return e;
    size_t blocks = 0;
    unsigned smem = 0;
    for (size_t i = 0; i < n; ++i) {
        for (size_t j = 0; j < i; ++j)
            if (*(void**)kp[i].kernelParams[KEY] == *(void**)kp[j].kernelParams[KEY]) return cudaSuccess;
        if (kp[i].blockDim.x != kp[0].blockDim.x) return cudaSuccess;  // members of several orders
        blocks += (size_t)kp[i].gridDim.x * kp[i].gridDim.y * kp[i].gridDim.z;
        smem = kp[i].sharedMemBytes > smem ? kp[i].sharedMemBytes : smem;
    }
    auto room = [&](size_t bytes) {
        const size_t at = (c.host.size() + 255) / 256 * 256;
        c.host.resize(at + bytes);
        return at;
    };
    const size_t at_a = room(sizeof(Tuple) * n), at_d = room(sizeof(uint4) * n),
                 at_b = room(sizeof(JoinBlock) * blocks);
    if (c.host.size() > c.cap) return cudaErrorMemoryAllocation;
    JoinBlock* jb = reinterpret_cast<JoinBlock*>(c.host.data() + at_b);
    for (size_t i = 0; i < n; ++i) {
        const Tuple t = join_args<Tuple>(kp[i].kernelParams, std::index_sequence_for<A...>{});
        memcpy(c.host.data() + at_a + sizeof(Tuple) * i, &t, sizeof t);
        const uint4 d = make_uint4(kp[i].gridDim.x, kp[i].gridDim.y, kp[i].gridDim.z, 0);
        memcpy(c.host.data() + at_d + sizeof(uint4) * i, &d, sizeof d);
        for (unsigned b = 0; b < d.x * d.y * d.z; ++b) *jb++ = JoinBlock{(int)i, (int)b};
    }
    auto joined = k_joined<Body, THREADS, A...>;
    if (smem > 0 && (e = join_smem_limit((const void*)joined)) != cudaSuccess) return e;
    const Tuple* da = reinterpret_cast<const Tuple*>(c.dev + at_a);
    const uint4* dd = reinterpret_cast<const uint4*>(c.dev + at_d);
    const JoinBlock* db = reinterpret_cast<const JoinBlock*>(c.dev + at_b);
    void* args[] = {(void*)&da, (void*)&dd, (void*)&db};
    cudaKernelNodeParams jp{};
    jp.func = (void*)joined;
    jp.gridDim = dim3((unsigned)blocks);
    jp.blockDim = kp[0].blockDim;
    jp.sharedMemBytes = smem;
    jp.kernelParams = args;
    return join_replace(c, found, jp, cluster);
}
#endif

}  // namespace pt
