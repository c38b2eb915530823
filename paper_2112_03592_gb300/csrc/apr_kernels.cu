// CUDA kernels (sm_103a) of the APR tree: restriction (Sec. 3.4) and its adjoint, single channel (FP32).
#include <cuda_runtime.h>

#include <cstdint>

#include "apr_device.cuh"
#include "apr_internal.h"

namespace aprk {

namespace {

using namespace dev;

// ------------------------------------------------------------------------------------------------
// Tree kernels, one launch per tree level, one thread per tree node. A node's children are the
// cells (2z + a, 2x + b, 2y + e) of level l+1, each a particle or a tree node of that level; the
// node's child map (TreeNodePlan, built once per APR) gives their indices, so a thread reads its map
// and then all eight children at once.
// ------------------------------------------------------------------------------------------------
// The children of one tree node from its child map (TreeNodePlan): child c = 2k + e (k = (a, b) the
// child row, e the child's y parity; (a, b, e) order) is a particle (kind 1) or a tree node (kind 2)
// at index ix[c], or not present (kind 0: outside the grid, or missing from a sub-domain's index).
struct NodeChildren {
    int ix[8];
    int kind[8];
    __device__ __forceinline__ NodeChildren(const int4 &pw, const int4 &tw) {
        const int pv[4] = {pw.x, pw.y, pw.z, pw.w}, tv[4] = {tw.x, tw.y, tw.z, tw.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned pm = unsigned(pv[k]) >> 30, tm = unsigned(tv[k]) >> 30;
            const int pi = int(unsigned(pv[k]) & TNP_INDEX), ti = int(unsigned(tv[k]) & TNP_INDEX);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                // the second child of a kind follows the first of that kind
                const int skip = e ? 1 : 0;
                const bool isp = (pm >> e) & 1u, ist = (tm >> e) & 1u;
                kind[2 * k + e] = isp ? 1 : (ist ? 2 : 0);
                ix[2 * k + e] = isp ? pi + (skip & int(pm & 1u)) : ti + (skip & int(tm & 1u));
            }
        }
    }
};

__device__ __forceinline__ void load_node_plan(const TreeNodePlan *np, int node, int4 &pw, int4 &tw) {
    const int4 *q = reinterpret_cast<const int4 *>(np + node);
    pw = __ldg(q);
    tw = __ldg(q + 1);
}

// APR tree restriction for one level l (Sec. 3.4), one thread per tree node of the level (nodes
// [node0, node0 + n)): the node's value is the average of its children (particles and tree nodes of
// level l+1), summed in (a, b, e) order. Channel ch of C channels-last values.
__global__ void __launch_bounds__(NT) tree_restrict_kernel(const TreeNodePlan *__restrict__ nplan, int node0, int n,
                                                           const float *__restrict__ vals, float *tree, int C,
                                                           int ch) {
    pdl_trigger();
    const int i = int(blockIdx.x) * NT + int(threadIdx.x);
    const bool live = i < n;
    // the child map is static: read before waiting for the finer level's restriction (the launch
    // before this one), whose node values this level reads
    int4 pw = make_int4(0, 0, 0, 0), tw = pw;
    if (live) load_node_plan(nplan, node0 + i, pw, tw);
    pdl_wait();
    if (!live) return;
    const NodeChildren ch8(pw, tw);
    float v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const size_t at = size_t(ch8.ix[c]) * C + ch;
        v[c] = ch8.kind[c] == 1 ? vals[at] : (ch8.kind[c] == 2 ? tree[at] : 0.f);
    }
    float s = 0.f;
    int cnt = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c)
        if (ch8.kind[c]) {
            s += v[c];
            ++cnt;
        }
    tree[size_t(node0 + i) * C + ch] = cnt ? s / float(cnt) : 0.f;
}

// Backward through the tree averages, one level l (coarse to fine), one thread per tree node t of the
// level: each child (particle or tree node of level l+1) receives gt[t] / n_children(t). Every child
// has one parent, so each is written by one thread.
__global__ void __launch_bounds__(NT) tree_pushdown_kernel(const TreeNodePlan *__restrict__ nplan, int node0, int n,
                                                           float *gp, float *gt) {
    pdl_trigger();
    const int i = int(blockIdx.x) * NT + int(threadIdx.x);
    const bool live = i < n;
    // the child map is static: read before waiting for the coarser level's push-down (the launch
    // before this one), which writes this level's gt
    int4 pw = make_int4(0, 0, 0, 0), tw = pw;
    if (live) load_node_plan(nplan, node0 + i, pw, tw);
    pdl_wait();
    if (!live) return;
    const NodeChildren ch8(pw, tw);
    int cnt = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) cnt += ch8.kind[c] ? 1 : 0;
    const float share = gt[node0 + i] / float(cnt ? cnt : 1);
    float v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = ch8.kind[c] == 1 ? gp[ch8.ix[c]] : (ch8.kind[c] == 2 ? gt[ch8.ix[c]] : 0.f);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        if (ch8.kind[c] == 1) gp[ch8.ix[c]] = v[c] + share;
        else if (ch8.kind[c] == 2) gt[ch8.ix[c]] = v[c] + share;
    }
}

}  // namespace

// ---- launch entry points used by the C ABI (apr_api.cu)
cudaError_t launch_tree_restrict(const TreeNodePlan *np, int node0, int n, const float *vals, float *tree,
                                 cudaStream_t s, int C, int ch, bool pdl) {
    if (n <= 0) return cudaSuccess;
    return launch_pdl(tree_restrict_kernel, dim3((n + NT - 1) / NT), dim3(NT), 0, s, pdl, np, node0, n, vals, tree, C,
                      ch);
}

cudaError_t launch_tree_pushdown(const TreeNodePlan *np, int node0, int n, float *gp, float *gt, cudaStream_t s,
                                 bool pdl) {
    if (n <= 0) return cudaSuccess;
    return launch_pdl(tree_pushdown_kernel, dim3((n + NT - 1) / NT), dim3(NT), 0, s, pdl, np, node0, n, gp, gt);
}

}  // namespace aprk
