// CUDA kernels (sm_103a) of the APR tree: restriction (Sec. 3.4) and its adjoint, FP32 and 16-channel BF16.
//
// A node's children are the cells (2z + a, 2x + b, 2y + e) of the next finer level, each a particle or a
// tree node; the node's child map (TreeNodePlan, built once per APR) gives their indices. One launch takes
// a group of G <= 4 consecutive levels: a block takes R nodes of the group's coarsest level ("roots") and
// walks their descendants down, entry e of depth d being child e & 7 of entry e >> 3 of depth d - 1, so
// that the 8^(G-1) R entries of the deepest level are the block's threads. Restriction then averages
// upwards, the adjoint shares downwards, through shared memory. The maps are static: the walk runs before
// the wait for the launch before it (programmatic dependent launch).
//
// Why groups: a level of its own costs 3.5 to 5 us however small it is (map, children, store: three
// dependent accesses and a launch), and an image has five to eight levels. Groups are formed from the
// coarsest level up as long as the deepest level has at most tree_group_threads entries (tree_groups in
// apr_api.cu): small images take one or two launches instead of one per level, large ones keep a launch of
// their own for the finest two or three levels, whose nodes fill the chip by themselves (there a group
// would give most of its threads to particles).
#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include <cstdint>

#include "apr_device.cuh"
#include "apr_internal.h"

namespace aprk {

namespace {

using namespace dev;

constexpr unsigned REF_PARTICLE = 1u << 30, REF_NODE = 2u << 30;  // entry: kind | index; 0: no such cell

// Child c of a node from words k = c >> 1 of its child map.
__device__ __forceinline__ unsigned child_ref(unsigned pw, unsigned tw, int e) {
    const unsigned pm = pw >> 30, tm = tw >> 30;
    if ((pm >> e) & 1u) return REF_PARTICLE | ((pw & TNP_INDEX) + (e ? pm & 1u : 0u));
    if ((tm >> e) & 1u) return REF_NODE | ((tw & TNP_INDEX) + (e ? tm & 1u : 0u));
    return 0u;
}
__device__ __forceinline__ void all_children(const TreeNodePlan *maps, unsigned node, unsigned (&r)[8]) {
    const int4 *q = reinterpret_cast<const int4 *>(maps + node);
    const int4 pw = __ldg(q), tw = __ldg(q + 1);
    const int p[4] = {pw.x, pw.y, pw.z, pw.w}, t[4] = {tw.x, tw.y, tw.z, tw.w};
#pragma unroll
    for (int c = 0; c < 8; ++c) r[c] = child_ref(unsigned(p[c >> 1]), unsigned(t[c >> 1]), c & 1);
}

// Single channel (channel ch of C channels-last FP32 values): one thread per entry.
struct TreeF32 {
    static constexpr int E = 512, PARTS = 1;
    using V = float;
    const float *vals;
    float *tree;
    int C, ch;
    __device__ __forceinline__ V load(unsigned ref, int) const {
        return ref >= REF_NODE ? tree[size_t(ref & TNP_INDEX) * C + ch] : vals[size_t(ref & TNP_INDEX) * C + ch];
    }
    __device__ __forceinline__ void store(unsigned node, int, V v) const { tree[size_t(node) * C + ch] = v; }
    // the mean of the existing children, summed in (a, b, e) order
    __device__ __forceinline__ static V mean(const unsigned (&r)[8], const V (&v)[8]) {
        float s = 0.f;
        int n = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (r[c]) {
                s += v[c];
                ++n;
            }
        return n ? s / float(n) : 0.f;
    }
};

// 16 BF16 channels: two threads per entry, 8 channels each. The children are summed in FP32 in (a, b, e)
// order, divided by their count in FP32 and rounded to BF16 (nearest even).
struct TreeBf16 {
    static constexpr int E = 512, PARTS = 2;
    using V = uint4;
    const uint4 *vals;
    uint4 *tree;
    __device__ __forceinline__ V load(unsigned ref, int part) const {
        return (ref >= REF_NODE ? tree : vals)[2 * size_t(ref & TNP_INDEX) + part];
    }
    __device__ __forceinline__ void store(unsigned node, int part, V v) const { tree[2 * size_t(node) + part] = v; }
    __device__ __forceinline__ static V mean(const unsigned (&r)[8], const V (&v)[8]) {
        float acc[8];
        int n = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q] = 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            if (!r[c]) continue;
            ++n;
            const __nv_bfloat162 *p = reinterpret_cast<const __nv_bfloat162 *>(&v[c]);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 f = __bfloat1622float2(p[q]);
                acc[2 * q] = __fadd_rn(acc[2 * q], f.x);
                acc[2 * q + 1] = __fadd_rn(acc[2 * q + 1], f.y);
            }
        }
        const float nf = float(n ? n : 1);
        uint4 o;
        __nv_bfloat162 *p = reinterpret_cast<__nv_bfloat162 *>(&o);
#pragma unroll
        for (int q = 0; q < 4; ++q) p[q] = __floats2bfloat162_rn(__fdiv_rn(acc[2 * q], nf), __fdiv_rn(acc[2 * q + 1], nf));
        return o;
    }
};

// Entries of depth d start at entry_off(d) (the deepest first).
template <int E>
__device__ __forceinline__ int entry_off(int G, int d) {
    int o = 0;
    for (int k = G - 1; k > d; --k) o += E >> (3 * (G - 1 - k));
    return o;
}
template <int E>
constexpr int entries_total = E + E / 8 + E / 64 + E / 512 + 1;

// Fills ref (all depths but the deepest, and the deepest if `deepest`) and returns this thread's deepest
// entry. Ends with a block barrier if G > 1.
template <int E>
__device__ __forceinline__ unsigned walk(const TreeNodePlan *__restrict__ maps, int node0, int n, int G, int e, bool first,
                                         unsigned *ref) {
    const int R = E >> (3 * (G - 1));
    unsigned mine = 0;
    for (int d = 0; d < G; ++d) {
        const int cnt = R << (3 * d);
        if (e < cnt) {
            mine = 0;
            if (d == 0) {
                const int i = int(blockIdx.x) * R + e;
                if (i < n) mine = REF_NODE | unsigned(node0 + i);
            } else {
                const unsigned up = ref[entry_off<E>(G, d - 1) + (e >> 3)];
                if (up >= REF_NODE) {
                    const TreeNodePlan *m = maps + (up & TNP_INDEX);
                    const int k = (e & 7) >> 1;
                    mine = child_ref(unsigned(__ldg(&m->p[k])), unsigned(__ldg(&m->t[k])), e & 1);
                }
            }
            if (first && G > 1) ref[entry_off<E>(G, d) + e] = mine;
        }
        if (G > 1) __syncthreads();
    }
    return mine;
}

template <typename P>
__global__ void __launch_bounds__(P::E *P::PARTS) tree_restrict_kernel(const TreeNodePlan *__restrict__ maps, int node0, int n,
                                                                       int G, const P pol) {
    using V = typename P::V;
    constexpr int E = P::E, PARTS = P::PARTS;
    __shared__ unsigned ref[entries_total<E>];
    __shared__ V val[entries_total<E> * PARTS];
    pdl_trigger();
    const int e = int(threadIdx.x) / PARTS, part = int(threadIdx.x) % PARTS;
    const unsigned mine = walk<E>(maps, node0, n, G, e, part == 0, ref);
    unsigned kids[8] = {};
    if (mine >= REF_NODE) all_children(maps, mine & TNP_INDEX, kids);
    pdl_wait();   // the finer level's nodes are written by the launch before this one
    V v{};
    if (mine >= REF_NODE) {
        V c[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            c[k] = V{};
            if (kids[k]) c[k] = pol.load(kids[k], part);
        }
        v = P::mean(kids, c);
        pol.store(mine & TNP_INDEX, part, v);
    } else if (mine && G > 1) {
        v = pol.load(mine, part);
    }
    if (G == 1) return;
    val[e * PARTS + part] = v;
    __syncthreads();
    for (int d = G - 2; d >= 0; --d) {
        const int o = entry_off<E>(G, d), od = entry_off<E>(G, d + 1);
        if (e < (E >> (3 * (G - 1 - d)))) {
            const unsigned r = ref[o + e];
            V u{};
            if (r >= REF_NODE) {
                V c[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    kids[k] = ref[od + 8 * e + k];
                    c[k] = val[(od + 8 * e + k) * PARTS + part];
                }
                u = P::mean(kids, c);
                pol.store(r & TNP_INDEX, part, u);
            } else if (r) {
                u = pol.load(r, part);
            }
            val[(o + e) * PARTS + part] = u;
        }
        __syncthreads();
    }
}

// ---- adjoint: every child receives its parent's gradient / #children added, coarse to fine. Every child
// has one parent, so each is written by one thread.
struct PushF32 {
    static constexpr int E = 512, PARTS = 1;
    using V = float;
    float *gp, *gt;
    __device__ __forceinline__ V add(unsigned ref, int, V s) const {
        float *q = (ref >= REF_NODE ? gt : gp) + (ref & TNP_INDEX);
        const float v = *q + s;
        *q = v;
        return v;
    }
    __device__ __forceinline__ void add8(const unsigned (&r)[8], int, V s) const {
        float v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = r[c] ? (r[c] >= REF_NODE ? gt : gp)[r[c] & TNP_INDEX] : 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (r[c]) (r[c] >= REF_NODE ? gt : gp)[r[c] & TNP_INDEX] = v[c] + s;
    }
    __device__ __forceinline__ V node(unsigned i, int) const { return gt[i]; }
    __device__ __forceinline__ static V share(V v, int n) { return v / float(n ? n : 1); }
};

// 16 FP32 gradient channels: four threads per entry, 4 channels each.
struct Push16 {
    static constexpr int E = 256, PARTS = 4;
    using V = float4;
    float4 *gp, *gt;
    __device__ __forceinline__ float4 *at(unsigned r, int part) const {
        return (r >= REF_NODE ? gt : gp) + size_t(r & TNP_INDEX) * 4 + part;
    }
    __device__ __forceinline__ V add(unsigned ref, int part, V s) const {
        float4 *q = at(ref, part);
        float4 v = *q;
        v = make_float4(v.x + s.x, v.y + s.y, v.z + s.z, v.w + s.w);
        *q = v;
        return v;
    }
    __device__ __forceinline__ void add8(const unsigned (&r)[8], int part, V s) const {
        float4 v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = r[c] ? *at(r[c], part) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (r[c]) *at(r[c], part) = make_float4(v[c].x + s.x, v[c].y + s.y, v[c].z + s.z, v[c].w + s.w);
    }
    __device__ __forceinline__ V node(unsigned i, int part) const { return gt[size_t(i) * 4 + part]; }
    __device__ __forceinline__ static V share(V v, int n) {
        const float f = float(n ? n : 1);
        return make_float4(v.x / f, v.y / f, v.z / f, v.w / f);
    }
};

template <typename P>
__global__ void __launch_bounds__(P::E *P::PARTS) tree_pushdown_kernel(const TreeNodePlan *__restrict__ maps, int node0, int n,
                                                                       int G, const P pol) {
    using V = typename P::V;
    constexpr int E = P::E, PARTS = P::PARTS;
    __shared__ unsigned ref[entries_total<E>];
    __shared__ V sh[(E / 8 + E / 64 + E / 512 + 1) * PARTS];   // shares of the entries above the deepest level
    pdl_trigger();
    const int e = int(threadIdx.x) / PARTS, part = int(threadIdx.x) % PARTS;
    const unsigned mine = walk<E>(maps, node0, n, G, e, part == 0, ref);
    unsigned kids[8] = {};
    int nkids = 0;
    if (mine >= REF_NODE) {
        all_children(maps, mine & TNP_INDEX, kids);
#pragma unroll
        for (int c = 0; c < 8; ++c) nkids += kids[c] ? 1 : 0;
    }
    pdl_wait();   // the coarser level's gradients are written by the launch before this one
    for (int d = 0; d + 1 < G; ++d) {
        const int o = entry_off<E>(G, d), od = entry_off<E>(G, d + 1);
        if (e < (E >> (3 * (G - 1 - d)))) {
            const unsigned r = ref[o + e];
            if (r) {
                V v = d == 0 ? pol.node(r & TNP_INDEX, part) : pol.add(r, part, sh[(entry_off<E>(G, d - 1) - E + (e >> 3)) * PARTS + part]);
                if (r >= REF_NODE) {
                    int cnt = 0;
#pragma unroll
                    for (int k = 0; k < 8; ++k) cnt += ref[od + 8 * e + k] ? 1 : 0;
                    sh[(o - E + e) * PARTS + part] = P::share(v, cnt);
                }
            }
        }
        __syncthreads();
    }
    if (!mine) return;
    const V v = G == 1 ? pol.node(mine & TNP_INDEX, part)
                       : pol.add(mine, part, sh[(entry_off<E>(G, G - 2) - E + (e >> 3)) * PARTS + part]);
    if (mine >= REF_NODE) pol.add8(kids, part, P::share(v, nkids));
}

template <typename P>
cudaError_t launch_group(void (*kernel)(const TreeNodePlan *, int, int, int, P), const TreeNodePlan *np, int node0, int n,
                         int G, const P &pol, cudaStream_t s, bool pdl) {
    if (n <= 0) return cudaSuccess;
    const int R = P::E >> (3 * (G - 1));
    return launch_pdl(kernel, dim3((n + R - 1) / R), dim3(P::E * P::PARTS), 0, s, pdl, np, node0, n, G, pol);
}

}  // namespace

// ---- launch entry points (apr_api.cu, apr_mc.cu). A group's coarsest level holds nodes [node0, node0 + n).
cudaError_t launch_tree_restrict(const TreeNodePlan *np, const TreeGroup &g, const float *vals, float *tree, cudaStream_t s,
                                 int C, int ch, bool pdl) {
    return launch_group(tree_restrict_kernel<TreeF32>, np, g.node0, g.n, g.levels, TreeF32{vals, tree, C, ch}, s, pdl);
}
cudaError_t launch_tree_restrict_bf16(const TreeNodePlan *np, const TreeGroup &g, const uint16_t *vals, uint16_t *tree,
                                      cudaStream_t s, bool pdl) {
    return launch_group(tree_restrict_kernel<TreeBf16>, np, g.node0, g.n, g.levels,
                        TreeBf16{reinterpret_cast<const uint4 *>(vals), reinterpret_cast<uint4 *>(tree)}, s, pdl);
}
cudaError_t launch_tree_pushdown(const TreeNodePlan *np, const TreeGroup &g, float *gp, float *gt, cudaStream_t s, bool pdl) {
    return launch_group(tree_pushdown_kernel<PushF32>, np, g.node0, g.n, g.levels, PushF32{gp, gt}, s, pdl);
}
cudaError_t launch_tree_pushdown16(const TreeNodePlan *np, const TreeGroup &g, float *gp, float *gt, cudaStream_t s, bool pdl) {
    return launch_group(tree_pushdown_kernel<Push16>, np, g.node0, g.n, g.levels,
                        Push16{reinterpret_cast<float4 *>(gp), reinterpret_cast<float4 *>(gt)}, s, pdl);
}

}  // namespace aprk
