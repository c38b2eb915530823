// Multi-channel APR convolution with bfloat16 features and weights on the fifth-generation tensor cores
// (tcgen05), FP32 accumulation: the per-level filters of an APR CNN layer (Sec. 6), with the isotropic
// patch of Sec. 3.5 and the per-level convolution of Sec. 4.1 applied per channel pair.
//
// The kernels work on the convolution units (apr_unitplan.cpp). A block takes one unit and builds, from its
// slot entries, the source row of every cell of every slot (a particle's, a tree node's, or none) in shared
// memory; no feature is staged per slot. Up to 128 records (parents of 2 x 2 x 2 cells) are the M rows of
// one accumulator tile:
//   forward       D[record][child c, co] += sum over the 64 cells around the record of
//                                           U(cell)[ci] W[tap from child c to cell][ci][co]
//   data adjoint  the same with dL/dout at the cells and the flipped, transposed weights (children: the
//                 record's particles and tree nodes; for a coarser particle, the sum over its children)
//   weights       D[tap row][cell y, ci][e, co] += U(cell)[ci] g(child)[co], summed over the records
// The A operand of a cell (16 channels = one K step) is loaded from global memory by the row's own threads
// (lane = record) and written to tensor memory, eight cells per step, while the MMAs of the step before run.
// One cell serves up to eight children: a cell in reach of both children of an axis takes one MMA of twice the N, so a tile takes
// 120 MMAs of N = 16 to 64 instead of 27 per 128 children, and gathers 64 cells per record where one row
// per child gathered 27 per child (216 per record).
//
// One warp issues the MMAs; completion is signalled through mbarriers whose waits are bounded in time.
//
// Measured (1.0 M particles of a 256^3 image, kernels alone): forward 223 -> 63 us, data adjoint 550 -> 173 us
// (97 onto the children, 76 onto coarser particles), weight gradient 400 -> 100 us. The kernels before cut
// 8 x 8 x 64-cell tiles, which particles in thin shells leave mostly empty, into sub-tiles staged in shared
// memory, and gathered 27 cells per target. Tried on the way here, forward: the A operand in shared memory
// through 16-byte cp.async 131 us (a wavefront of the L1 pipe per 32-byte sector), with the four cells of a
// row in one instruction 113 us, MMAs issued by a warp of their own 102 us, through registers into tensor
// memory with warp-uniform MMA operands 74 us, 32-byte stores 66 us, records staged once per unit and more L1
// 60 us (63 with the weights laid out by every block, copy_weights). What bounds it now: the L1 pipe (68 %: the gather touches about a line per 32-byte cell) and a unit's
// chain of latencies, at two blocks per SM; without the gather 42 us, without the MMAs 61 of then 66 us. DRAM
// traffic is 73 MB, 11 us. The adjoints have fewer sources to gather and more rows: edge units take further
// tiles for their images (a third of the node adjoint's time at 256^3), leaf rows have few sources each.
#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <mutex>
#include <utility>

#include "apr_device.cuh"
#include "apr_internal.h"
#include "apr_units.cuh"

namespace aprk {

// apr_kernels.cu
cudaError_t launch_tree_restrict_bf16(const TreeNodePlan *np, const TreeGroup &g, const uint16_t *vals, uint16_t *tree,
                                      cudaStream_t s, bool pdl);
cudaError_t launch_tree_pushdown16(const TreeNodePlan *np, const TreeGroup &g, float *gp, float *gt, cudaStream_t s, bool pdl);

namespace {

using namespace dev;

constexpr int MC = 16;                      // channels (c_in = c_out)
constexpr int NTAP = 27;
constexpr int TILE = 128;                   // records per accumulator tile (M)
constexpr int WBLK = MC * MC * 2;           // one tap's 16 x 16 weights
constexpr int NWB = 36;                     // weight blocks of a level (see weight_block)
constexpr int W_LEVEL = NTAP * MC * MC;     // weights of a level
constexpr uint32_t TMEM_COLS = 256;         // D: child c = 4a + 2b + e in columns 16c .. 16c + 15; then the
constexpr uint32_t TM_A = 128;              // A operand: two buffers of eight cells of 8 columns
constexpr int STAGES = 2;
constexpr int NO_SOURCE = 0x7fffffff;       // source code of an empty cell; tree nodes have bit 31 set
constexpr int TNT = NT + 32;                // threads of the tile kernels: eight warps gather, the ninth issues the MMAs
static_assert(NT == 2 * TILE, "two threads per row");

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return uint32_t(__cvta_generic_to_shared(p)); }

// Shared-memory matrix descriptor, no swizzle: start address, leading-dimension byte offset (stride
// between core matrices along K) and stride-dimension byte offset (along M or N), version 1.
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return uint64_t((addr & 0x3FFFF) >> 4) | (uint64_t((lbo & 0x3FFFF) >> 4) << 16) |
           (uint64_t((sbo & 0x3FFFF) >> 4) << 32) | (uint64_t(1) << 46);
}

// Instruction descriptor of kind::f16: BF16 A and B, FP32 D, M x N, A and B both K-major or both MN-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, bool mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (mn ? (3u << 15) : 0u) | ((uint32_t(N) >> 3) << 17) |
           ((uint32_t(M) >> 4) << 24);
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t *bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ uint64_t globaltimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Wait for phase `parity` of the mbarrier; gives up after limit_ns nanoseconds (default one second)
// or 2^24 polls, whichever comes first.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, uint64_t limit_ns = 1000000000ull) {
    const uint32_t a = smem_u32(bar);
    uint64_t t0 = 0;
    for (uint32_t it = 0; it < (1u << 24); ++it) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
        if ((it & 15u) == 15u) {   // the clock is read at every 16th poll only
            const uint64_t t = globaltimer();
            if (t0 == 0) t0 = t;
            else if (t - t0 > limit_ns) return false;
        }
    }
    return false;
}

// D (tensor memory) [+]= A (tensor memory) x B (shared memory descriptor); executed by a converged warp, issued
// by the lane with `elected`, so that the operands stay warp-uniform.
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t bdesc, uint32_t idesc, uint32_t acc, uint32_t elected) {
    asm volatile(
        "{\n.reg .pred p, e;\nsetp.ne.b32 p, %4, 0;\nsetp.ne.b32 e, %5, 0;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(d),
        "r"(a), "l"(bdesc), "r"(idesc), "r"(acc), "r"(elected)
        : "memory");
}
__device__ __forceinline__ uint32_t elect_one() {
    uint32_t e;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(e));
    return e;
}
// D (tensor memory) [+]= A (shared memory descriptor) x B (shared memory descriptor); a converged warp, as mma_ts.
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc, uint32_t elected) {
    asm volatile(
        "{\n.reg .pred p, e;\nsetp.ne.b32 p, %4, 0;\nsetp.ne.b32 e, %5, 0;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc), "r"(elected)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint4 &a, const uint4 &b) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(a.x),
                 "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// 32 bytes at a 32-byte aligned address (16 below); not through the read-only path, as load_after_wait.
__device__ __forceinline__ void load32(const uint4 *p, uint4 &a, uint4 &b) {
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
                 : "l"(p));
}

__device__ __forceinline__ void load16(const uint4 *p, uint4 &a) {
    asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w) : "l"(p));
}
__device__ __forceinline__ uint16_t load_u16(const uint16_t *p) {
    uint16_t v;
    asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float load_bf16(const uint16_t *p) { return __uint_as_float(uint32_t(load_u16(p)) << 16); }
// 32 bytes to a 32-byte aligned address.
__device__ __forceinline__ void store32(void *p, const uint4 &a, const uint4 &b) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w),
                 "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
                 : "memory");
}
// 16 channels to a 16-byte aligned address; wide: 32-byte aligned. A lane per particle touches a line per store, so
// half as many stores are half the wavefronts (1 M particles: forward 75 -> 66 us, data adjoint 119 -> 108 us).
__device__ __forceinline__ void store_channels(float *p, const float (&v)[16], bool wide) {
    uint4 u[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        u[k] = make_uint4(__float_as_uint(v[4 * k]), __float_as_uint(v[4 * k + 1]), __float_as_uint(v[4 * k + 2]), __float_as_uint(v[4 * k + 3]));
    if (wide) {
        store32(p, u[0], u[1]);
        store32(p + 8, u[2], u[3]);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) reinterpret_cast<uint4 *>(p)[k] = u[k];
    }
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Bounded-wait outcome shared by the block: on a timeout every thread leaves through the same path;
// thread 0 records the error and waits once more (bounded) for the MMAs in flight.
__device__ __forceinline__ bool block_timed_out(bool ok, uint64_t *bar, uint32_t parity, unsigned *err) {
    const bool bad = __syncthreads_or(!ok) != 0;
    if (bad && threadIdx.x == 0) {
        atomicOr(err, ERR_TIMEOUT);
        mbar_wait(bar, parity);
    }
    return bad;
}

// Completion of the MMAs committed to `bar`: thread 0 (the issuing thread) waits on the mbarrier,
// the others at the block barrier that shares the outcome (so they spend no issue slots polling);
// tcgen05.fence::after_thread_sync after it orders their tensor-memory reads. True on a timeout.
__device__ __forceinline__ bool block_wait_mma(uint64_t *bar, uint32_t parity, unsigned *err) {
    const bool ok = threadIdx.x == 0 ? mbar_wait(bar, parity) : true;
    return block_timed_out(ok, bar, parity, err);
}

// Self-test of the bounded-wait path: one block waits on an mbarrier that nothing arrives at, gives up
// after limit_ns and records ERR_TIMEOUT, exactly as the tensor-core kernels do when their MMAs do
// not complete. Nothing faults; the context stays usable.
__global__ void bounded_wait_selftest_kernel(uint64_t limit_ns, unsigned *err) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) mbar_init(&bar);
    __syncthreads();
    const bool ok = mbar_wait(&bar, 0, limit_ns);
    if (__syncthreads_or(!ok) && threadIdx.x == 0) atomicOr(err, ERR_TIMEOUT);
}


// Records that the index does not cover the patch of a particle (a layout that was not validated).
__global__ void uncovered_kernel(unsigned *err) { atomicOr(err, ERR_DEVICE_CHECK); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ---------------------------------------------------------------- weights
// Weight blocks of a level: tap (tz, tx, ty) as a K-major B operand block (8-row groups of N at 256 bytes, K
// chunks of 8 at 128 bytes). A cell reaches, along each axis, child 0 with tap t and child 1 with tap
// t - 1, so the taps of neighbouring children are laid out one after the other: pair p = 0, 1 of (tz, tx) at
// blocks 18 p + 2 (3 tz + 2 - tx), holding ty = p + 1 (for child e = 0), then ty = p (e = 1). Two consecutive
// tx then serve the children b = 0, 1 of one MMA.
__host__ __device__ constexpr int pair_block(int p, int tz, int tx) { return 18 * p + 2 * (3 * tz + 2 - tx); }
__device__ __forceinline__ void weight_block(int blk, int &tz, int &tx, int &ty) {
    const int p = blk / 18, r = (blk % 18) >> 1;
    ty = p + 1 - (blk & 1);
    tz = r / 3;
    tx = 2 - r % 3;
}

// ---------------------------------------------------------------- unit staging
struct Rows {                         // row slots of the unit's records, then of a tile's image or leaf rows
    uint16_t base[9][UNIT_RECS + TILE];
    uint32_t mask[TILE];              // bit 3r + j: parent j of row r is a slot, at base[r] + the bits before it
};

// What every tile kernel keeps in shared memory. The gather reads every cell about eight times and lives on the L1
// cache, which is what two blocks leave of 256 KB: nothing else belongs here (forward of 1 M particles with 28 KB
// of L1 82 to 86 us, with 60 KB 66 us, with 92 KB 60 us).
struct McSmem {
    int code[8][PLANE];               // source of every cell c of every slot
    Rows rows;
    alignas(128) unsigned char W[NWB * WBLK];
    int4 children[UNIT_RECS];         // the records' child particles (TreeNodePlan::p)
    uint64_t bar[STAGES];             // MMAs that read buffer s have completed
    uint32_t tmem;
};
constexpr int IMAGE_ROWS = TILE / 2;   // image rows of a tile
struct McRowLists {                   // rows of several images per record
    int first[UNIT_RECS + 1];         // first row of each record
    int wsum[NWARP];
};
struct McAdjSmem {
    McSmem s;
    alignas(16) float4 sums[IMAGE_ROWS * 32];   // image sums (image_chunk)
    int4 nodes[UNIT_RECS];            // the records' tree-node children (TreeNodePlan::t)
    uint16_t edge[UNIT_RECS];         // their edge words
    McRowLists list;
};
struct McLeafSmem {
    McSmem s;
    alignas(16) float4 sums[2][TILE * 4];   // a row's sums over the four cells of one z plane
    uint32_t mask[UNIT_RECS];         // of the records
    int particle[UNIT_RECS];
    uint16_t edge[UNIT_RECS];
    uint8_t skip[TILE];               // cells of a row outside the grid: no part of the source (zero boundary)
    McRowLists list;
};

// Source codes of the unit's slots. VALUES: particles, tree nodes and coarser particles; else the level-l
// particles only, and nothing outside the grid.
template <bool VALUES>
__device__ __forceinline__ void stage_codes(const UnitView &U, const UnitHdr &h, bool leaf, bool reflect, int (*code)[PLANE]) {
    const int tid = threadIdx.x, nt = int(blockDim.x);
    const uint4 *pure = (leaf ? U.lpure : U.pure) + h.pure0;
    const TreeNodePlan *nmap = (leaf ? U.lnmap : U.nmap) + h.node0;
    const uint32_t *ninfo = (leaf ? U.lninfo : U.ninfo) + h.node0;
    if (tid < 3)
#pragma unroll
        for (int c = 0; c < 8; ++c) code[c][ZERO_SLOT + tid] = NO_SOURCE;
    auto put_pure = [&](const uint4 &q) {
        const unsigned p[4] = {q.x, q.y, q.z, q.w}, s = pure_slot(q);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            code[2 * k][s] = int(p[k] & 0x0fffffffu);
            code[2 * k + 1][s] = int(p[k] & 0x0fffffffu) + 1;
        }
    };
    auto put_node = [&](const int4 &pw, const int4 &tw, unsigned info) {
        const Octet o(pw, tw);
        int v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c)
            v[c] = o.kind[c] == 1 ? o.ix[c] : (VALUES && o.kind[c] == 2 ? int(unsigned(o.ix[c]) | 0x80000000u) : NO_SOURCE);
        if (info >> UE_MIRROR) edge_octet(v, info, VALUES && reflect, NO_SOURCE);
#pragma unroll
        for (int c = 0; c < 8; ++c) code[c][info & UE_SLOT] = v[c];
    };
    auto put_other = [&](const uint2 &e, int i) {
        int v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = VALUES && i < h.nleaf ? int(e.x) : NO_SOURCE;
        if (e.y >> UE_MIRROR) edge_octet(v, e.y, VALUES && reflect, NO_SOURCE);
#pragma unroll
        for (int c = 0; c < 8; ++c) code[c][e.y & UE_SLOT] = v[c];
    };
    // the first entries of every kind in flight together, then what is left
    const uint2 *oth = U.oth + h.oth0;
    uint4 q[2];
    uint2 e[2];
    int4 pw = make_int4(0, 0, 0, 0), tw = pw;
    unsigned info = 0;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        q[u] = tid + u * nt < h.npure ? __ldg(pure + tid + u * nt) : make_uint4(0, 0, 0, 0);
        e[u] = tid + u * nt < h.noth ? __ldg(oth + tid + u * nt) : make_uint2(0, 0);
    }
    if (tid < h.nnode) {
        const int4 *m = reinterpret_cast<const int4 *>(nmap + tid);
        pw = __ldg(m);
        if (VALUES) tw = __ldg(m + 1);
        info = __ldg(ninfo + tid);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        if (tid + u * nt < h.npure) put_pure(q[u]);
        if (tid + u * nt < h.noth) put_other(e[u], tid + u * nt);
    }
    if (tid < h.nnode) put_node(pw, tw, info);
    for (int i = tid + 2 * nt; i < h.npure; i += nt) put_pure(__ldg(pure + i));
    for (int i = tid + 2 * nt; i < h.noth; i += nt) put_other(__ldg(oth + i), i);
    for (int i = tid + nt; i < h.nnode; i += nt) {
        const int4 *m = reinterpret_cast<const int4 *>(nmap + i);
        put_node(__ldg(m), VALUES ? __ldg(m + 1) : make_int4(0, 0, 0, 0), __ldg(ninfo + i));
    }
}

// Record `rec` of a node unit at its own place: all 27 parents are slots (one set of loads: nine dependent
// ones would cost more than the row's sums). Thread r keeps record r of the unit from its header to the staging,
// so that neither the rows nor the children of any tile wait for another chain of loads (record by record per tile:
// forward of 1 M particles 66 us, data adjoint 108 us, leaf adjoint 76 us; so 60, 96 and 71 us, the last two with the
// images' sums below).
struct NodeRow {
    uint2 r0, r1, r2;
    int4 pw, tw;
    __device__ __forceinline__ void load(const UnitView &U, const UnitHdr &h, bool nodes) {
        if (int(threadIdx.x) >= h.nrec) return;
        const uint2 *q = reinterpret_cast<const uint2 *>(U.rec + h.rec0 + threadIdx.x);
        r0 = __ldg(q);
        r1 = __ldg(q + 1);
        r2 = __ldg(q + 2);
        const int4 *m = reinterpret_cast<const int4 *>(U.nplan + r0.x);
        pw = __ldg(m);
        if (nodes) tw = __ldg(m + 1);
    }
    // Rows past the unit's records read the empty slots.
    template <typename Smem>
    __device__ __forceinline__ void put(Smem &S, const UnitHdr &h) const {
        const int r = threadIdx.x;
        if (r >= UNIT_RECS) return;
        unsigned b[9];
        unpack_bases(r0.y, r1, r2, b);
#pragma unroll
        for (int k = 0; k < 9; ++k) S.rows.base[k][r] = uint16_t(r < h.nrec ? b[k] : ZERO_SLOT);
        S.children[r] = r < h.nrec ? pw : make_int4(0, 0, 0, 0);
    }
    __device__ __forceinline__ void put_nodes(McAdjSmem &A, const UnitHdr &h) const {
        const int r = threadIdx.x;
        if (r >= UNIT_RECS) return;
        A.nodes[r] = r < h.nrec ? tw : make_int4(0, 0, 0, 0);
        A.edge[r] = uint16_t(r < h.nrec ? r0.y & 0xffffu : 0u);
    }
};
// Row r of a tile: in the adjoint record i of the unit at the image of shift t (edge_shifts; 0: its own place), ...
__device__ __forceinline__ void put_image_row(Rows &R, int r, int i, int t) {
    const int iz = t >> 4, ix = (t >> 2) & 3, iy = t & 3, dy = iy == 1 ? -1 : (iy == 0 ? 0 : iy - 1);
    unsigned mask = 0;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const int oz = image_layer(iz, q / 3), ox = image_layer(ix, q % 3);
        if (oz >= 0 && ox >= 0) {
            R.base[q][UNIT_RECS + r] = uint16_t(int(R.base[3 * oz + ox][i]) + dy);
            mask |= 7u << (3 * q);
        }
    }
    R.mask[r] = mask;
}
// ... record i, with slots `all`, of a leaf unit.
__device__ __forceinline__ void put_leaf_row(Rows &R, int r, int i, unsigned all, int t) {
    const int iz = t >> 4, ix = (t >> 2) & 3, iy = t & 3;
    unsigned mask = 0;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const int oz = image_layer(iz, q / 3), ox = image_layer(ix, q % 3), o = 3 * oz + ox;
        if (oz >= 0 && ox >= 0) {
            const unsigned m = (all >> (3 * o)) & 7u;
            R.base[q][UNIT_RECS + r] = uint16_t(R.base[o][i] + (iy == 0 ? 0 : __popc(m & (iy == 3 ? 3u : 1u))));
            mask |= (iy == 0 ? m : (iy == 1 ? (m << 1) & 4u : (m >> (iy - 1)) & 1u)) << (3 * q);
        }
    }
    R.mask[r] = mask;
}

// Source code of cell (iz, ix, iy) (0..3 per axis, from one before the parent's first cell) of row r.
__device__ __forceinline__ int cell_code(const int (*code)[PLANE], unsigned m, unsigned base, int c0, int iy) {
    const int j = (iy + 1) >> 1;
    return (m >> j) & 1u ? code[c0 + ((iy + 1) & 1)][base + __popc(m & ((1u << j) - 1u))] : NO_SOURCE;
}

__device__ __forceinline__ const uint4 *source_row(const uint4 *vals, const uint4 *tree, int code) {
    return (code < 0 ? tree : vals) + 2 * size_t(code == NO_SOURCE ? 0 : code & 0x7fffffff);
}

// ---------------------------------------------------------------- the tile GEMM
// Step k: the cell rows (iz, ix = x0) and (iz, x0 + 1), iz and x0 from the order below (the first step's rows
// both reach both z children, and its second row all eight children; see issue_row).
__device__ __forceinline__ int step_z(int k) { return k < 2 ? 1 : (k < 4 ? 0 : k >> 1); }
__device__ __forceinline__ int step_x(int k) { return 2 * (k & 1); }

// The four cells of row (iz, ix) of tile row r: up to 128 contiguous bytes. wide: 32-byte aligned features,
// one load per cell (lane = record touches 16 lines per load either way; 16-byte loads touch them twice).
// FULL: node records at their own place (no mask: all 27 parents are slots).
template <bool FULL>
struct CellRow {
    uint4 v[4][2];
    __device__ __forceinline__ void load(const int (*code)[PLANE], const Rows &rows, int r, int iz, int ix,
                                         const uint4 *__restrict__ vals, const uint4 *__restrict__ tree, bool wide) {
        const int q = ((iz + 1) >> 1) * 3 + ((ix + 1) >> 1), c0 = ((iz + 1) & 1) * 4 + ((ix + 1) & 1) * 2;
        const unsigned m = FULL ? 7u : (rows.mask[r - UNIT_RECS] >> (3 * q)) & 7u, base = rows.base[q][r];
        int src[4];
#pragma unroll
        for (int iy = 0; iy < 4; ++iy)
            src[iy] = FULL ? code[c0 + ((iy + 1) & 1)][base + ((iy + 1) >> 1)] : cell_code(code, m, base, c0, iy);
#pragma unroll
        for (int iy = 0; iy < 4; ++iy) {
            v[iy][0] = v[iy][1] = make_uint4(0, 0, 0, 0);
            if (src[iy] != NO_SOURCE) {
                const uint4 *p = source_row(vals, tree, src[iy]);
                if (wide) {
                    load32(p, v[iy][0], v[iy][1]);
                } else {
                    load16(p, v[iy][0]);
                    load16(p + 1, v[iy][1]);
                }
            }
        }
    }
    __device__ __forceinline__ void store(uint32_t a) const {
#pragma unroll
        for (int iy = 0; iy < 4; ++iy) tmem_st8(a + 8 * iy, v[iy][0], v[iy][1]);
    }
};

// MMAs of cell row (iz, ix) (one warp), all operands constants away from the bases: built at run time they
// cost more than the MMAs take. INIT: the first MMAs of the tile; cell (1, 1, 1) reaches all eight children
// and overwrites D.
template <int iz, int ix, bool INIT>
__device__ __forceinline__ void issue_row(uint32_t D, uint32_t A, uint64_t W, uint32_t el) {
    constexpr int b0 = ix == 3 ? 1 : 0, nb = ix == 0 || ix == 3 ? 1 : 2;
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        const int iy = o == 0 ? 1 : (o == 1 ? 2 : (o == 2 ? 0 : 3));
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const int tz = iz - a;
            if (tz < 0 || tz > 2) continue;
            if (iy == 1 || iy == 2) {
                mma_ts(D + 64 * a + 32 * b0, A + 8 * iy, W + pair_block(iy - 1, tz, ix - b0) * (WBLK >> 4), idesc_bf16(128, 32 * nb, false),
                       INIT && o == 0 ? 0u : 1u, el);
            } else {
#pragma unroll
                for (int b = b0; b < b0 + nb; ++b)   // ty = 0 for child e = 0, ty = 2 for e = 1
                    mma_ts(D + 64 * a + 32 * b + (iy == 3 ? 16 : 0), A + 8 * iy,
                           W + (iy == 0 ? pair_block(0, tz, ix - b) + 1 : pair_block(1, tz, ix - b)) * (WBLK >> 4),
                           idesc_bf16(128, 16, false), 1u, el);
            }
        }
    }
}
__device__ __forceinline__ void issue_step(uint32_t D, uint32_t A, uint64_t W, int k, uint32_t el) {
    switch (k) {
        case 0: issue_row<1, 1, true>(D, A + 32, W, el); issue_row<1, 0, false>(D, A, W, el); break;
        case 1: issue_row<1, 2, false>(D, A, W, el); issue_row<1, 3, false>(D, A + 32, W, el); break;
        case 2: issue_row<0, 0, false>(D, A, W, el); issue_row<0, 1, false>(D, A + 32, W, el); break;
        case 3: issue_row<0, 2, false>(D, A, W, el); issue_row<0, 3, false>(D, A + 32, W, el); break;
        case 4: issue_row<2, 0, false>(D, A, W, el); issue_row<2, 1, false>(D, A + 32, W, el); break;
        case 5: issue_row<2, 2, false>(D, A, W, el); issue_row<2, 3, false>(D, A + 32, W, el); break;
        case 6: issue_row<3, 0, false>(D, A, W, el); issue_row<3, 1, false>(D, A + 32, W, el); break;
        default: issue_row<3, 2, false>(D, A, W, el); issue_row<3, 3, false>(D, A + 32, W, el); break;
    }
}

// D = the tile's sums (S.rows, S.code, S.W and the tensor memory are set up, with a barrier since). Eight
// warps load: warps q and q + 4 the rows 32 q .. 32 q + 31, one cell row each; the loads of step k + 1 are in
// flight while step k is written to tensor memory and handed to the ninth warp, which issues the MMAs. A
// buffer is written again once the MMAs of two steps before have completed. phase: one bit per buffer.
// True on a timeout. FULL: rows row0 .. of the unit's records; else the tile's rows.
template <bool FULL>
__device__ __forceinline__ bool tile_gemm(McSmem &S, int row0, const uint4 *__restrict__ vals, const uint4 *__restrict__ tree, bool wide,
                                          uint32_t D, uint32_t &phase, unsigned *err) {
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int q = warp & 3, half = warp >> 2, r = (FULL ? row0 : UNIT_RECS) + 32 * q + lane;
    const uint64_t W = sdesc(smem_u32(S.W), 128, 256);
    bool ok = true;
    if (warp < NWARP) {
        const uint32_t a0 = D + TM_A + (uint32_t(32 * q) << 16) + 32 * half;
        CellRow<FULL> c;
        c.load(S.code, S.rows, r, step_z(0), step_x(0) + half, vals, tree, wide);
#pragma unroll 1
        for (int k = 0; k < 8; ++k) {
            if (k >= 2) ok = mbar_wait(&S.bar[k & 1], (phase >> (k & 1)) & 1u);
            if (k >= 2) phase ^= 1u << (k & 1);
            __syncwarp();
            tc_fence_after();
            c.store(a0 + 64 * (k & 1));
            tmem_wait_st();
            tc_fence_before();
            if (k + 1 < 8) c.load(S.code, S.rows, r, step_z(k + 1), step_x(k + 1) + half, vals, tree, wide);
            if (__syncthreads_or(!ok)) break;
        }
    } else {
        const uint32_t el = elect_one();
#pragma unroll 1
        for (int k = 0; k < 8; ++k) {
            if (k >= 2) phase ^= 1u << (k & 1);
            if (__syncthreads_or(false)) {
                ok = false;
                break;
            }
            tc_fence_after();
            issue_step(D, D + TM_A + 64 * (k & 1), W, k, el);
            if (el) mma_commit(&S.bar[k & 1]);
            __syncwarp();
        }
    }
    // the last two steps
    if (ok) ok = mbar_wait(&S.bar[0], phase & 1u) && mbar_wait(&S.bar[1], (phase >> 1) & 1u);
    const bool bad = block_timed_out(ok, &S.bar[1], (phase >> 1) & 1u, err);
    phase ^= 3u;
    tc_fence_after();
    return bad;
}

// A level's weights W[co][ci][tap] into S.W as the B operand's blocks (weight_block): forward N = co, K = ci, adjoint
// N = ci, K = co, taps flipped. They arrive as they lie in memory, every thread takes the 27 taps of one (n, k),
// and the blocks are written over them. Every block does this for itself: a kernel that laid them out ahead of each
// convolution needed a buffer in the handle, which calls on two streams overwrote for one another. Measured with that
// kernel and without: training step of 1 M particles 394.7 and 393.5 us, of 45 k 80.1 and 77.5, four layers of 2.4 M 658.7
// and 658.2 (661 with the copy behind the tensor-memory allocation).
__device__ __forceinline__ void copy_weights(McSmem &S, const uint16_t *__restrict__ W, int lev) {
    const int tid = threadIdx.x;
    const uint16_t *src = W + size_t(lev) * W_LEVEL;
    uint16_t *w = reinterpret_cast<uint16_t *>(S.W);
    if ((reinterpret_cast<uintptr_t>(W) & 15u) == 0) {
        for (int i = tid; i < W_LEVEL / 8; i += TNT) cp_async16(smem_u32(w + 8 * i), src + 8 * i, true);
    } else {
        for (int i = tid; i < W_LEVEL; i += TNT) w[i] = load_u16(src + i);
    }
    cp_commit();
}
template <bool ADJ>
__device__ __forceinline__ void transpose_weights(McSmem &S) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint16_t *w = reinterpret_cast<uint16_t *>(S.W);
    cp_wait<0>();
    block_sync();
    // a warp's lanes: 4 n x 8 k (its 2-byte stores fill 16 banks)
    const int n = 4 * (warp >> 1) + (lane >> 3), k = 8 * (warp & 1) + (lane & 7);
    uint16_t t[NTAP];
    if (warp < NWARP)
#pragma unroll
        for (int e = 0; e < NTAP; ++e) t[e] = w[(ADJ ? k * MC + n : n * MC + k) * NTAP + (ADJ ? NTAP - 1 - e : e)];
    block_sync();
    if (warp < NWARP)
#pragma unroll
        for (int blk = 0; blk < NWB; ++blk) {
            int tz, tx, ty;
            weight_block(blk, tz, tx, ty);
            w[blk * MC * MC + ((n >> 3) * 2 + (k >> 3)) * 64 + (n & 7) * 8 + (k & 7)] = t[(tz * 3 + tx) * 3 + ty];
        }
}

// Block set-up shared by the tile kernels: tensor memory, mbarrier, the level's weights. The caller's next
// tile_ready publishes S.tmem and the weights.
template <bool ADJ>
__device__ __forceinline__ void tile_setup(McSmem &S, const uint16_t *W, int lev) {
    const int tid = threadIdx.x;
    copy_weights(S, W, lev);   // (before the allocation, which its warp waits for)
    if (tid < STAGES) mbar_init(&S.bar[tid]);
    __syncwarp();
    if ((tid >> 5) == 0) tmem_alloc(smem_u32(&S.tmem), TMEM_COLS);
    transpose_weights<ADJ>(S);
}
// Ends the set-up: weights visible to the tensor cores, rows and codes visible to the block.
__device__ __forceinline__ void tile_ready() {
    fence_async_smem();
    tc_fence_before();
    block_sync();
    tc_fence_after();
}
__device__ __forceinline__ void tile_teardown(const McSmem &S) {
    tc_fence_before();
    block_sync();
    if ((threadIdx.x >> 5) == 0) tmem_dealloc(S.tmem, TMEM_COLS);
}

// Orders the tile's tensor-memory reads before the next tile's MMAs.
__device__ __forceinline__ void tile_done() {
    tc_fence_before();
    block_sync();
    tc_fence_after();
}

// ---------------------------------------------------------------- forward
// Where the outputs go: out (float32 [N][16]) receives the convolution; if out_bf16 is given instead, it
// receives bf16(max(conv, 0)), the next layer's input in an APR CNN; if y is given instead, it receives the
// network's read-out x + inv_scale conv[0], and the convolution itself is not written (2.4 M particles: 65 us
// less than writing 64 bytes per particle and reading 4 of them back).
struct McOutput {
    float *out;
    uint4 *out_bf16;
    float *y;
    const float *x;
    float inv_scale;
};
__global__ void __launch_bounds__(TNT, 2) mc_fwd_kernel(const UnitView U, const uint4 *__restrict__ vals,
                                                       const uint4 *__restrict__ tree, const uint16_t *__restrict__ W, int bc,
                                                       const McOutput o, unsigned *err) {
    extern __shared__ __align__(128) unsigned char smraw[];
    McSmem &S = *reinterpret_cast<McSmem *>(smraw);
    pdl_trigger();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const UnitHdr h = U.work[blockIdx.x];
    NodeRow row;
    row.load(U, h, false);
    stage_codes<true>(U, h, false, bc == APR_BC_REFLECT, S.code);
    row.put(S, h);
    pdl_wait();   // the tree is written by the launch before this one
    tile_setup<false>(S, W, h.lev);
    tile_ready();
    const uint32_t D = S.tmem;
    const bool wide = ((reinterpret_cast<uintptr_t>(vals) | reinterpret_cast<uintptr_t>(tree)) & 31u) == 0;
    const bool wide_out = ((reinterpret_cast<uintptr_t>(o.out) | reinterpret_cast<uintptr_t>(o.out_bf16)) & 31u) == 0;
    uint32_t phase = 0;
    const int q = warp & 3, a = warp >> 2;
    for (int t0 = 0; t0 < h.nrec; t0 += TILE) {
        if (tile_gemm<true>(S, t0, vals, tree, wide, D, phase, err)) break;
        // lane = record, this warp's half of the children (a): the particles' outputs
        int2 pw = make_int2(0, 0);
        if (warp < NWARP) pw = reinterpret_cast<const int2 *>(S.children + t0 + 32 * q + lane)[a];
        if (warp < NWARP)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float v[16];
            tmem_ld16(D + (uint32_t(32 * q) << 16) + 64 * a + 16 * c, v);
            const unsigned w = unsigned(c < 2 ? pw.x : pw.y), pm = w >> 30;
            if ((pm >> (c & 1)) & 1u) {
                const size_t p = (w & TNP_INDEX) + (c & 1 ? pm & 1u : 0u);
                if (o.y) {
                    o.y[p] = __fadd_rn(o.x[p], __fmul_rn(o.inv_scale, v[0]));
                } else if (o.out_bf16) {
                    uint4 w2[2];
                    __nv_bfloat162 *b2 = reinterpret_cast<__nv_bfloat162 *>(w2);
#pragma unroll
                    for (int k = 0; k < MC / 2; ++k) b2[k] = __floats2bfloat162_rn(fmaxf(v[2 * k], 0.f), fmaxf(v[2 * k + 1], 0.f));
                    if (wide_out) {
                        store32(o.out_bf16 + 2 * p, w2[0], w2[1]);
                    } else {
                        o.out_bf16[2 * p] = w2[0];
                        o.out_bf16[2 * p + 1] = w2[1];
                    }
                } else {
                    store_channels(o.out + p * MC, v, wide_out);
                }
            }
        }
        tile_done();
    }
    tile_teardown(S);
}

// ---------------------------------------------------------------- data adjoint
// 4 channels at p, added.
__device__ __forceinline__ void add4(float *p, const float4 &s) {
    float4 *q = reinterpret_cast<float4 *>(p);
    float4 v = *q;
    v.x += s.x;
    v.y += s.y;
    v.z += s.z;
    v.w += s.w;
    *q = v;
}

// Exclusive prefix of n (one value of each of the first NT threads) into first[0 .. NT]. Ends with a barrier.
__device__ __forceinline__ int prefix_rows(McRowLists &S, int n) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31 && warp < NWARP) S.wsum[warp] = incl;
    block_sync();
    int before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < NWARP; ++w) {
        before += w < warp ? S.wsum[w] : 0;
        total += S.wsum[w];
    }
    if (tid < NT) S.first[tid] = before + incl - n;
    if (tid == 0) S.first[NT] = total;
    block_sync();
    return total;
}
// The record (of n) that owns row k.
__device__ __forceinline__ int row_owner(const McRowLists &S, int n, int k) {
    int a = 0, b = n;
    while (b - a > 1) {
        const int m = (a + b) / 2;
        if (S.first[m] <= k) a = m;
        else b = m;
    }
    return a;
}
// The n-th set bit of m (n < its population count).
__device__ __forceinline__ int nth_bit(unsigned long long m, int n) {
    for (; n > 0; --n) m &= m - 1ull;
    return __ffsll((long long)m) - 1;
}
// Images of an edge record (edge_shifts<1> without its own place), after them one row that repeats its own
// place if it has missing children (their sums belong to their siblings).
__device__ __forceinline__ int image_rows(unsigned edge) {
    return __popcll(edge_shifts<1>(edge)) - 1 + (missing_children(edge) ? 1 : 0);
}
__device__ __forceinline__ int image_row(unsigned edge, int j) {
    const unsigned long long m = edge_shifts<1>(edge) & ~1ull;
    return j < __popcll(m) ? nth_bit(m, j) : 0;
}

// Float4 chunk k (0..31) of row r in the 64 x 128-float staging of the image sums (16-byte chunks swizzled by
// the row: conflict-free for lane = row).
__device__ __forceinline__ float4 *image_chunk(McAdjSmem &S, int r, int k) {
    return S.sums + r * 32 + (k ^ (r & 31));
}

// Data adjoint onto the children of every record: particles (gp) and tree nodes (gt) are stored, then, with
// reflection, the images of the edge records are added.
__global__ void __launch_bounds__(TNT, 2) mc_adjoint_kernel(const UnitView U, const uint16_t *__restrict__ W, int bc,
                                                           const uint4 *__restrict__ gout, float *__restrict__ gp,
                                                           float *__restrict__ gt, unsigned *err) {
    extern __shared__ __align__(128) unsigned char smraw[];
    McAdjSmem &M = *reinterpret_cast<McAdjSmem *>(smraw);
    pdl_trigger();
    McSmem &S = M.s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const UnitHdr h = U.work_adj[blockIdx.x];
    NodeRow row;
    row.load(U, h, true);
    stage_codes<false>(U, h, false, false, S.code);
    row.put(S, h);
    row.put_nodes(M, h);
    pdl_wait();   // dL/dout and the weights may be written by the launch before this one
    tile_setup<true>(S, W, h.lev);
    tile_ready();
    const uint32_t D = S.tmem;
    const bool wide = (reinterpret_cast<uintptr_t>(gout) & 31u) == 0;
    const bool wide_out = ((reinterpret_cast<uintptr_t>(gp) | reinterpret_cast<uintptr_t>(gt)) & 31u) == 0;
    uint32_t phase = 0;
    const int q = warp & 3, a = warp >> 2;
    bool failed = false;
    for (int t0 = 0; t0 < h.nrec && !failed; t0 += TILE) {
        failed = tile_gemm<true>(S, t0, gout, gout, wide, D, phase, err);
        if (failed) break;
        int pk[2] = {}, tk[2] = {};
        if (warp < NWARP) {
            const int2 p = reinterpret_cast<const int2 *>(S.children + t0 + 32 * q + lane)[a];
            const int2 t = reinterpret_cast<const int2 *>(M.nodes + t0 + 32 * q + lane)[a];
            pk[0] = p.x;
            pk[1] = p.y;
            tk[0] = t.x;
            tk[1] = t.y;
        }
        if (warp < NWARP)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float v[16];
            tmem_ld16(D + (uint32_t(32 * q) << 16) + 64 * a + 16 * c, v);
            const unsigned p = unsigned(pk[c >> 1]), t = unsigned(tk[c >> 1]), pm = p >> 30, tm = t >> 30;
            const int e = c & 1;
            float *dst = nullptr;
            if ((pm >> e) & 1u) dst = gp + (size_t(p & TNP_INDEX) + (e ? pm & 1u : 0u)) * MC;
            else if ((tm >> e) & 1u) dst = gt + (size_t(t & TNP_INDEX) + (e ? tm & 1u : 0u)) * MC;
            if (dst) store_channels(dst, v, wide_out);
        }
        tile_done();
    }
    if (!failed && bc == APR_BC_REFLECT && h.nflag > 0) {
        const int total = prefix_rows(M.list, tid < h.nflag ? image_rows(M.edge[tid]) : 0);
        for (int k0 = 0; k0 < total && !failed; k0 += IMAGE_ROWS) {
            const int k1 = min(k0 + IMAGE_ROWS, total);
            if (tid < TILE) {
                const int k = k0 + tid;
                if (k < k1) {
                    const int i = row_owner(M.list, h.nflag, k);
                    put_image_row(S.rows, tid, i, image_row(M.edge[i], k - M.list.first[i]));
                } else {
                    S.rows.mask[tid] = 0;
                }
            }
            tile_ready();
            failed = tile_gemm<false>(S, 0, gout, gout, wide, D, phase, err);
            if (failed) break;
            // source children through shared memory; one thread per (record, child, four channels) adds the
            // sums of the record's rows in order, then adds them to the child
            if (warp < NWARP && 32 * q < IMAGE_ROWS)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    float v[16];
                    tmem_ld16(D + (uint32_t(32 * q) << 16) + 64 * a + 16 * c, v);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        *image_chunk(M, 32 * q + lane, 16 * a + 4 * c + k) = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
                }
            block_sync();
            const int i0 = row_owner(M.list, h.nflag, k0), i1 = row_owner(M.list, h.nflag, k1 - 1);
            for (int w = tid; w < (i1 - i0 + 1) * 32; w += TNT) {
                const int i = i0 + (w >> 5), ch = w & 3;
                const unsigned to = (w >> 2) & 7, edge = M.edge[i], miss = missing_children(edge);
                const unsigned p = unsigned(reinterpret_cast<const int *>(S.children + i)[to >> 1]), pm = p >> 30;
                const unsigned t = unsigned(reinterpret_cast<const int *>(M.nodes + i)[to >> 1]), tm = t >> 30;
                const int e = int(to & 1u);
                float *dst;
                if ((pm >> e) & 1u) dst = gp + (size_t(p & TNP_INDEX) + (e ? pm & 1u : 0u)) * MC + 4 * ch;
                else if ((tm >> e) & 1u) dst = gt + (size_t(t & TNP_INDEX) + (e ? tm & 1u : 0u)) * MC + 4 * ch;
                else continue;
                float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int k = max(M.list.first[i], k0); k < min(M.list.first[i + 1], k1); ++k) {
                    const int sh = image_row(edge, k - M.list.first[i]);
                    const unsigned mir = (sh >> 4 ? 4u : 0u) | ((sh >> 2) & 3 ? 2u : 0u) | (sh & 3 ? 1u : 0u);
                    unsigned f = 0;   // the child itself, then the missing ones that it stands for
                    do {
                        if (sh != 0 || f != 0) {
                            const float4 v = *image_chunk(M, k - k0, int((to | f) ^ mir) * 4 + ch);
                            s = make_float4(s.x + v.x, s.y + v.y, s.z + v.z, s.w + v.w);
                        }
                        f = (f - miss) & miss;
                    } while (f != 0);
                }
                add4(dst, s);
            }
            tile_done();
        }
    }
    tile_teardown(S);
}

// Data adjoint onto the coarser particles next to nodes: the sums over their eight cells, added to gp
// (after mc_adjoint_kernel). Rows: every record at its own place and, with reflection, at its images.
__global__ void __launch_bounds__(TNT, 2) mc_leaf_adjoint_kernel(const UnitView U, const uint16_t *__restrict__ W, int bc,
                                                                const uint4 *__restrict__ gout, float *__restrict__ gp,
                                                                unsigned *err) {
    extern __shared__ __align__(128) unsigned char smraw[];
    McLeafSmem &M = *reinterpret_cast<McLeafSmem *>(smraw);
    pdl_trigger();
    McSmem &S = M.s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const UnitHdr h = U.lwork[blockIdx.x];
    const bool reflect = bc == APR_BC_REFLECT;
    // thread i keeps record i from its header to the staging
    uint4 q0 = make_uint4(0, 0, 0, 0), q1 = q0;
    if (tid < h.nrec) {
        const uint4 *r = reinterpret_cast<const uint4 *>(U.lrec + h.rec0 + tid);
        q0 = __ldg(r);
        q1 = __ldg(r + 1);
    }
    stage_codes<false>(U, h, true, false, S.code);
    const unsigned edge = q0.z & 0xffffu;
    if (tid < UNIT_RECS) {
        unsigned b[9];
        unpack_bases(q0.z, make_uint2(q0.w, q1.x), make_uint2(q1.y, q1.z), b);
#pragma unroll
        for (int k = 0; k < 9; ++k) S.rows.base[k][tid] = uint16_t(b[k]);
        M.particle[tid] = int(q0.x);
        M.mask[tid] = q0.y;
        M.edge[tid] = uint16_t(edge);
    }
    pdl_wait();   // dL/dout, the weights, and gp of the launch before
    tile_setup<true>(S, W, h.lev);
    const bool wide = (reinterpret_cast<uintptr_t>(gout) & 31u) == 0;
    uint32_t phase = 0;
    const int total = prefix_rows(M.list, tid < h.nrec ? (reflect ? __popcll(edge_shifts<1>(edge)) : 1) : 0);
    for (int k0 = 0; k0 < total; k0 += TILE) {
        if (tid < TILE) {
            const int k = k0 + tid;
            if (k < total) {
                const int i = total == h.nrec ? k : row_owner(M.list, h.nrec, k);
                put_leaf_row(S.rows, tid, i, M.mask[i], reflect ? nth_bit(edge_shifts<1>(M.edge[i]), k - M.list.first[i]) : 0);
                M.skip[tid] = uint8_t(reflect ? 0u : missing_children(M.edge[i]));
            } else {
                S.rows.mask[tid] = 0;
                M.skip[tid] = 0;
            }
        }
        tile_ready();
        const uint32_t D = S.tmem;
        if (tile_gemm<false>(S, 0, gout, gout, wide, D, phase, err)) break;
        if (warp < NWARP) {   // lane = row, half of the cells
            const int q = warp & 3, a = warp >> 2, r = 32 * q + lane;
            float s[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) s[k] = 0.f;
            for (unsigned c = 0; c < 4; ++c) {
                float v[16];
                tmem_ld16(D + (uint32_t(32 * q) << 16) + 64 * a + 16 * c, v);
                if (!((4u * a + c) & M.skip[r]))
#pragma unroll
                    for (int k = 0; k < 16; ++k) s[k] += v[k];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                M.sums[a][r * 4 + (k ^ (r & 3))] = make_float4(s[4 * k], s[4 * k + 1], s[4 * k + 2], s[4 * k + 3]);
        }
        block_sync();
        const int k1 = min(k0 + TILE, total);
        const int i0 = total == h.nrec ? k0 : row_owner(M.list, h.nrec, k0), i1 = total == h.nrec ? k1 - 1 : row_owner(M.list, h.nrec, k1 - 1);
        for (int w = tid; w < (i1 - i0 + 1) * 4; w += TNT) {
            const int i = i0 + (w >> 2), ch = w & 3;
            float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int k = max(M.list.first[i], k0); k < min(M.list.first[i + 1], k1); ++k) {
                const int j = (k - k0) * 4 + (ch ^ ((k - k0) & 3));
                const float4 u = M.sums[0][j], v = M.sums[1][j];
                s = make_float4(s.x + (u.x + v.x), s.y + (u.y + v.y), s.z + (u.z + v.z), s.w + (u.w + v.w));
            }
            add4(gp + size_t(M.particle[i]) * MC + 4 * ch, s);
        }
        tile_done();
    }
    tile_teardown(S);
}

// ---------------------------------------------------------------- weight gradient
// One block per SM takes a contiguous range of the units of the levels that hold particles. Per tile of 128
// records, the four planes iz of cells are gathered one after the other (16 cells, two buffers), and for
// every child row (a, b) the taps tz = iz - a and tx = 0..2 take MMAs over K = the records:
//   D[tx block][tz][(tx, iy, ci)][(e, co)] += U(cell (iz, b + tx, iy))[ci] g(child (a, b, e))[co]
// with M = 128 = two rows of four cells x 16 channels (the second block's second half is not used: it reads
// the next row or past the plane, inside the block's shared memory). The tap along y is iy - e. After
// every tile D is added to FP32 registers (96 per thread), so that the tensor cores' accumulation chains stay
// at 32 MMAs; a level's sums are written to the level's partial of the block and reduced in order.
// Bound by the A operand's reads from shared memory (an MMA of 32 columns reads as much as one of 64) and by the gather's
// issue, in turn. 1 M particles: 126 us with a diverged issuing lane and records, children and gradients fetched per
// tile; converged issue 115, one stream of planes per unit 110, both child planes in one MMA 98 us.
constexpr int WG_SBO = 2048 + 16;           // 8 channels of a cell for 128 records, padded: eight lanes write
                                            // eight pieces of one record without bank conflicts
constexpr int WG_CELL = 2 * WG_SBO;
constexpr int PLANE_BYTES = 16 * WG_CELL;
constexpr uint32_t WG_TMEM = 256;           // D: (tx block, tz) in columns 96 block + 32 (2 - tz), 192 used
constexpr int WG_OUT = NTAP * MC * MC;      // floats of one partial: [tap][ci][co]
struct WgradSmem {
    int code[8][PLANE];
    Rows rows;
    alignas(128) unsigned char A[2][PLANE_BYTES];   // cell-major: (2 cell + h) WG_SBO + (r / 8) 128 + (r % 8) 16
    alignas(128) unsigned char g[8 * WG_CELL];      // the same for the children (b, a, e)
    int4 children[UNIT_RECS];
    uint64_t bar;
    uint32_t tmem;
};

// Cells (iz, .., ..) of records t0 .. t0 + 127 of the unit. Eight lanes per row.
__device__ __forceinline__ void gather_plane(const WgradSmem &S, const uint4 *__restrict__ vals, const uint4 *__restrict__ tree,
                                             int t0, int iz, uint32_t A) {
    const int lane = threadIdx.x & 31, iy = (lane >> 1) & 3, h = lane & 1;
    const uint32_t dst = A + uint32_t((2 * iy + h) * WG_SBO);
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
        const int r = (threadIdx.x >> 5) * 16 + 4 * j + (lane >> 3);
#pragma unroll
        for (int ix = 0; ix < 4; ++ix) {
            const int q = ((iz + 1) >> 1) * 3 + ((ix + 1) >> 1), c0 = ((iz + 1) & 1) * 4 + ((ix + 1) & 1) * 2;
            const int code = S.code[c0 + ((iy + 1) & 1)][S.rows.base[q][t0 + r] + ((iy + 1) >> 1)];
            cp_async16(dst + 4 * ix * WG_CELL + (r >> 3) * 128 + (r & 7) * 16, source_row(vals, tree, code) + h, code != NO_SOURCE);
        }
    }
}
// dL/dout of their children (zero where the child is no particle). Eight lanes per row: child (b, e), half.
__device__ __forceinline__ void gather_gradient(const WgradSmem &S, const uint4 *__restrict__ gout, int t0, uint32_t G) {
    const int lane = threadIdx.x & 31, be = (lane >> 1) & 3, hh = lane & 1;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int r = (threadIdx.x >> 5) * 16 + 4 * j + (lane >> 3);
        const int4 pw = S.children[t0 + r];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const unsigned w = unsigned(be < 2 ? (a ? pw.z : pw.x) : (a ? pw.w : pw.y)), pm = w >> 30;
            const size_t p = (w & TNP_INDEX) + (be & 1 ? pm & 1u : 0u);
            cp_async16(G + uint32_t((2 * (4 * (be >> 1) + 2 * a + (be & 1)) + hh) * WG_SBO + (r >> 3) * 128 + (r & 7) * 16), gout + 2 * p + hh,
                       (pm >> (be & 1)) & 1u);
        }
    }
}

// A tile's sums added to acc (thread: row 32 q + lane of D, columns 96 half ..) without what no target reads. The
// MMAs multiply every cell around a record with the zero that stands for a child that is no particle, so an
// infinity or NaN there is in sums of targets that do not read it. If one of the warp's sums that make up taps
// (iy - e = 0, 1, 2; the second block has one tx) is not finite, they are summed again over the particles alone.
// Taken only in the second pass over a level whose first one left a sum that is not finite: a block that meets none
// pays for the test of what it writes (nothing measurable); 1 M particles, 98 us: one infinite feature 0.5 ms, every
// feature infinite 1.5 ms.
__device__ __forceinline__ void add_live_targets(const WgradSmem &S, const uint4 *vals, const uint4 *tree, int t0, int nrec, uint32_t D,
                                                 float (&acc)[96]) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = warp & 3, half = warp >> 2;
    const int iy = (2 * q + (lane >> 4)) & 3, ci = lane & 15, tx = 2 * half + (q >> 1);
    bool finite = true;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        float v[16];
        tmem_ld16(D + (uint32_t(32 * q) << 16) + 96 * half + 16 * k, v);
        if (tx < 3 && unsigned(iy - (k & 1)) < 3u)
#pragma unroll
            for (int c = 0; c < 16; ++c) finite = finite && isfinite(v[c]);
    }
    if (__all_sync(0xffffffffu, finite)) {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            float v[16];
            tmem_ld16(D + (uint32_t(32 * q) << 16) + 96 * half + 16 * k, v);
#pragma unroll
            for (int c = 0; c < 16; ++c) acc[16 * k + c] += v[c];
        }
        return;
    }
#pragma unroll 1
    for (int r = 0; r < min(TILE, nrec - t0); ++r) {
        const int4 pw = S.children[t0 + r];
        if (unsigned(pw.x | pw.y | pw.z | pw.w) >> 30 == 0) continue;   // no particle among the children
        float x[4][2];   // cells (iz, tx + b, iy)
#pragma unroll
        for (int iz = 0; iz < 4; ++iz)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int ix = tx + b, s = ((iz + 1) >> 1) * 3 + ((ix + 1) >> 1), c0 = ((iz + 1) & 1) * 4 + ((ix + 1) & 1) * 2;
                const int code = S.code[c0 + ((iy + 1) & 1)][S.rows.base[s][t0 + r] + ((iy + 1) >> 1)];
                const float u = load_bf16(reinterpret_cast<const uint16_t *>(source_row(vals, tree, code)) + ci);
                x[iz][b] = code == NO_SOURCE ? 0.f : u;
            }
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int a = c >> 2, b = (c >> 1) & 1, e = c & 1;
            const unsigned w = unsigned(b ? (a ? pw.w : pw.y) : (a ? pw.z : pw.x));
            if (!((w >> (30 + e)) & 1u)) continue;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint4 gq = *reinterpret_cast<const uint4 *>(S.g + (2 * (4 * b + 2 * a + e) + h) * WG_SBO + (r >> 3) * 128 + (r & 7) * 16);
                const unsigned gw[4] = {gq.x, gq.y, gq.z, gq.w};
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float g = __uint_as_float(k & 1 ? gw[k >> 1] & 0xffff0000u : gw[k >> 1] << 16);
#pragma unroll
                    for (int tz = 0; tz < 3; ++tz) {
                        float &s = acc[32 * (2 - tz) + 16 * e + 8 * h + k];
                        s = fmaf(x[tz + a][b], g, s);
                    }
                }
            }
        }
    }
}

__global__ void __launch_bounds__(NT, 1) mc_wgrad_kernel(const UnitView U, const UnitLevels L, const uint4 *__restrict__ vals,
                                                         const uint4 *__restrict__ tree, int bc,
                                                         const uint4 *__restrict__ gout, float *__restrict__ partial,
                                                         unsigned *err) {
    extern __shared__ __align__(128) unsigned char smraw[];
    WgradSmem &S = *reinterpret_cast<WgradSmem *>(smraw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q = warp & 3, half = warp >> 2;
    const int total = L.begin[L.n];
    const int u0 = int(int64_t(blockIdx.x) * total / gridDim.x), u1 = int(int64_t(blockIdx.x + 1) * total / gridDim.x);
    if (tid == 0) mbar_init(&S.bar);
    if (warp == 0) tmem_alloc(smem_u32(&S.tmem), WG_TMEM);
    tile_done();
    const uint32_t D = S.tmem, A = smem_u32(S.A[0]), G = smem_u32(S.g);
    constexpr uint32_t idesc = idesc_bf16(128, 32, true);
    uint32_t phase = 0;
    bool failed = false, live_only = false;   // second pass over a level: add_live_targets
    for (int i = 0; i < L.n && !failed; ++i) {
        const int ua = max(u0, L.begin[i]), ub = min(u1, L.begin[i + 1]);
        if (ua >= ub) continue;
        float acc[96];
#pragma unroll
        for (int k = 0; k < 96; ++k) acc[k] = 0.f;
        for (int u = ua; u < ub && !failed; ++u) {
            const UnitHdr h = U.hdr[L.unit0[i] + u - L.begin[i]];
            NodeRow row;
            row.load(U, h, false);
            stage_codes<true>(U, h, false, bc == APR_BC_REFLECT, S.code);
            row.put(S, h);
            block_sync();
            // planes pl = 4 tile + iz in one stream: two are in flight while one is used, across the unit's tiles
            const int planes = 4 * ((h.nrec + TILE - 1) / TILE);
            gather_gradient(S, gout, 0, G);
            gather_plane(S, vals, tree, 0, 0, A);
            cp_commit();
            gather_plane(S, vals, tree, 0, 1, A + PLANE_BYTES);
            cp_commit();
#pragma unroll 1
            for (int pl = 0; pl < planes; ++pl) {
                const int iz = pl & 3;
                cp_wait<1>();
                fence_async_smem();
                tile_done();
                if (warp == 0) {   // converged: a single diverged lane issues an MMA in 125 cycles
                    const uint32_t el = elect_one();
                    const uint64_t P = sdesc(A + (iz & 1) * PLANE_BYTES, 128, WG_SBO), B = sdesc(G, 128, WG_SBO);
                    // child planes a = 0 (tz = iz) and a = 1 (tz = iz - 1) in one MMA of 64 columns where both exist
                    const bool two = iz == 1 || iz == 2;
                    const uint32_t wide = two ? idesc_bf16(128, 64, true) : idesc, Dt = D + (iz == 3 ? 0 : 32 * (2 - iz));
                    const uint64_t Bt = B + (iz == 3 ? 2 * WG_CELL >> 4 : 0);
#pragma unroll
                    for (int b = 0; b < 2; ++b)
#pragma unroll
                        for (int blk = 0; blk < 2; ++blk)
#pragma unroll
                            for (int ks = 0; ks < TILE / 16; ++ks) {
                                const uint64_t Ak = P + (((b + 2 * blk) * 4 * WG_CELL + ks * 256) >> 4), Bk = Bt + ((4 * b * WG_CELL + ks * 256) >> 4);
                                if (b == 0 && ks == 0) {   // the plane's first products overwrite tz = iz only
                                    mma_ss(Dt + 96 * blk, Ak, Bk, idesc, iz == 3 ? 1u : 0u, el);
                                    if (two) mma_ss(Dt + 96 * blk + 32, Ak, Bk + (2 * WG_CELL >> 4), idesc, 1u, el);
                                } else {
                                    mma_ss(Dt + 96 * blk, Ak, Bk, wide, 1u, el);
                                }
                            }
                    if (el) mma_commit(&S.bar);
                    __syncwarp();
                }
                if (block_wait_mma(&S.bar, phase, err)) {
                    failed = true;
                    break;
                }
                phase ^= 1;
                if (live_only && iz == 3) {
                    tc_fence_after();
                    add_live_targets(S, vals, tree, pl / 4 * TILE, h.nrec, D, acc);
                    tile_done();   // S.g has been read
                }
                if (iz == 3 && pl + 1 < planes) gather_gradient(S, gout, (pl + 1) / 4 * TILE, G);
                cp_commit();   // before the plane after the next one, so that the next one's wait covers it
                if (pl + 2 < planes) gather_plane(S, vals, tree, (pl + 2) / 4 * TILE, (pl + 2) & 3, A + (iz & 1) * PLANE_BYTES);
                cp_commit();
                if (iz < 3 || live_only) continue;
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    float v[16];
                    tmem_ld16(D + (uint32_t(32 * q) << 16) + 96 * half + 16 * k, v);
#pragma unroll
                    for (int c = 0; c < 16; ++c) acc[16 * k + c] += v[c];
                }
                tc_fence_before();   // the next MMAs follow a block barrier
            }
            cp_wait<0>();
            tile_done();
        }
        if (failed) break;
        float *dst = partial + size_t(blockIdx.x + i) * WG_OUT;
        // sums of the level: thread (row 32 q + lane, columns 96 half ..) to shared memory, block by block of
        // 32 columns, then tap (tz, tx, ty), ci, co = its two children e of rows (tx, iy = ty + e, ci)
        float *stage = reinterpret_cast<float *>(S.A[0]);   // [128][33]
        bool finite = true;
#pragma unroll
        for (int blk = 0; blk < 6; ++blk) {                 // (tx block, 2 - tz)
            block_sync();
            if (half == blk / 3)
#pragma unroll
                for (int c = 0; c < 32; ++c) stage[(32 * q + lane) * 33 + c] = acc[32 * (blk % 3) + c];
            block_sync();
            const int ntx = blk / 3 ? 1 : 2;
            for (int o = tid; o < ntx * 3 * MC * MC; o += NT) {
                const int co = o % MC, ci = (o / MC) % MC, ty = (o / (MC * MC)) % 3, txo = o / (3 * MC * MC);
                const float *s = stage + ((txo * 4 + ty) * MC + ci) * 33 + co;
                const int tap = ((2 - blk % 3) * 3 + 2 * (blk / 3) + txo) * 3 + ty;
                const float v = s[0] + s[MC * 33 + 16];   // e = 0: iy = ty; e = 1: iy = ty + 1
                dst[(tap * MC + ci) * MC + co] = v;
                finite = finite && isfinite(v);
            }
        }
        __syncwarp();
        live_only = __syncthreads_or(!finite) != 0 && !live_only;
        if (live_only) --i;   // the level again
    }
    tile_done();
    if (warp == 0) tmem_dealloc(D, WG_TMEM);
}

// grad_weights[lev][co][ci][e] = sum over the level's partials, in a fixed order; zero for a level without particles.
// A chain of up to 152 loads per output is a latency of its own (8 us however small the APR): eight warps take
// every eighth partial of 32 outputs.
constexpr int RED_OUT = 32, RED_WARPS = 8;
static_assert(WG_OUT % RED_OUT == 0, "a block's outputs belong to one level");
__global__ void __launch_bounds__(RED_OUT *RED_WARPS) mc_wgrad_reduce_kernel(const float *__restrict__ partial, const UnitRanges R,
                                                                            float *__restrict__ gw) {
    __shared__ float sums[RED_WARPS][RED_OUT];
    const int lane = threadIdx.x % RED_OUT, w = threadIdx.x / RED_OUT, i = blockIdx.x * RED_OUT + lane;
    const int lev = i / WG_OUT, r = i % WG_OUT;
    float s = 0.f;
#pragma unroll 4
    for (int c = R.first[lev] + w; c <= R.last[lev]; c += RED_WARPS) s += partial[size_t(c) * WG_OUT + r];
    sums[w][lane] = s;
    __syncthreads();
    if (w != 0) return;
#pragma unroll
    for (int k = 1; k < RED_WARPS; ++k) s += sums[k][lane];
    const int co = r % MC, ci = (r / MC) % MC, e = r / (MC * MC);
    gw[((size_t(lev) * MC + co) * MC + ci) * NTAP + e] = s;
}

// The tile kernels' shared memory admits two blocks per SM (228 KB per SM, 1 KB reserved per block), each
// with half of the SM's 512 tensor-memory columns; the weight gradient takes an SM to itself.
// A third block would wait for tensor memory with its SM's other resources in hand (leaf adjoint of 1 M particles: 95
// instead of 76 us): the leaf kernel, whose registers admit three, takes more than a third of the shared memory.
constexpr size_t TWO_BLOCKS = 228 * 1024 / 3;
static_assert(sizeof(McLeafSmem) <= 113 * 1024, "leaf units: two blocks per SM");
static_assert(2 * (sizeof(McAdjSmem) + 1024) <= 228 * 1024, "tile kernels: two blocks per SM");
static_assert(sizeof(WgradSmem) <= 227 * 1024, "weight gradient: one block per SM");
static_assert(offsetof(McSmem, W) % 128 == 0 && offsetof(McSmem, bar) % 8 == 0, "alignment");
static_assert(offsetof(WgradSmem, A) % 128 == 0 && offsetof(WgradSmem, g) % 128 == 0 && offsetof(WgradSmem, bar) % 8 == 0, "alignment");
static_assert(PLANE_BYTES >= 128 * 33 * 4, "sums staged in an A buffer");

// Partials the workspace of the weight gradient holds (without the levels): the blocks are at most as many.
int wgrad_ctas(int n_units) {
    static int sms = 0;
    static std::once_flag once;
    std::call_once(once, [] {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            sms = 152;
    });
    return std::max(1, std::min(n_units, 8 * sms));
}

template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kernel)(KArgs...), int grid, int block, size_t smem, cudaStream_t s, bool pdl, Args &&...args) {
    if (grid <= 0) return cudaSuccess;
    // two tile kernels' blocks on a multiprocessor (tensor memory admits no more), one of the weight gradient. Left to
    // itself the split leaves 28 or 60 KB of L1 cache
    const int blocks = 2 * (smem + 1024) <= 228 * 1024 ? 2 : 1;
    const cudaError_t e = set_max_dynamic_smem(reinterpret_cast<const void *>(kernel), smem, blocks);
    if (e != cudaSuccess) return e;
    return launch_pdl(kernel, dim3(grid), dim3(block), smem, s, pdl, std::forward<Args>(args)...);
}

bool mc_args_ok(int32_t c_in, int32_t c_out, int32_t k) { return c_in == MC && c_out == MC && k == 3; }
bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

}  // namespace

}  // namespace aprk

using namespace aprk;

extern "C" {

apr_status_t apr_selftest_bounded_wait(apr_handle_t h, uint32_t limit_us, apr_stream_t stream) {
    if (!h || h->host_only || limit_us == 0 || limit_us > 2000000u) return APR_ERR_INVALID_ARG;
    bounded_wait_selftest_kernel<<<1, 32, 0, stream>>>(uint64_t(limit_us) * 1000ull, h->d_err);
    return cuda_status(cudaGetLastError());
}

apr_status_t apr_tree_restrict_bf16(apr_handle_t h, const uint16_t *particles, uint16_t *tree, int32_t channels,
                                    apr_stream_t stream) {
    if (!h || h->host_only) return APR_ERR_INVALID_ARG;
    if (channels != MC) return APR_ERR_UNSUPPORTED;
    const HostIndex &X = h->X;
    if ((X.np && !particles) || (X.nt && !tree) || !aligned16(particles) || !aligned16(tree)) return APR_ERR_INVALID_ARG;
    cudaError_t e = cudaSuccess;
    const TreeGroups T = tree_groups(X, X.l_min, X.l_max - 1, 4);
    for (int i = T.n - 1; i >= 0 && e == cudaSuccess; --i) {   // the finest group first
        e = launch_tree_restrict_bf16(h->d_tnplan, T.g[i], particles, tree, stream, true);
    }
    return cuda_status(e);
}

static apr_status_t convolve_mc(apr_handle_t h, const uint16_t *particles, const uint16_t *tree,
                                const uint16_t *weights, int32_t c_in, int32_t c_out, int32_t k, int32_t bc,
                                const McOutput &o, apr_stream_t stream) {
    if (!h || h->host_only) return APR_ERR_INVALID_ARG;
    if (!mc_args_ok(c_in, c_out, k)) return APR_ERR_UNSUPPORTED;
    if (bc != APR_BC_REFLECT && bc != APR_BC_ZERO) return APR_ERR_INVALID_ARG;
    const HostIndex &X = h->X;
    if (!weights || (X.np && !particles) || (X.nt && !tree)) return APR_ERR_INVALID_ARG;
    if (!aligned16(particles) || !aligned16(tree) || !aligned16(o.out) || !aligned16(o.out_bf16)) return APR_ERR_INVALID_ARG;
    return cuda_status(launch(mc_fwd_kernel, h->n_fwd_units, TNT, sizeof(McSmem), stream, true, h->U, reinterpret_cast<const uint4 *>(particles),
                              reinterpret_cast<const uint4 *>(tree), weights, bc, o, h->d_err));
}

apr_status_t apr_convolve_mc(apr_handle_t h, const uint16_t *particles, const uint16_t *tree, const uint16_t *weights,
                             int32_t c_in, int32_t c_out, int32_t k, int32_t bc, float *out, apr_stream_t stream) {
    if (!out && h && h->X.np) return APR_ERR_INVALID_ARG;
    return convolve_mc(h, particles, tree, weights, c_in, c_out, k, bc, McOutput{out, nullptr, nullptr, nullptr, 0.f}, stream);
}

apr_status_t apr_convolve_mc_relu_bf16(apr_handle_t h, const uint16_t *particles, const uint16_t *tree,
                                       const uint16_t *weights, int32_t c_in, int32_t c_out, int32_t k, int32_t bc,
                                       uint16_t *out, apr_stream_t stream) {
    if (!out && h && h->X.np) return APR_ERR_INVALID_ARG;
    return convolve_mc(h, particles, tree, weights, c_in, c_out, k, bc,
                       McOutput{nullptr, reinterpret_cast<uint4 *>(out), nullptr, nullptr, 0.f}, stream);
}

apr_status_t apr_convolve_mc_readout(apr_handle_t h, const uint16_t *particles, const uint16_t *tree, const uint16_t *weights,
                                     int32_t c_in, int32_t c_out, int32_t k, int32_t bc, const float *x, float inv_scale,
                                     float *y, apr_stream_t stream) {
    if ((!x || !y) && h && h->X.np) return APR_ERR_INVALID_ARG;
    return convolve_mc(h, particles, tree, weights, c_in, c_out, k, bc, McOutput{nullptr, nullptr, y, x, inv_scale}, stream);
}

size_t apr_mc_backward_workspace_bytes(apr_handle_t h, int32_t c_in, int32_t c_out, int32_t k) {
    if (!h || !mc_args_ok(c_in, c_out, k)) return 0;
    const int L = h->X.l_max - h->X.l_min + 1;
    const int units = int(h->X.fwd_items.size()) * 4;
    const size_t gt = (size_t(h->X.nt) * MC * sizeof(float) + 255) / 256 * 256;
    return gt + size_t(wgrad_ctas(units) + L) * WG_OUT * sizeof(float);
}

apr_status_t apr_convolve_mc_backward(apr_handle_t h, const uint16_t *particles, const uint16_t *tree,
                                      const uint16_t *weights, int32_t c_in, int32_t c_out, int32_t k, int32_t bc,
                                      const uint16_t *grad_out, float *grad_particles, float *grad_weights,
                                      void *workspace, size_t workspace_bytes, apr_stream_t stream) {
    if (!h || h->host_only) return APR_ERR_INVALID_ARG;
    if (!mc_args_ok(c_in, c_out, k)) return APR_ERR_UNSUPPORTED;
    if (bc != APR_BC_REFLECT && bc != APR_BC_ZERO) return APR_ERR_INVALID_ARG;
    const HostIndex &X = h->X;
    if (!weights || (X.np && !grad_out)) return APR_ERR_INVALID_ARG;
    if (grad_weights && ((X.np && !particles) || (X.nt && !tree))) return APR_ERR_INVALID_ARG;
    if (!aligned16(particles) || !aligned16(tree) || !aligned16(grad_out) || !aligned16(grad_particles) ||
        !aligned16(grad_weights))
        return APR_ERR_INVALID_ARG;
    const size_t need = apr_mc_backward_workspace_bytes(h, c_in, c_out, k);
    if (!workspace || workspace_bytes < need || (reinterpret_cast<uintptr_t>(workspace) & 255)) return APR_ERR_INVALID_ARG;
    const size_t gt_bytes = (size_t(X.nt) * MC * sizeof(float) + 255) / 256 * 256;
    float *gt = static_cast<float *>(workspace);
    float *partial = reinterpret_cast<float *>(static_cast<char *>(workspace) + gt_bytes);
    const int n_levels = X.l_max - X.l_min + 1;
    cudaError_t e = cudaSuccess;
    if (grad_particles) {
        // every particle and tree node is the child of one record, which stores its gradient; only in an
        // index in which some have no record (a layout that was not validated) are the arrays cleared first
        if (!X.complete && X.np) e = cudaMemsetAsync(grad_particles, 0, size_t(X.np) * MC * sizeof(float), stream);
        if (!X.complete && e == cudaSuccess && X.nt) e = cudaMemsetAsync(gt, 0, size_t(X.nt) * MC * sizeof(float), stream);
        if (h->uncovered) uncovered_kernel<<<1, 1, 0, stream>>>(h->d_err);
        const uint4 *g4 = reinterpret_cast<const uint4 *>(grad_out);
        if (e == cudaSuccess)
            e = launch(mc_adjoint_kernel, h->U.n, TNT, sizeof(McAdjSmem), stream, true, h->U, weights, bc, g4, grad_particles, gt, h->d_err);
        if (e == cudaSuccess)
            e = launch(mc_leaf_adjoint_kernel, h->U.nl, TNT, std::max(sizeof(McLeafSmem), TWO_BLOCKS), stream, true, h->U, weights, bc, g4, grad_particles, h->d_err);
        const TreeGroups T = tree_groups(X, X.l_min, X.l_max - 1, 3);
        for (int i = 0; i < T.n && e == cudaSuccess; ++i) {
            e = launch_tree_pushdown16(h->d_tnplan, T.g[i], grad_particles, gt, stream, true);
        }
    }
    if (e == cudaSuccess && grad_weights) {
        UnitLevels L;
        UnitRanges R;
        const int slots = wgrad_ctas(int(X.fwd_items.size()) * 4);
        const int G = unit_levels(h, std::min(slots, (wgrad_ctas(1 << 30) + 7) / 8), L, R);
        if (G > 0)
            e = launch(mc_wgrad_kernel, G, NT, sizeof(WgradSmem), stream, false, h->U, L, reinterpret_cast<const uint4 *>(particles),
                       reinterpret_cast<const uint4 *>(tree), bc, reinterpret_cast<const uint4 *>(grad_out), partial, h->d_err);
        if (e == cudaSuccess) {
            mc_wgrad_reduce_kernel<<<n_levels * (WG_OUT / RED_OUT), RED_OUT * RED_WARPS, 0, stream>>>(partial, R, grad_weights);
            e = cudaGetLastError();
        }
    }
    return cuda_status(e);
}

}  // extern "C"
