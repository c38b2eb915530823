// Internal definitions shared by the host index builder, the C-ABI entry points and the kernels.
#pragma once

#include <cstddef>
#include <cstdint>
#include <mutex>
#include <utility>
#include <vector>

#include <cuda_runtime.h>

#include "apr.h"

namespace aprk {

// y-block of the brick index and of every work item: rows are cut into blocks of BY cells along y,
// and each row stores, per block, the offset of its first element (a finer-grained xz_end).
constexpr int BY = 64;
// (z, x) rows per convolution tile at the tile's own level (APR_TILE_ZX in apr.h).
constexpr int TZ = APR_TILE_ZX;
constexpr int TX = APR_TILE_ZX;
static_assert(BY == APR_BLOCK_Y, "y-block must match apr.h");
constexpr int MAXL = 24;

// Geometry of one level, passed to kernels by value.
struct LevelGeo {
    int32_t dz, dx, dy;  // level grid size
    int32_t nb;          // ceil(dy / BY) blocks per row
    int32_t row0;        // index of the level's first particle row (into row_ptr)
    int32_t off0;        // index of the level's first entry in the particle block-offset array
    int32_t trow0;       // same for the tree (levels < l_max)
    int32_t toff0;
};

// Tile plans: per work item, the non-empty source segments of its staged patch (index range of one
// row's elements) in the kernels' segment order, built once per APR on the host. For each item,
// hdr = {first entry, count}; entries [first, first + count) hold {lo, meta, pre}, pre = the number
// of elements of the item's entries before this one; entry first + count holds the total in pre.
struct PlanHdr {
    int32_t first, count;
};
// Child map of one tree node (built once per APR; one per node, in tree order): for each of the four
// child rows k = (a, b) = (k >> 1, k & 1) of level l+1 over the node, p[k] = index of its first
// particle child there and t[k] = index of its first tree child (bits 0..29), and in bits 30, 31 of
// p[k] (t[k]) whether child cell y = 2 y_node (bit 30) and 2 y_node + 1 (bit 31) is a particle (a
// tree node). A child cell with neither bit lies outside the grid (or, in a sub-domain's partial
// index, outside the sub-domain). The second child of a kind in a row follows the first at index + 1.
struct alignas(16) TreeNodePlan {
    int32_t p[4];
    int32_t t[4];
};
static_assert(sizeof(TreeNodePlan) == 32, "node plans are two 16-byte words");
constexpr uint32_t TNP_INDEX = (1u << 30) - 1u;
struct HostFPlan {
    std::vector<PlanHdr> hdr;
    std::vector<uint2> ent;
};

// Convolution units (built once per APR by build_units, apr_unitplan.cpp): groups of parents ("records")
// with the list of the parents around them ("slots"), see there. All units of a level are consecutive,
// the finest level first.
constexpr int UNIT_RECS = 256;    // most records of a unit
constexpr int UNIT_SLOTS = 1152;  // most slots of a unit
struct alignas(16) UnitHdr {
    int32_t pure0, node0, oth0, rec0;  // first pure, node and other entry, first record
    int16_t npure;                // slots whose eight cells are particles of the level
    int16_t nnode;                // the other slots that are nodes
    int16_t nleaf, noth;          // coarser particles; with the empty slots after them
    int16_t nrec, nflag;          // records; the first nflag lie at the level grid's edges
    int16_t lev, pad;             // l - l_min of the child cells
};
static_assert(sizeof(UnitHdr) == 32, "unit headers are two 16-byte words");
// Pure entry: word k = first particle of child row k (28 bits; the second follows it) | 4 bits of the slot
// number << 28 (bits 4k .. 4k + 3 of it). One 16-byte load gives a slot's eight sources.
// Node entry: the child map of a slot that is not pure (a copy, so that no load depends on an index), and
// its info word. Other entry: x = particle index (coarser particles), y = info word.
// info: slot number (11 bits) | mirror bits << UE_MIRROR | missing bits << UE_MISS, each 3 bits (z 4, x 2,
// y 1). mirror: the slot lies outside the grid along that axis, its children are the source's in
// reversed order; missing: the source's second child along that axis lies outside the grid.
constexpr int UE_MIRROR = 16, UE_MISS = 20;
constexpr unsigned UE_SLOT = 0x7ffu;
// A record: a parent whose children are computed, and the slot of the y - 1 neighbour in each of the
// nine rows (z + dz, x + dx) around it. edge: per axis (z bits 0-2, x 3-5, y 6-8) bit 0 = first parent,
// bits 1-2 = child cells from the parent's first one to the grid's end if at most 3, else 0.
struct alignas(8) NodeRec {
    uint32_t node;
    uint16_t edge;
    uint16_t base[9];
};
static_assert(sizeof(NodeRec) == 24, "node records are three 8-byte words");
// A level-(l-1) particle next to nodes, as a coarse source of level l: mask bit 3r + j = neighbour j of
// row r is a node (a slot); base[r] = slot of the row's first such neighbour.
struct alignas(16) LeafRec {
    uint32_t particle, mask;
    uint16_t edge;
    uint16_t base[9];
    uint32_t pad;
};
static_assert(sizeof(LeafRec) == 32, "leaf records are two 16-byte words");
struct UnitSpan {                          // units [first, last)
    int32_t first, last;
};
// The units that hold records of the work items of a range call, as a span of the units' own order (the finest
// level first, along the curve); others in the span hold none of the range.
class UnitSpans {
  public:
    void set(std::vector<UnitSpan> items);
    UnitSpan of(int64_t first, int64_t n) const;   // of the items [first, first + n)
    const std::vector<UnitSpan> &items() const { return item_; }

  private:
    static constexpr int64_t G = 64;
    std::vector<UnitSpan> item_, group_;   // per work item, per G of them
};
struct UnitPlan {                          // host
    std::vector<UnitHdr> hdr, lhdr;        // node units, leaf units: finest level first, along the curve
    std::vector<UnitHdr> work, work_adj;   // the node units again, longest first: those of the forward pass, then the rest; all
    std::vector<UnitHdr> lwork;            // the leaf units again, longest first
    UnitSpans fwd_units, bwd_units, bwd_leaves;   // of the forward items; of the adjoint items, node and leaf units
    int32_t n_forward = 0;                 // node units of the levels down to the coarsest that holds particles
    std::vector<uint4> pure, lpure;        // entries: pure slots, other nodes, the rest
    std::vector<TreeNodePlan> nmap, lnmap;
    std::vector<uint32_t> ninfo, lninfo;
    std::vector<uint2> oth;
    std::vector<NodeRec> rec;
    std::vector<LeafRec> lrec;
    std::vector<int32_t> tile_f, tile_b, ltile_b;  // work item of each record (-1: none): forward, adjoint
    int32_t level_begin[MAXL + 1] = {};    // first node unit of level l_min + i
    bool complete = false;                 // every particle and tree node is the child of a record
    bool uncovered = false;                // a cell next to a particle has no source (invalid layout)
};
// Blocks of a stencil or weight gradient: a contiguous range of the units of the levels that hold particles
// each (finest level first); block b writes the sums of its i-th level to partial b + i.
struct UnitLevels {
    int n = 0;
    int unit0[MAXL] = {};          // first unit of the level
    int begin[MAXL + 1] = {};      // prefix of the levels' unit counts
};
struct UnitRanges {                // partials of level l_min + i: first[i] .. last[i] (none if first > last)
    int first[MAXL], last[MAXL];
};
struct UnitView {                          // device
    const UnitHdr *hdr, *lhdr, *work, *work_adj, *lwork;
    const uint4 *pure, *lpure;
    const TreeNodePlan *nmap, *lnmap;
    const uint32_t *ninfo, *lninfo;
    const uint2 *oth;
    const NodeRec *rec;
    const LeafRec *lrec;
    const int32_t *tile_f, *tile_b, *ltile_b;
    const TreeNodePlan *nplan;             // child maps: tree nodes, then virtual parents
    int32_t n, nl;                         // node units, leaf units
};

// What the host builders need to walk the index.
struct DevLayout {
    const uint32_t *row_ptr;   // [R+1]
    const uint16_t *y;         // [N_p]
    const uint16_t *off;       // [sum_l rows_l * nb_l]: first element of block j, relative to row start
    const uint32_t *trow_ptr;  // [R_t+1]
    const uint16_t *ty;        // [N_t]
    const uint16_t *toff;
    int32_t np, nt;            // particles, tree nodes (value array lengths)
    int32_t l_min, l_max;
    LevelGeo geo[MAXL];
};

struct Item {  // a work item: level, tile (or row) coordinates, y block
    int32_t l, a, b, yb;
};

// Host-side index, built by build_index(); uploaded by apr_build_device.
struct HostIndex {
    int32_t l_min = 0, l_max = 0;
    int64_t dims[3] = {0, 0, 0};
    LevelGeo geo[MAXL] = {};
    int64_t np = 0, nt = 0, R = 0, Rt = 0, noff = 0, ntoff = 0;
    std::vector<uint32_t> row_ptr, trow_ptr;
    std::vector<uint16_t> y, ty, off, toff;
    std::vector<Item> fwd_items;              // non-empty (l, tz, tx, yb) tiles, by level
    std::vector<Item> bwd_items;              // tiles whose interior cells receive gradient
    std::vector<Item> tree_items;             // non-empty (l, z, x, yb) tree bricks, by level
    int64_t fwd_level_begin[MAXL + 1] = {};   // fwd_items of level l: [begin[l], begin[l+1])
    int64_t bwd_level_begin[MAXL + 1] = {};   // bwd_items of level l: [begin[l], begin[l+1])
    int64_t tree_level_begin[MAXL + 1] = {};
    HostFPlan fplan[2];                       // forward tile plans (build_plans), radius 1 and 2
    HostFPlan bplan[2];                       // data-adjoint tile plans (build_plans), radius 1 and 2
    std::vector<TreeNodePlan> tnplan;         // child maps of the tree nodes (tree_node_plan)
    std::vector<uint32_t> vrow_ptr;           // virtual parents of the cells of l_min: rows, y, child maps
    std::vector<uint16_t> vy;
    std::vector<TreeNodePlan> vplan;
    UnitPlan units;                           // convolution units (build_units)
    bool complete = false;                    // every particle and tree node is the child of a record (kept from units)
};

// The tree nodes of level l (l_min <= l < l_max): [b, b + n) in tree order.
inline void tree_level_nodes(const HostIndex &X, int l, int64_t &b, int64_t &n) {
    const LevelGeo &g = X.geo[l];
    b = X.trow_ptr[size_t(g.trow0)];
    n = int64_t(X.trow_ptr[size_t(g.trow0) + size_t(g.dz) * size_t(g.dx)]) - b;
}

// Consecutive tree levels taken by one launch (apr_kernels.cu): `levels` of them from the coarsest one,
// whose nodes are [node0, node0 + n).
struct TreeGroup {
    int32_t node0, n, levels;
};
// The groups of the tree levels [l0, l1] (within [l_min, l_max - 1]), coarsest first: each takes as many
// levels (at most max_levels) as keep its deepest level at or below tree_group_threads entries.
// 2^17 entries are less than half of what is resident at once; with 2^20 a group's idle threads cost more than
// the launches it saves (16-channel restriction of 1 M particles 28 -> 50 us, push-down of 8 M 45 -> 84 us at 2^22).
// A group finds the nodes of its finer levels from their parents; where a cell is a particle and a node at once (a
// layout that was not validated) the node is no parent's child, so that every level is a group of its own.
constexpr int64_t tree_group_threads = int64_t(1) << 17;
struct TreeGroups {
    int n = 0;
    TreeGroup g[MAXL];
};
TreeGroups tree_groups(const HostIndex &X, int l0, int l1, int max_levels);

// Builds and validates the index from the host layout. Returns APR_OK or an error code; `msg`
// receives a short reason on failure.
apr_status_t build_index(const apr_host_layout &L, uint32_t flags, HostIndex &out, const char **msg);

// Builds what the kernels read on a device of `sms` multiprocessors (apr_plan.cu): the child maps and the units. Returns APR_OK, APR_ERR_OOM (host allocation) or APR_ERR_UNSUPPORTED.
apr_status_t build_plans(HostIndex &X, int sms);
// Builds the tile plans of X's forward and data-adjoint work items (apr_export_structure).
apr_status_t build_tile_plans(HostIndex &X);
// The convolution units of X (after tree_node_plan) for a device of `sms` multiprocessors; throws std::bad_alloc.
void build_units(HostIndex &X, int sms);
constexpr int HOST_ONLY_SMS = 152;   // the units of a host-only handle are a GB300's
// The child map of every tree node (TreeNodePlan), by one merge of each tree row with its child rows.
// In a complete index every in-grid child cell of a node is a particle or a node of the next level.
bool tree_node_plan(const DevLayout &L, const HostIndex &X, std::vector<TreeNodePlan> &P);
// apr_convolve_backward; concurrent: the stencil gradient on the handle's second stream
apr_status_t convolve_backward(apr_handle_t h, const float *particles, const float *tree, const float *stencils,
                               int32_t k, int32_t bc, const float *grad_out, float *grad_particles,
                               float *grad_stencils, void *workspace, size_t workspace_bytes, apr_stream_t stream,
                               bool concurrent);
// The levels, the ranges and the number of blocks (at most max_blocks; 0 without particles).
int unit_levels(apr_handle_t h, int max_blocks, UnitLevels &L, UnitRanges &R);
// DevLayout over X's index.
DevLayout host_layout_view(const HostIndex &X);

// Record a short reason for the last failure on this thread (read by apr_last_error_message).
void set_last_message(const char *msg);

// Epilogues of the convolution kernel (launch_conv_fwd)
constexpr int EPI_PLAIN = 0, EPI_DIVIDE = 1, EPI_MULTIPLY = 2;

// Bits of the device error word, read and cleared by apr_sync_status.
constexpr unsigned ERR_DEVICE_CHECK = 1u;  // a device-side consistency check failed
constexpr unsigned ERR_TIMEOUT = 2u;       // a bounded wait (tensor-core completion) gave up

// Map a CUDA error to a status code, recording its message for apr_last_error_message.
apr_status_t cuda_status(cudaError_t e);

// Raise a kernel's dynamic shared-memory limit to `bytes` on the current device, once per (kernel,
// device): later calls make no CUDA call, so launches can be captured into CUDA graphs. blocks > 0: that many
// are to be resident on a multiprocessor, and what their shared memory leaves goes to the L1 cache.
cudaError_t set_max_dynamic_smem(const void *fn, size_t bytes, int blocks = 0);

// kernel<<<grid, block, smem, s>>>(args...), with programmatic stream serialization when `pdl`: the
// kernel may then start while the kernel before it on s finishes, and waits for it with pdl_wait
// (apr_device.cuh) before it reads what that kernel writes.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool pdl,
                       Args &&...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

inline int64_t level_cells(int64_t D, int l_max, int l) {
    int64_t s = int64_t(1) << (l_max - l);
    return (D + s - 1) / s;
}

}  // namespace aprk

// The object behind apr_handle_t: the host index and its device copy.
struct apr_handle_s {
    aprk::HostIndex X;
    bool host_only = false;
    unsigned *d_err = nullptr;
    apr_stream_t stream = nullptr;                      // the build stream (uploads, stream-ordered allocation)
    apr_allocator alloc{};                              // the caller's allocator, if has_alloc
    bool has_alloc = false;
    std::vector<std::pair<void *, size_t>> blocks;      // every device block of the handle
    aprk::TreeNodePlan *d_tnplan = nullptr;
    // host-only handles: tile plans built on the first apr_export_structure request for them
    std::mutex plan_mu;
    bool host_plans = false, host_units = false;
    aprk::UnitView U{};   // convolution units; those of the levels down to the coarsest one with particles
    int n_fwd_units = 0;
    aprk::UnitSpans fwd_units, bwd_units, bwd_leaves;   // UnitPlan
    int32_t unit_begin[aprk::MAXL + 1] = {};   // first unit of level l_min + i
    bool level_has[aprk::MAXL + 1] = {};       // whether level l_min + i holds particles
    bool uncovered = false;                    // a cell next to a particle has no source (invalid layout)
    int n_levels_with = 0, sms = 0;            // levels with particles; multiprocessors of the device
    size_t dev_bytes = 0;
    // apr_convolve_backward runs the stencil gradient on a second stream, forked from and joined back
    // to the caller's stream with these events (created on first use; side_mu orders the enqueues)
    cudaStream_t side = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    std::mutex side_mu;
};
