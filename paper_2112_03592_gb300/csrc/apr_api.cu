// C ABI entry points (include/apr.h): handle lifetime, upload of the index, kernel launches.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "apr_internal.h"

namespace aprk {
cudaError_t launch_tree_restrict(const TreeNodePlan *np, const TreeGroup &g, const float *vals, float *tree, cudaStream_t s,
                                 int C, int ch, bool pdl);
cudaError_t launch_tree_pushdown(const TreeNodePlan *np, const TreeGroup &g, float *gp, float *gt, cudaStream_t s, bool pdl);
// apr_units.cu
cudaError_t launch_conv_fwd(int k, const UnitView &U, int n_units, const float *vals, const float *tree, const float *st,
                            int bc, float *out, cudaStream_t s, int epi_mode = EPI_PLAIN, bool flip = false,
                            const float *aux = nullptr, const UnitSpan &span = UnitSpan{0, 0}, int first_tile = 0,
                            int n_tiles = -1);
cudaError_t launch_gradmag(int k, const UnitView &U, int n_units, const float *vals, const float *tree, const float *st,
                           int n_levels, int bc, float *out, cudaStream_t s);
cudaError_t launch_adjoint(int k, const UnitView &U, const float *st, int bc, const float *gout, float *gp, float *gt,
                           cudaStream_t s, const UnitSpan &nodes = UnitSpan{0, 0}, const UnitSpan &leaves = UnitSpan{0, 0},
                           int first_tile = 0, int n_tiles = -1);
int stencil_grad_blocks(int k);   // blocks of it that are resident on a multiprocessor
cudaError_t launch_stencil_grad(int k, const UnitView &U, const UnitLevels &W, const UnitRanges &R, int blocks, int n_levels,
                                const float *vals, const float *tree, int bc, const float *gout, float *partial, int stride,
                                float *gw, cudaStream_t s);
}  // namespace aprk

using namespace aprk;

namespace {

thread_local char g_last_msg[256] = "";

// One device block of the handle: from the caller's allocator when one was given, else
// stream-ordered (cudaMallocAsync on the build stream). Every block is recorded for apr_destroy.
cudaError_t dev_alloc(apr_handle_s *h, void **p, size_t bytes) {
    *p = nullptr;
    if (h->has_alloc) {
        *p = h->alloc.alloc(bytes, h->stream, h->alloc.ctx);
        if (!*p) return cudaErrorMemoryAllocation;
        if (reinterpret_cast<uintptr_t>(*p) % 16 != 0) {  // the kernels read the index with 16-byte loads
            h->alloc.free(*p, bytes, h->stream, h->alloc.ctx);
            *p = nullptr;
            return cudaErrorMisalignedAddress;
        }
    } else {
        const cudaError_t e = cudaMallocAsync(p, bytes, reinterpret_cast<cudaStream_t>(h->stream));
        if (e != cudaSuccess) return e;
    }
    h->blocks.emplace_back(*p, bytes);
    h->dev_bytes += bytes;
    return cudaSuccess;
}

// Device copy of n elements on the build stream (an empty array gets one element's space, so that its pointer is one).
// The host arrays are pageable, so cudaMemcpyAsync has staged them when it returns; the caller may free them.
template <typename T>
cudaError_t upload(apr_handle_s *h, T **dst, const T *src, size_t n) {
    *dst = nullptr;
    void *p = nullptr;
    cudaError_t e = dev_alloc(h, &p, std::max<size_t>(n, 1) * sizeof(T));
    if (e != cudaSuccess) return e;
    *dst = static_cast<T *>(p);
    if (n) e = cudaMemcpyAsync(*dst, src, n * sizeof(T), cudaMemcpyHostToDevice, reinterpret_cast<cudaStream_t>(h->stream));
    return e;
}

// The value arrays of the forward-type calls (particles and tree values) must be 16-byte aligned. The multi-channel
// kernels load 16 and 32 bytes; the single-channel ones load single floats, and for them the rule stands as
// part of the interface, which has always refused other addresses.
bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Releases every device block of the handle (the caller has synchronised the device).
void free_device(apr_handle_s *h) {
    for (const auto &b : h->blocks) {
        if (h->has_alloc) h->alloc.free(b.first, b.second, h->stream, h->alloc.ctx);
        else cudaFree(b.first);
    }
    h->blocks.clear();
}

bool stencil_k_ok(int32_t k) { return k == 3 || k == 5; }

// The paper's forward pipeline (Sec. 5.2): the tree restriction of `vals` into `tree`, then the
// convolution over every particle (with the Richardson-Lucy epilogues).
apr_status_t restrict_then_conv(apr_handle_t h, int k, const float *vals, float *tree, const float *st, int bc,
                                float *out, cudaStream_t s, int epi_mode = EPI_PLAIN, bool flip = false,
                                const float *aux = nullptr) {
    const apr_status_t r = apr_tree_restrict(h, vals, tree, 1, s);
    if (r != APR_OK) return r;
    return cuda_status(launch_conv_fwd(k, h->U, h->n_fwd_units, vals, tree, st, bc, out, s, epi_mode, flip, aux));
}

// The tree push-down (apr_tree_restrict_adjoint) of the tree levels [l0, l1] within [l_min, l_max - 1],
// coarsest first.
apr_status_t pushdown_levels(apr_handle_t h, float *grad_tree, float *grad_particles, int l0, int l1,
                             cudaStream_t s) {
    const HostIndex &X = h->X;
    if ((X.nt && !grad_tree) || (X.np && !grad_particles)) return APR_ERR_INVALID_ARG;
    if (l0 < X.l_min) l0 = X.l_min;
    if (l1 > X.l_max - 1) l1 = X.l_max - 1;
    cudaError_t e = cudaSuccess;
    const TreeGroups T = tree_groups(X, l0, l1, 4);
    for (int i = 0; i < T.n && e == cudaSuccess; ++i) {
        e = launch_tree_pushdown(h->d_tnplan, T.g[i], grad_particles, grad_tree, s, true);
    }
    return cuda_status(e);
}

apr_status_t misaligned() {
    aprk::set_last_message("staged value arrays (particles, tree values) must be 16-byte aligned");
    return APR_ERR_INVALID_ARG;
}

}  // namespace

namespace aprk {
TreeGroups tree_groups(const HostIndex &X, int l0, int l1, int max_levels) {
    TreeGroups out;
    if (!X.complete) max_levels = 1;
    for (int l = l0; l <= l1;) {
        int64_t b = 0, n = 0;
        tree_level_nodes(X, l, b, n);
        int g = 1;
        while (g < max_levels && l + g <= l1 && (n << (3 * g)) <= tree_group_threads) ++g;
        if (n > 0) out.g[out.n++] = TreeGroup{int32_t(b), int32_t(n), g};
        l += g;
    }
    return out;
}

int unit_levels(apr_handle_t h, int max_blocks, UnitLevels &L, UnitRanges &R) {
    const int n_levels = h->X.l_max - h->X.l_min + 1;
    L = UnitLevels{};
    int lev[MAXL];
    for (int i = n_levels - 1; i >= 0; --i) {
        R.first[i] = 0;
        R.last[i] = -1;
        const int end = i == 0 ? h->U.n : h->unit_begin[i - 1];
        if (!h->level_has[i] || end <= h->unit_begin[i]) continue;
        lev[L.n] = i;
        L.unit0[L.n] = h->unit_begin[i];
        L.begin[L.n + 1] = L.begin[L.n] + end - h->unit_begin[i];
        ++L.n;
    }
    const int total = L.begin[L.n];
    if (total == 0) return 0;
    const int G = std::max(1, std::min(total, max_blocks));
    auto block_of = [&](int u) {   // block b with b total / G <= u < (b + 1) total / G
        int b = int(int64_t(u) * G / total);
        while (b + 1 < G && int64_t(b + 1) * total / G <= u) ++b;
        while (b > 0 && int64_t(b) * total / G > u) --b;
        return b;
    };
    for (int i = 0; i < L.n; ++i) {
        R.first[lev[i]] = block_of(L.begin[i]) + i;
        R.last[lev[i]] = block_of(L.begin[i + 1] - 1) + i;
    }
    return G;
}

void set_last_message(const char *msg) { snprintf(g_last_msg, sizeof(g_last_msg), "%s", msg); }

cudaError_t set_max_dynamic_smem(const void *fn, size_t bytes, int blocks) {
    static std::mutex mu;
    static std::vector<std::pair<const void *, int>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    for (const auto &d : done)
        if (d.first == fn && d.second == dev) return cudaSuccess;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes));
    if (e == cudaSuccess && blocks > 0) {
        const size_t want = blocks * (bytes + 1024), sm = 228 * 1024;   // 1 KB of every block is reserved
        e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, int(std::min<size_t>(100, (100 * want + sm - 1) / sm)));
    }
    if (e == cudaSuccess) done.emplace_back(fn, dev);
    return e;
}

apr_status_t cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return APR_OK;
    if (e == cudaErrorMemoryAllocation) return APR_ERR_OOM;
    snprintf(g_last_msg, sizeof(g_last_msg), "%s", cudaGetErrorString(e));
    return APR_ERR_CUDA;
}
}  // namespace aprk

extern "C" {

const char *apr_status_string(apr_status_t s) {
    switch (s) {
        case APR_OK: return "ok";
        case APR_ERR_INVALID_ARG: return "invalid argument";
        case APR_ERR_INVALID_LAYOUT: return "invalid APR layout";
        case APR_ERR_UNSUPPORTED: return "unsupported";
        case APR_ERR_OOM: return "out of memory";
        case APR_ERR_CUDA: return "CUDA error";
        case APR_ERR_TIMEOUT: return "device wait timed out";
        case APR_ERR_DEVICE: return "device-side check failed";
    }
    return "unknown status";
}

// Reason of the last failure on this thread (build errors, CUDA messages); not part of apr.h.
const char *apr_last_error_message(void) { return g_last_msg; }

apr_status_t apr_build_device(const apr_host_layout *layout, uint32_t flags, apr_stream_t stream, apr_handle_t *out) {
    return apr_build_device_ex(layout, flags, stream, nullptr, out);
}

apr_status_t apr_build_device_ex(const apr_host_layout *layout, uint32_t flags, apr_stream_t stream,
                                 const apr_allocator *allocator, apr_handle_t *out) {
    if (!out) return APR_ERR_INVALID_ARG;
    *out = nullptr;
    if (!layout || (flags & ~(APR_VALIDATE | APR_REQUIRE_BALANCE | APR_HOST_ONLY | APR_SUBDOMAIN))) return APR_ERR_INVALID_ARG;
    if (allocator && (!allocator->alloc || !allocator->free)) return APR_ERR_INVALID_ARG;
    apr_handle_s *h = new (std::nothrow) apr_handle_s();
    if (!h) return APR_ERR_OOM;
    h->stream = stream;
    if (allocator) {
        h->alloc = *allocator;
        h->has_alloc = true;
    }
    const char *msg = "";
    apr_status_t st;
    try {
        st = build_index(*layout, flags, h->X, &msg);
    } catch (const std::bad_alloc &) {
        st = APR_ERR_OOM;
        msg = "host allocation failed";
    }
    if (st != APR_OK) {
        snprintf(g_last_msg, sizeof(g_last_msg), "%s", msg);
        delete h;
        return st;
    }
    h->host_only = (flags & APR_HOST_ONLY) != 0;
    if (h->host_only) {
        // the tree-node child maps, for apr_export_structure (a device handle builds them with its plans)
        try {
            tree_node_plan(host_layout_view(h->X), h->X, h->X.tnplan);
        } catch (const std::bad_alloc &) {
            snprintf(g_last_msg, sizeof(g_last_msg), "%s", "host allocation failed (tree-node child maps)");
            delete h;
            return APR_ERR_OOM;
        }
    }
    if (!h->host_only) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) {
            delete h;
            return cuda_status(e);
        }
        const apr_status_t pst = build_plans(h->X, h->sms);
        if (pst != APR_OK) {
            snprintf(g_last_msg, sizeof(g_last_msg), "%s", pst == APR_ERR_OOM ? "host allocation failed (units)"
                                                                                : "more than 2^28 particles or tree nodes");
            delete h;
            return pst;
        }
        const HostIndex &X = h->X;
        // child maps: the tree nodes, then the virtual parents of the cells of l_min
        {
            void *p = nullptr;
            const size_t nb = X.tnplan.size() * sizeof(TreeNodePlan), vb = X.vplan.size() * sizeof(TreeNodePlan);
            e = dev_alloc(h, &p, std::max<size_t>(nb + vb, sizeof(TreeNodePlan)));
            h->d_tnplan = static_cast<TreeNodePlan *>(p);
            const cudaStream_t cs = reinterpret_cast<cudaStream_t>(stream);
            if (e == cudaSuccess && nb) e = cudaMemcpyAsync(p, X.tnplan.data(), nb, cudaMemcpyHostToDevice, cs);
            if (e == cudaSuccess && vb)
                e = cudaMemcpyAsync(static_cast<char *>(p) + nb, X.vplan.data(), vb, cudaMemcpyHostToDevice, cs);
        }
        const UnitPlan &UP = X.units;
        UnitHdr *d_hdr = nullptr, *d_lhdr = nullptr, *d_work = nullptr, *d_adj = nullptr, *d_lwork = nullptr;
        uint4 *d_pure = nullptr, *d_lpure = nullptr;
        TreeNodePlan *d_nmap = nullptr, *d_lnmap = nullptr;
        uint32_t *d_ninfo = nullptr, *d_lninfo = nullptr;
        uint2 *d_oth = nullptr;
        NodeRec *d_rec = nullptr;
        LeafRec *d_lrec = nullptr;
        int32_t *d_tf = nullptr, *d_tb = nullptr, *d_ltb = nullptr;
        if (e == cudaSuccess) e = upload(h, &d_hdr, UP.hdr.data(), UP.hdr.size());
        if (e == cudaSuccess) e = upload(h, &d_lhdr, UP.lhdr.data(), UP.lhdr.size());
        if (e == cudaSuccess) e = upload(h, &d_work, UP.work.data(), UP.work.size());
        if (e == cudaSuccess) e = upload(h, &d_adj, UP.work_adj.data(), UP.work_adj.size());
        if (e == cudaSuccess) e = upload(h, &d_lwork, UP.lwork.data(), UP.lwork.size());
        if (e == cudaSuccess) e = upload(h, &d_pure, UP.pure.data(), UP.pure.size());
        if (e == cudaSuccess) e = upload(h, &d_lpure, UP.lpure.data(), UP.lpure.size());
        if (e == cudaSuccess) e = upload(h, &d_nmap, UP.nmap.data(), UP.nmap.size());
        if (e == cudaSuccess) e = upload(h, &d_lnmap, UP.lnmap.data(), UP.lnmap.size());
        if (e == cudaSuccess) e = upload(h, &d_ninfo, UP.ninfo.data(), UP.ninfo.size());
        if (e == cudaSuccess) e = upload(h, &d_lninfo, UP.lninfo.data(), UP.lninfo.size());
        if (e == cudaSuccess) e = upload(h, &d_oth, UP.oth.data(), UP.oth.size());
        if (e == cudaSuccess) e = upload(h, &d_rec, UP.rec.data(), UP.rec.size());
        if (e == cudaSuccess) e = upload(h, &d_lrec, UP.lrec.data(), UP.lrec.size());
        if (e == cudaSuccess) e = upload(h, &d_tf, UP.tile_f.data(), UP.tile_f.size());
        if (e == cudaSuccess) e = upload(h, &d_tb, UP.tile_b.data(), UP.tile_b.size());
        if (e == cudaSuccess) e = upload(h, &d_ltb, UP.ltile_b.data(), UP.ltile_b.size());
        h->U = UnitView{d_hdr, d_lhdr, d_work, d_adj, d_lwork, d_pure, d_lpure, d_nmap, d_lnmap, d_ninfo, d_lninfo, d_oth, d_rec, d_lrec, d_tf, d_tb, d_ltb, h->d_tnplan,
                        int32_t(UP.hdr.size()), int32_t(UP.lhdr.size())};
        h->n_fwd_units = UP.n_forward;
        for (int i = X.l_max - X.l_min; i >= 0; --i) {   // finest first
            const int l = X.l_min + i;
            h->level_has[i] = X.fwd_level_begin[l + 1] > X.fwd_level_begin[l];
            h->unit_begin[i] = UP.level_begin[i];
        }
        h->X.complete = UP.complete;
        h->uncovered = UP.uncovered;
        h->n_levels_with = 0;
        for (int i = 0; i <= X.l_max - X.l_min; ++i) h->n_levels_with += h->level_has[i] ? 1 : 0;
        if (e == cudaSuccess) {
            void *p = nullptr;
            e = dev_alloc(h, &p, sizeof(unsigned));
            h->d_err = static_cast<unsigned *>(p);
            if (e == cudaSuccess) e = cudaMemsetAsync(h->d_err, 0, sizeof(unsigned), reinterpret_cast<cudaStream_t>(stream));
        }
        if (e != cudaSuccess) {
            st = cuda_status(e);
            cudaStreamSynchronize(reinterpret_cast<cudaStream_t>(stream));
            free_device(h);
            delete h;
            return st;
        }
        h->fwd_units = std::move(h->X.units.fwd_units);
        h->bwd_units = std::move(h->X.units.bwd_units);
        h->bwd_leaves = std::move(h->X.units.bwd_leaves);
        // the plans live on the device now; the host copies are not needed again
        h->X.tnplan = std::vector<TreeNodePlan>{};
        h->X.vplan = std::vector<TreeNodePlan>{};
        h->X.vrow_ptr = std::vector<uint32_t>{};
        h->X.vy = std::vector<uint16_t>{};
        h->X.units = UnitPlan{};
        // the second stream of apr_convolve_backward and its events are made here, so that no later call
        // creates them inside a stream capture
        e = cudaStreamCreateWithFlags(&h->side, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->ev_join, cudaEventDisableTiming);
        if (e != cudaSuccess) {
            st = cuda_status(e);
            apr_destroy(h);
            return st;
        }
    }
    *out = h;
    return APR_OK;
}

apr_status_t apr_destroy(apr_handle_t h) {
    if (!h) return APR_OK;
    if (!h->host_only) {
        cudaDeviceSynchronize();
        free_device(h);
        if (h->ev_fork) cudaEventDestroy(h->ev_fork);
        if (h->ev_join) cudaEventDestroy(h->ev_join);
        if (h->side) cudaStreamDestroy(h->side);
    }
    delete h;
    return APR_OK;
}

int64_t apr_num_particles(apr_handle_t h) { return h ? h->X.np : -1; }
int64_t apr_num_tree(apr_handle_t h) { return h ? h->X.nt : -1; }

apr_status_t apr_level_range(apr_handle_t h, int32_t *l_min, int32_t *l_max) {
    if (!h || !l_min || !l_max) return APR_ERR_INVALID_ARG;
    *l_min = h->X.l_min;
    *l_max = h->X.l_max;
    return APR_OK;
}

size_t apr_layout_bytes(apr_handle_t h) { return h ? h->dev_bytes : 0; }

namespace {
// The tile plans of a host-only handle (built once, on request); nullptr for a device handle, whose
// plans live only on the device.
const HostFPlan *host_plan(apr_handle_t h, int32_t which) {
    if (!h->host_only || which < APR_STRUCT_FWD_PLAN_R1 || which > APR_STRUCT_BWD_PLAN_R2) return nullptr;
    std::lock_guard<std::mutex> lk(h->plan_mu);
    if (!h->host_plans) {
        if (build_tile_plans(h->X) != APR_OK) return nullptr;
        h->host_plans = true;
    }
    const int i = which - APR_STRUCT_FWD_PLAN_R1;
    return i < 2 ? &h->X.fplan[i] : &h->X.bplan[i - 2];
}

// One array of the convolution units of a host-only handle (built once, on request).
bool host_unit_array(apr_handle_t h, int32_t which, const void **src, size_t *bytes) {
    *src = nullptr;
    *bytes = 0;
    if (!h->host_only) return true;
    {
        std::lock_guard<std::mutex> lk(h->plan_mu);
        if (!h->host_units) {
            try {
                build_units(h->X, HOST_ONLY_SMS);
            } catch (const std::bad_alloc &) {
                return false;
            }
            h->host_units = true;
        }
    }
    const UnitPlan &U = h->X.units;
    auto give = [&](const auto &v) {
        *src = v.data();
        *bytes = v.size() * sizeof(v[0]);
    };
    switch (which) {
        case APR_STRUCT_UNIT_HDR: give(U.hdr); break;
        case APR_STRUCT_UNIT_OTHER: give(U.oth); break;
        case APR_STRUCT_UNIT_REC: give(U.rec); break;
        case APR_STRUCT_UNIT_MAP: give(h->X.vplan); break;
        case APR_STRUCT_LEAF_HDR: give(U.lhdr); break;
        case APR_STRUCT_LEAF_REC: give(U.lrec); break;
        case APR_STRUCT_UNIT_PURE: give(U.pure); break;
        case APR_STRUCT_LEAF_PURE: give(U.lpure); break;
        case APR_STRUCT_UNIT_NODE: give(U.nmap); break;
        case APR_STRUCT_LEAF_NODE: give(U.lnmap); break;
        case APR_STRUCT_UNIT_NODE_INFO: give(U.ninfo); break;
        case APR_STRUCT_LEAF_NODE_INFO: give(U.lninfo); break;
        case APR_STRUCT_FWD_UNIT_SPANS: give(U.fwd_units.items()); break;
        case APR_STRUCT_BWD_UNIT_SPANS: give(U.bwd_units.items()); break;
        case APR_STRUCT_BWD_LEAF_SPANS: give(U.bwd_leaves.items()); break;
    }
    return true;
}
}  // namespace

size_t apr_structure_bytes(apr_handle_t h, int32_t which) {
    if (!h) return 0;
    const HostIndex &X = h->X;
    if (which >= APR_STRUCT_UNIT_HDR && which <= APR_STRUCT_BWD_LEAF_SPANS) {
        const void *src;
        size_t n;
        return host_unit_array(h, which, &src, &n) ? n : 0;
    }
    if (which >= APR_STRUCT_FWD_PLAN_R1 && which <= APR_STRUCT_BWD_PLAN_R2) {
        const HostFPlan *P = host_plan(h, which);
        return P ? (P->hdr.size() + P->ent.size()) * sizeof(uint2) : 0;
    }
    switch (which) {
        case APR_STRUCT_ROW_PTR: return X.row_ptr.size() * sizeof(uint32_t);
        case APR_STRUCT_Y_IDX: return X.y.size() * sizeof(uint16_t);
        case APR_STRUCT_TREE_ROW_PTR: return X.trow_ptr.size() * sizeof(uint32_t);
        case APR_STRUCT_TREE_Y_IDX: return X.ty.size() * sizeof(uint16_t);
        case APR_STRUCT_FWD_ITEMS: return X.fwd_items.size() * sizeof(Item);
        case APR_STRUCT_TREE_ITEMS: return X.tree_items.size() * sizeof(Item);
        case APR_STRUCT_BWD_ITEMS: return X.bwd_items.size() * sizeof(Item);
        case APR_STRUCT_TREE_NODE_MAP: return size_t(X.nt) * sizeof(TreeNodePlan);
    }
    return 0;
}

apr_status_t apr_export_structure(apr_handle_t h, int32_t which, void *dst, size_t bytes) {
    if (!h || (!dst && bytes)) return APR_ERR_INVALID_ARG;
    const size_t need = apr_structure_bytes(h, which);
    if (which < APR_STRUCT_ROW_PTR || which > APR_STRUCT_BWD_LEAF_SPANS) return APR_ERR_INVALID_ARG;
    if (bytes < need) return APR_ERR_INVALID_ARG;
    if (need == 0) return APR_OK;
    if (which >= APR_STRUCT_UNIT_HDR) {  // host-only handle (need > 0)
        const void *src;
        size_t n;
        if (!host_unit_array(h, which, &src, &n)) return APR_ERR_OOM;
        memcpy(dst, src, n);
        return APR_OK;
    }
    if (which >= APR_STRUCT_FWD_PLAN_R1) {  // host-only handle (need > 0)
        const HostFPlan *P = host_plan(h, which);
        memcpy(dst, P->hdr.data(), P->hdr.size() * sizeof(PlanHdr));
        memcpy(static_cast<char *>(dst) + P->hdr.size() * sizeof(PlanHdr), P->ent.data(), P->ent.size() * sizeof(uint2));
        return APR_OK;
    }
    const HostIndex &X = h->X;
    if (which == APR_STRUCT_TREE_NODE_MAP && !h->host_only) {
        // the device copy is the one the kernels read (uploaded on the build stream)
        cudaError_t e = cudaStreamSynchronize(reinterpret_cast<cudaStream_t>(h->stream));
        if (e == cudaSuccess) e = cudaMemcpy(dst, h->d_tnplan, need, cudaMemcpyDeviceToHost);
        return cuda_status(e);
    }
    const void *src = nullptr;
    switch (which) {
        case APR_STRUCT_ROW_PTR: src = X.row_ptr.data(); break;
        case APR_STRUCT_Y_IDX: src = X.y.data(); break;
        case APR_STRUCT_TREE_ROW_PTR: src = X.trow_ptr.data(); break;
        case APR_STRUCT_TREE_Y_IDX: src = X.ty.data(); break;
        case APR_STRUCT_FWD_ITEMS: src = X.fwd_items.data(); break;
        case APR_STRUCT_TREE_ITEMS: src = X.tree_items.data(); break;
        case APR_STRUCT_TREE_NODE_MAP: src = X.tnplan.data(); break;
        case APR_STRUCT_BWD_ITEMS: src = X.bwd_items.data(); break;
    }
    memcpy(dst, src, need);
    return APR_OK;
}

apr_status_t apr_tree_restrict(apr_handle_t h, const float *particles, float *tree, int32_t channels,
                               apr_stream_t stream) {
    if (!h || h->host_only) return APR_ERR_INVALID_ARG;
    if (channels < 1 || channels > 64) return APR_ERR_INVALID_ARG;
    if ((!particles && h->X.np) || (!tree && h->X.nt)) return APR_ERR_INVALID_ARG;
    const HostIndex &X = h->X;
    const TreeGroups T = tree_groups(X, X.l_min, X.l_max - 1, 4);
    for (int i = T.n - 1; i >= 0; --i) {   // the finest group first
        for (int c = 0; c < channels; ++c) {  // channels-last values: one strided pass per channel
            const cudaError_t e = launch_tree_restrict(h->d_tnplan, T.g[i], particles, tree, stream, channels, c, true);
            if (e != cudaSuccess) return cuda_status(e);
        }
    }
    return APR_OK;
}

apr_status_t apr_convolve(apr_handle_t h, const float *particles, const float *tree, const float *stencils,
                          int32_t k, int32_t bc, float *out, apr_stream_t stream) {
    if (!h || h->host_only) return APR_ERR_INVALID_ARG;
    if (!stencil_k_ok(k)) return APR_ERR_UNSUPPORTED;
    if (bc != APR_BC_REFLECT && bc != APR_BC_ZERO) return APR_ERR_INVALID_ARG;
    if (!stencils || (h->X.np && (!particles || !out)) || (h->X.nt && !tree)) return APR_ERR_INVALID_ARG;
    if (!aligned16(particles) || !aligned16(tree)) return misaligned();
    return cuda_status(launch_conv_fwd(k, h->U, h->n_fwd_units, particles, tree, stencils, bc, out, stream));
}

apr_status_t apr_convolve_tiles(apr_handle_t h, const float *particles, const float *tree, const float *stencils,
                                int32_t k, int32_t bc, float *out, int64_t first_tile, int64_t n_tiles,
                                apr_stream_t stream) {
    if (!h || h->host_only) return APR_ERR_INVALID_ARG;
    if (!stencil_k_ok(k)) return APR_ERR_UNSUPPORTED;
    if (bc != APR_BC_REFLECT && bc != APR_BC_ZERO) return APR_ERR_INVALID_ARG;
    const int64_t nt = int64_t(h->X.fwd_items.size());
    if (first_tile < 0 || n_tiles < 0 || first_tile + n_tiles > nt) return APR_ERR_INVALID_ARG;
    if (!stencils || (h->X.np && (!particles || !out)) || (h->X.nt && !tree)) return APR_ERR_INVALID_ARG;
    if (!aligned16(particles) || !aligned16(tree)) return misaligned();
    return cuda_status(launch_conv_fwd(k, h->U, h->n_fwd_units, particles, tree, stencils, bc, out, stream, EPI_PLAIN, false,
                                       nullptr, h->fwd_units.of(first_tile, n_tiles), int(first_tile), int(n_tiles)));
}

apr_status_t apr_convolve_adjoint_tiles(apr_handle_t h, const float *stencils, int32_t k, int32_t bc,
                                        const float *grad_out, float *grad_particles, float *grad_tree,
                                        int64_t first_tile, int64_t n_tiles, apr_stream_t stream) {
    if (!h || h->host_only) return APR_ERR_INVALID_ARG;
    if (!stencil_k_ok(k)) return APR_ERR_UNSUPPORTED;
    if (bc != APR_BC_REFLECT && bc != APR_BC_ZERO) return APR_ERR_INVALID_ARG;
    const HostIndex &X = h->X;
    const int64_t nt = int64_t(X.bwd_items.size());
    if (first_tile < 0 || n_tiles < 0 || first_tile + n_tiles > nt) return APR_ERR_INVALID_ARG;
    if (!stencils || (X.np && (!grad_out || !grad_particles)) || (X.nt && !grad_tree)) return APR_ERR_INVALID_ARG;
    return cuda_status(launch_adjoint(k, h->U, stencils, bc, grad_out, grad_particles, grad_tree, stream,
                                      h->bwd_units.of(first_tile, n_tiles), h->bwd_leaves.of(first_tile, n_tiles), int(first_tile),
                                      int(n_tiles)));
}

size_t apr_convolve_auto_workspace_bytes(apr_handle_t h) {
    return h ? size_t(h->X.nt > 0 ? h->X.nt : 1) * sizeof(float) : 0;
}

apr_status_t apr_convolve_auto(apr_handle_t h, const float *particles, const float *stencils, int32_t k, int32_t bc,
                               float *out, void *workspace, size_t workspace_bytes, apr_stream_t stream) {
    if (!h || h->host_only) return APR_ERR_INVALID_ARG;
    if (!workspace || workspace_bytes < apr_convolve_auto_workspace_bytes(h) ||
        !aligned16(workspace))
        return APR_ERR_INVALID_ARG;
    if (!stencil_k_ok(k)) return APR_ERR_UNSUPPORTED;
    if (bc != APR_BC_REFLECT && bc != APR_BC_ZERO) return APR_ERR_INVALID_ARG;
    if (!stencils || (h->X.np && (!particles || !out))) return APR_ERR_INVALID_ARG;
    if (!aligned16(particles)) return misaligned();
    return restrict_then_conv(h, k, particles, static_cast<float *>(workspace), stencils, bc, out, stream);
}

apr_status_t apr_gradient_magnitude(apr_handle_t h, const float *particles, const float *tree, const float *stencils,
                                    int32_t k, int32_t bc, float *out, apr_stream_t stream) {
    if (!h || h->host_only) return APR_ERR_INVALID_ARG;
    if (!stencil_k_ok(k)) return APR_ERR_UNSUPPORTED;
    if (bc != APR_BC_REFLECT && bc != APR_BC_ZERO) return APR_ERR_INVALID_ARG;
    if (!stencils || (h->X.np && (!particles || !out)) || (h->X.nt && !tree)) return APR_ERR_INVALID_ARG;
    if (!aligned16(particles) || !aligned16(tree)) return misaligned();
    return cuda_status(launch_gradmag(k, h->U, h->n_fwd_units, particles, tree, stencils, h->X.l_max - h->X.l_min + 1, bc, out,
                                      stream));
}

size_t apr_backward_workspace_bytes(apr_handle_t h, int32_t k) {
    if (!h || !stencil_k_ok(k)) return 0;
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    return al(size_t(h->X.nt) * sizeof(float)) + al(h->X.fwd_items.size() * size_t(k * k * k) * sizeof(float));
}

apr_status_t apr_convolve_adjoint(apr_handle_t h, const float *stencils, int32_t k, int32_t bc, const float *grad_out,
                                  float *grad_particles, float *grad_tree, apr_stream_t stream) {
    if (!h || h->host_only) return APR_ERR_INVALID_ARG;
    if (!stencil_k_ok(k)) return APR_ERR_UNSUPPORTED;
    if (bc != APR_BC_REFLECT && bc != APR_BC_ZERO) return APR_ERR_INVALID_ARG;
    const HostIndex &X = h->X;
    if (!stencils || (X.np && (!grad_out || !grad_particles)) || (X.nt && !grad_tree)) return APR_ERR_INVALID_ARG;
    // the units store the gradient of every particle and tree node; only in an index in which some have
    // no record (a layout that was not validated) are the arrays cleared first
    cudaError_t e = cudaSuccess;
    if (!X.complete && X.np) e = cudaMemsetAsync(grad_particles, 0, size_t(X.np) * sizeof(float), stream);
    if (!X.complete && e == cudaSuccess && X.nt) e = cudaMemsetAsync(grad_tree, 0, size_t(X.nt) * sizeof(float), stream);
    if (e == cudaSuccess) e = launch_adjoint(k, h->U, stencils, bc, grad_out, grad_particles, grad_tree, stream);
    return cuda_status(e);
}

apr_status_t apr_tree_restrict_adjoint(apr_handle_t h, float *grad_tree, float *grad_particles, apr_stream_t stream) {
    if (!h || h->host_only) return APR_ERR_INVALID_ARG;
    return pushdown_levels(h, grad_tree, grad_particles, h->X.l_min, h->X.l_max - 1, stream);
}

apr_status_t apr_tree_restrict_adjoint_levels(apr_handle_t h, float *grad_tree, float *grad_particles,
                                              int32_t level_first, int32_t level_last, apr_stream_t stream) {
    if (!h || h->host_only || level_first > level_last) return APR_ERR_INVALID_ARG;
    return pushdown_levels(h, grad_tree, grad_particles, level_first, level_last, stream);
}

size_t apr_stencil_grad_workspace_bytes(apr_handle_t h, int32_t k) {
    if (!h || !stencil_k_ok(k)) return 0;
    return (h->X.fwd_items.size() * size_t(k * k * k) * sizeof(float) + 255) / 256 * 256;
}

apr_status_t apr_convolve_stencil_grad(apr_handle_t h, const float *particles, const float *tree, int32_t k, int32_t bc,
                                       const float *grad_out, float *grad_stencils, void *workspace,
                                       size_t workspace_bytes, apr_stream_t stream) {
    if (!h || h->host_only) return APR_ERR_INVALID_ARG;
    if (!stencil_k_ok(k)) return APR_ERR_UNSUPPORTED;
    if (bc != APR_BC_REFLECT && bc != APR_BC_ZERO) return APR_ERR_INVALID_ARG;
    const HostIndex &X = h->X;
    if (!grad_stencils || (X.np && (!particles || !grad_out)) || (X.nt && !tree)) return APR_ERR_INVALID_ARG;
    if (!aligned16(particles) || !aligned16(tree)) return misaligned();
    const size_t need = apr_stencil_grad_workspace_bytes(h, k);
    if (need && (!workspace || workspace_bytes < need || (reinterpret_cast<uintptr_t>(workspace) & 255))) return APR_ERR_INVALID_ARG;
    // One wave: the blocks have equal shares, so more than are resident (2 per SM at 3^3, 3 at 5^3) would take two
    // waves of them (3^3, 3 instead of 2 per SM: 8 M particles 172 instead of 152 us, 1 M 27 instead of 23 us, all-finest
    // 128^3 image 35 instead of 31 us). The workspace has a column per forward work item, and a
    // block needs one per level beyond its first.
    UnitLevels L;
    UnitRanges R;
    const int stride = int(X.fwd_items.size());
    const int blocks = unit_levels(h, std::min(stencil_grad_blocks(k) * h->sms, stride - h->n_levels_with + 1), L, R);
    return cuda_status(launch_stencil_grad(k, h->U, L, R, blocks, X.l_max - X.l_min + 1, particles, tree, bc, grad_out,
                                           static_cast<float *>(workspace), stride, grad_stencils, stream));
}

}  // extern "C"

namespace aprk {
apr_status_t convolve_backward(apr_handle_t h, const float *particles, const float *tree, const float *stencils,
                               int32_t k, int32_t bc, const float *grad_out, float *grad_particles,
                               float *grad_stencils, void *workspace, size_t workspace_bytes, apr_stream_t stream,
                               bool concurrent) {
    if (!h || h->host_only) return APR_ERR_INVALID_ARG;
    if (!stencil_k_ok(k)) return APR_ERR_UNSUPPORTED;
    if (bc != APR_BC_REFLECT && bc != APR_BC_ZERO) return APR_ERR_INVALID_ARG;
    const HostIndex &X = h->X;
    if (!stencils || (X.np && !grad_out)) return APR_ERR_INVALID_ARG;
    if (grad_stencils && ((X.np && !particles) || (X.nt && !tree))) return APR_ERR_INVALID_ARG;
    const size_t need = apr_backward_workspace_bytes(h, k);
    if (!workspace || workspace_bytes < need || (reinterpret_cast<uintptr_t>(workspace) & 255)) return APR_ERR_INVALID_ARG;
    const size_t gt_bytes = (size_t(X.nt) * sizeof(float) + 255) / 256 * 256;
    float *gt = static_cast<float *>(workspace);
    void *partial = static_cast<char *>(workspace) + gt_bytes;
    apr_status_t st = APR_OK;
    if (concurrent && grad_particles && grad_stencils) {
        // the stencil gradient reads only the values, the tree and dL/dout: it runs on the handle's
        // second stream while the data adjoint and the tree adjoint run on the caller's (their
        // workspace regions are disjoint); the caller's stream then waits for it
        std::lock_guard<std::mutex> lock(h->side_mu);
        cudaError_t e = cudaSuccess;
        if (!h->side) e = cudaStreamCreateWithFlags(&h->side, cudaStreamNonBlocking);
        if (e == cudaSuccess && !h->ev_fork) e = cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming);
        if (e == cudaSuccess && !h->ev_join) e = cudaEventCreateWithFlags(&h->ev_join, cudaEventDisableTiming);
        const cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
        if (e == cudaSuccess) e = cudaEventRecord(h->ev_fork, s);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(h->side, h->ev_fork, 0);
        if (e != cudaSuccess) return cuda_status(e);
        const apr_status_t sg = apr_convolve_stencil_grad(h, particles, tree, k, bc, grad_out, grad_stencils, partial,
                                                          workspace_bytes - gt_bytes, reinterpret_cast<apr_stream_t>(h->side));
        st = apr_convolve_adjoint(h, stencils, k, bc, grad_out, grad_particles, gt, stream);
        if (st == APR_OK) st = apr_tree_restrict_adjoint(h, gt, grad_particles, stream);
        // always joined, so that a stream capture of the caller's stream ends joined
        e = cudaEventRecord(h->ev_join, h->side);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, h->ev_join, 0);
        if (st == APR_OK) st = sg;
        if (st == APR_OK && e != cudaSuccess) st = cuda_status(e);
        return st;
    }
    if (grad_particles) {
        st = apr_convolve_adjoint(h, stencils, k, bc, grad_out, grad_particles, gt, stream);
        if (st == APR_OK) st = apr_tree_restrict_adjoint(h, gt, grad_particles, stream);
    }
    if (st == APR_OK && grad_stencils)
        st = apr_convolve_stencil_grad(h, particles, tree, k, bc, grad_out, grad_stencils, partial,
                                       workspace_bytes - gt_bytes, stream);
    return st;
}
}  // namespace aprk

extern "C" {

apr_status_t apr_convolve_backward(apr_handle_t h, const float *particles, const float *tree, const float *stencils,
                                   int32_t k, int32_t bc, const float *grad_out, float *grad_particles,
                                   float *grad_stencils, void *workspace, size_t workspace_bytes,
                                   apr_stream_t stream) {
    return aprk::convolve_backward(h, particles, tree, stencils, k, bc, grad_out, grad_particles, grad_stencils,
                                   workspace, workspace_bytes, stream, true);
}

size_t apr_rl_workspace_bytes(apr_handle_t h) {
    if (!h) return 0;
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    return al(size_t(h->X.nt) * sizeof(float)) + al(size_t(h->X.np) * sizeof(float));
}

apr_status_t apr_richardson_lucy(apr_handle_t h, const float *observed, const float *stencils, int32_t k, int32_t bc,
                                 int32_t n_iter, float *estimate, void *workspace, size_t workspace_bytes,
                                 apr_stream_t stream) {
    if (!h || h->host_only) return APR_ERR_INVALID_ARG;
    if (!stencil_k_ok(k)) return APR_ERR_UNSUPPORTED;
    if (bc != APR_BC_REFLECT && bc != APR_BC_ZERO) return APR_ERR_INVALID_ARG;
    const HostIndex &X = h->X;
    if (n_iter < 0 || !stencils || (X.np && (!observed || !estimate))) return APR_ERR_INVALID_ARG;
    if (!aligned16(estimate)) return misaligned();
    const size_t need = apr_rl_workspace_bytes(h);
    if (need && (!workspace || workspace_bytes < need || (reinterpret_cast<uintptr_t>(workspace) & 255)))
        return APR_ERR_INVALID_ARG;
    float *tree = static_cast<float *>(workspace);
    float *ratio = reinterpret_cast<float *>(static_cast<char *>(workspace) + (size_t(X.nt) * sizeof(float) + 255) / 256 * 256);
    for (int it = 0; it < n_iter; ++it) {
        // ratio = u / (i_k conv w); i_{k+1} = i_k * (ratio conv w_flipped); each convolution with the
        // tree restriction of its input before it
        apr_status_t st = restrict_then_conv(h, k, estimate, tree, stencils, bc, ratio, stream, EPI_DIVIDE, false, observed);
        if (st != APR_OK) return st;
        st = restrict_then_conv(h, k, ratio, tree, stencils, bc, estimate, stream, EPI_MULTIPLY, true, estimate);
        if (st != APR_OK) return st;
    }
    return APR_OK;
}

apr_status_t apr_sync_status(apr_handle_t h, apr_stream_t stream) {
    if (!h) return APR_ERR_INVALID_ARG;
    if (h->host_only) return APR_OK;
    cudaError_t e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return cuda_status(e);
    unsigned v = 0;
    e = cudaMemcpy(&v, h->d_err, sizeof(unsigned), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_status(e);
    if (v) {
        cudaMemset(h->d_err, 0, sizeof(unsigned));
        return (v & ERR_TIMEOUT) ? APR_ERR_TIMEOUT : APR_ERR_DEVICE;
    }
    return APR_OK;
}

}  // extern "C"
