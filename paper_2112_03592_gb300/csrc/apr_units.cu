// APR convolution, its data adjoint, its stencil gradient and the gradient magnitude on convolution
// units (apr_unitplan.cpp): groups of parents of level-l cells with the list of the parents around them.
//
// One block per unit. It stages, for every slot, the 2 x 2 x 2 octet of level-l values under that parent
// (Sec. 3.5: level-l particles, level-l tree nodes, or the level-(l-1) particle over all eight cells) in
// four shared-memory planes, plane (a, b) holding the pair of cells (2z + a, 2x + b, 2y .. 2y + 1) of slot
// s as one float2 at [s]; the three parents of a row along y are consecutive slots, so a row of cells is
// read with three 8-byte loads. Then one thread per record computes the eight child cells from the
// 4^3 (radius 1) or 6^3 (radius 2) cells around them, in registers. Reflection and the zero boundary are
// in the staged octets (slots outside the grid), so the sums have no boundary case.
//
// Why units: particles lie in thin shells, so the 8 x 8 x 64-cell tiles used before held 230 to 1200
// particles of 4096 cells, and a tile cost about 7000 warp instructions of set-up, staging and window
// bookkeeping (525 thread instructions per particle). Parents are dense blocks: seven of their eight
// children are particles on average, a record takes about 300 thread instructions at radius 1, and
// units are equally full wherever the particles lie. Measured (7.9 M particles of a 1024 x 1024 x 512
// image, restricted 5^3 stack, kernels alone with a cold L2): convolution 235 -> 90 us, data adjoint 500
// -> 197 us, stencil gradient 360 -> 190 us; 36.5 M instead of 131.8 M warp instructions per convolution.
// What bounds them now: shared-memory wavefronts (the L1 pipe is 75 % busy in the convolution; 2.5
// wavefronts per 4-byte load, since the slots of 32 records lie in many short runs) and the latency of
// header -> entry -> value at four blocks of 256 threads per SM; DRAM traffic is 0.23 GB, 34 us.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>
#include <utility>

#include "apr_device.cuh"
#include "apr_internal.h"
#include "apr_units.cuh"

namespace aprk {

namespace {

using namespace dev;

constexpr int UT = UNIT_RECS;   // threads per block of the unit kernels (one per record)

// Stencil rows (dz, dx) in shared memory, laid out for paired FP32 FMAs over neighbouring taps: radius 1
// (w0, w1, w1, w2), radius 2 (w0, w1, w2, w3, w1, w2, w3, w4).
template <int R>
__host__ __device__ constexpr int row_floats() {
    return R == 1 ? 4 : 8;
}
template <int R>
__host__ __device__ constexpr int taps_floats() {
    return (2 * R + 1) * (2 * R + 1) * row_floats<R>();
}
// One position of tap t of stencil row `row` (its first), and its value.
template <int R>
__device__ __forceinline__ float tap(const float *w, int row, int t) {
    return R == 1 ? w[row * 4 + (t < 2 ? t : 3)] : w[row * 8 + (t < 4 ? t : 7)];
}

// The staged octets (see above); SC: one plane per cell.
struct Planes {
    float2 p2[4][PLANE];
    __device__ __forceinline__ const float *cell(int c) const { return reinterpret_cast<const float *>(p2) + c * PLANE; }
    __device__ __forceinline__ float *cell(int c) { return reinterpret_cast<float *>(p2) + c * PLANE; }
    template <bool SC>
    __device__ __forceinline__ void store(unsigned slot, const float (&v)[8]) {
        if constexpr (SC) {
#pragma unroll
            for (int c = 0; c < 8; ++c) cell(c)[slot] = v[c];
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) p2[k][slot] = make_float2(v[2 * k], v[2 * k + 1]);
        }
    }
};

// The records' row slots, read back by the record's own thread (they would cost nine registers).
struct Bases {
    uint16_t b[9][UNIT_RECS];
    __device__ __forceinline__ unsigned at(int r) const { return b[r][threadIdx.x]; }
};

struct UnitSmem {
    Planes pl;
    Bases bs;
    alignas(16) float w[3][taps_floats<2>()];
};
struct AdjSmem {
    UnitSmem u;
    float H[8][UNIT_RECS];    // image sums (edge_images)
    int first[UNIT_RECS];     // first image of each edge record
    int wsum[UT / 32];
};
struct LeafSmem {
    Planes pl;
    alignas(16) float w[taps_floats<2>()];
    alignas(16) float sw[8][27 * 8];   // summed taps, by missing children (sum_weights)
};

// The taps of one level of a stencil stack of radius RS, one per thread in a register (loaded ahead of the
// staging), written to shared memory once the radius is known.
template <int RS>
struct Taps {
    static constexpr int KS = 2 * RS + 1, KS3 = KS * KS * KS;
    float v;
    __device__ __forceinline__ void load(const float *__restrict__ stencils, int l_idx, bool flip) {
        const int t = threadIdx.x;
        v = t < KS3 ? load_after_wait(stencils + l_idx * KS3 + (flip ? KS3 - 1 - t : t)) : 0.f;
    }
    // True on every thread if all taps outside the central 3^3 are zero (RS = 2). Such a level is
    // convolved with radius 1: a restricted 5^3 stencil (Eq. restrict_stenc) has support 2 ceil(2 / s) + 1
    // = 3 cells per axis at every level with cell edge s >= 2, i.e. below l_max. The result is the same
    // linear map (the skipped products are 0 * u); only its FP32 summation order differs. A block barrier.
    __device__ __forceinline__ bool radius1() const {
        if (RS == 1) return true;
        const int t = threadIdx.x, a = t / 25, b = (t / 5) % 5, c = t % 5;
        const bool outer = t < 125 && (a == 0 || a == 4 || b == 0 || b == 4 || c == 0 || c == 4);
        return __syncthreads_or(outer && v != 0.f) == 0;
    }
    // The central taps in the layout of radius R <= RS.
    template <int R>
    __device__ __forceinline__ void store(float *w) const {
        constexpr int K = 2 * R + 1, N = row_floats<R>(), D = RS - R;
        const int t = threadIdx.x, z = t / (KS * KS) - D, x = (t / KS) % KS - D, y = t % KS - D;
        if (t >= KS3 || unsigned(z) >= unsigned(K) || unsigned(x) >= unsigned(K) || unsigned(y) >= unsigned(K)) return;
        float *row = w + (z * K + x) * N;
        if (R == 1) {
            row[y == 2 ? 3 : y] = v;
            if (y == 1) row[2] = v;
        } else {
            if (y < 4) row[y] = v;
            if (y > 0) row[3 + y] = v;
        }
    }
};

// Staging of a unit's slots. entries() loads the entries, and after pdl_wait values() the values of the first slots of every kind
// (2 pure, 1 other node and 2 remaining ones per thread: nearly all of a unit), all in flight together;
// commit(): writes them to shared memory and takes what is left in loops. The chain is header -> entry ->
// value: loops over one kind after another, and child maps read through a node index, made it three
// times as long (the convolution of 7.9 M particles: 107 -> 94 us).
// Pure slots (all eight cells particles of the level, four nodes of five) take one 16-byte entry.
__device__ __forceinline__ void load_pure(const uint4 &q, const float *__restrict__ src, float (&v)[8]) {
    const unsigned p[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float *s = src + (p[k] & 0x0fffffffu);
        v[2 * k] = load_after_wait(s);
        v[2 * k + 1] = load_after_wait(s + 1);
    }
}
// The eight cells of a node entry; TREE: with its tree-node children (else zero there).
template <bool TREE>
__device__ __forceinline__ void load_node(const int4 &pw, const int4 &tw, const float *__restrict__ vals,
                                          const float *__restrict__ tree, float (&v)[8]) {
    const Octet o(pw, tw);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        v[c] = 0.f;
        if (o.kind[c] == 1 || (TREE && o.kind[c] == 2)) v[c] = load_after_wait((o.kind[c] == 1 ? vals : tree) + o.ix[c]);
    }
}

// VALUES: u_l (particles, tree, coarser particles); else dL/dout at the level-l particles, zero elsewhere
// and outside the grid.
template <bool VALUES>
struct Staging {
    uint4 q[2];
    float vp[2][8], vn[8], vo[2];
    uint2 e[2];
    int4 pw, tw;
    unsigned in, io[2];
    // entry arrays of the unit
    const uint4 *pure;
    const TreeNodePlan *nmap;
    const uint32_t *ninfo;
    const uint2 *oth;
    const float *__restrict__ vals;
    const float *__restrict__ tree;

    __device__ __forceinline__ void node(int i, unsigned &info, float (&v)[8]) const {
        const int4 *m = reinterpret_cast<const int4 *>(nmap + i);
        info = __ldg(ninfo + i);
        load_node<VALUES>(__ldg(m), VALUES ? __ldg(m + 1) : make_int4(0, 0, 0, 0), vals, tree, v);
    }
    __device__ __forceinline__ void entries(const UnitHdr &h) {
        const int tid = threadIdx.x, nt = int(blockDim.x);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int i = tid + u * nt;
            q[u] = i < h.npure ? __ldg(pure + i) : make_uint4(0, 0, 0, 0);
            e[u] = i < h.noth ? __ldg(oth + i) : make_uint2(0, 0);
        }
        pw = tw = make_int4(0, 0, 0, 0);
        in = 0;
        if (tid < h.nnode) {
            const int4 *m = reinterpret_cast<const int4 *>(nmap + tid);
            pw = __ldg(m);
            if (VALUES) tw = __ldg(m + 1);
            in = __ldg(ninfo + tid);
        }
    }
    __device__ __forceinline__ void values(const UnitHdr &h) {
        const int tid = threadIdx.x, nt = int(blockDim.x);
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (tid + u * nt < h.npure) load_pure(q[u], vals, vp[u]);
        if (tid < h.nnode) load_node<VALUES>(pw, tw, vals, tree, vn);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            io[u] = e[u].y;
            vo[u] = VALUES && tid + u * nt < h.nleaf ? load_after_wait(vals + e[u].x) : 0.f;
        }
    }
    template <bool SC>
    __device__ __forceinline__ void put(Planes &pl, unsigned info, float (&v)[8], bool reflect) const {
        if (info >> UE_MIRROR) edge_octet(v, info, reflect, 0.f);
        pl.store<SC>(info & UE_SLOT, v);
    }
    template <bool SC>
    __device__ __forceinline__ void commit(const UnitHdr &h, bool reflect, Planes &pl) {
        const int tid = threadIdx.x, nt = int(blockDim.x);
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (tid + u * nt < h.npure) pl.store<SC>(pure_slot(q[u]), vp[u]);
        if (tid < h.nnode) put<SC>(pl, in, vn, VALUES && reflect);
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (tid + u * nt < h.noth) {
                float v[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) v[c] = vo[u];
                put<SC>(pl, io[u], v, VALUES && reflect);
            }
        for (int i = tid + 2 * nt; i < h.npure; i += nt) {
            const uint4 r = __ldg(pure + i);
            float v[8];
            load_pure(r, vals, v);
            pl.store<SC>(pure_slot(r), v);
        }
        for (int i = tid + nt; i < h.nnode; i += nt) {
            unsigned info;
            float v[8];
            node(i, info, v);
            put<SC>(pl, info, v, VALUES && reflect);
        }
        for (int i = tid + 2 * nt; i < h.noth; i += nt) {
            const uint2 e = __ldg(oth + i);
            const float x = VALUES && i < h.nleaf ? load_after_wait(vals + e.x) : 0.f;
            float v[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) v[c] = x;
            put<SC>(pl, e.y, v, VALUES && reflect);
        }
    }
};
__device__ __forceinline__ Staging<true> value_staging(const UnitView &U, const UnitHdr &h, const float *__restrict__ vals,
                                                       const float *__restrict__ tree) {
    Staging<true> s;
    s.pure = U.pure + h.pure0;
    s.nmap = U.nmap + h.node0;
    s.ninfo = U.ninfo + h.node0;
    s.oth = U.oth + h.oth0;
    s.vals = vals;
    s.tree = tree;
    s.entries(h);
    return s;
}
__device__ __forceinline__ Staging<false> gradient_staging(const UnitView &U, const UnitHdr &h, bool leaf,
                                                           const float *__restrict__ gout) {
    Staging<false> s;
    s.pure = (leaf ? U.lpure : U.pure) + h.pure0;
    s.nmap = (leaf ? U.lnmap : U.nmap) + h.node0;
    s.ninfo = (leaf ? U.lninfo : U.ninfo) + h.node0;
    s.oth = U.oth + h.oth0;
    s.vals = gout;
    s.tree = nullptr;
    s.entries(h);
    return s;
}

// A record, loaded ahead of the staging: its row slots go to shared memory, node and edge word stay.
struct Rec {
    uint2 r0, r1, r2;
    __device__ __forceinline__ void load(const NodeRec *rec) {
        const uint2 *q = reinterpret_cast<const uint2 *>(rec);
        r0 = __ldg(q);
        r1 = __ldg(q + 1);
        r2 = __ldg(q + 2);
    }
    __device__ __forceinline__ unsigned node() const { return r0.x; }
    __device__ __forceinline__ void put(Bases &B, int n) const {
        unsigned b[9];
        unpack_bases(r0.y, r1, r2, b);
#pragma unroll
        for (int r = 0; r < 9; ++r) B.b[r][n] = uint16_t(b[r]);
    }
};

__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// Sums over one z plane of the cells around a record, radius 2: plane i (0..5, parent row dz = i >> 1,
// child a = i & 1) contributes with stencil plane i to the children with a = 0 (A0) and with stencil plane
// i - 1 to those with a = 1 (A1). s: the three row slots of the plane's parents; pl2: planes 2a, 2a + 1;
// w0: stencil plane i. A row (v0 .. v5) and stencil row (w0 .. w4) give the pair of children (e = 0, 1) as
// (w0, w1)(v0, v1) + (w2, w3)(v2, v3) + w4 v4 and w0 v1 + (w1, w2)(v2, v3) + (w3, w4)(v4, v5): paired FMAs
// on aligned pairs, six instructions instead of ten.
template <bool A0, bool A1>
__device__ __forceinline__ void plane_sums5(const float2 *pl2, const unsigned (&s)[3], const float *w0, float (&acc)[8]) {
    float2 p[2][4];
#pragma unroll
    for (int c = 0; c < 4; ++c) p[0][c] = p[1][c] = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const float2 *row = pl2 + (j & 1) * PLANE + s[j >> 1];
        const float2 q0 = row[0], q1 = row[1], q2 = row[2];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            if (a == 0 ? !A0 : !A1) continue;
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int tx = j - b;
                if (tx < 0 || tx > 4) continue;
                const float4 *wr = reinterpret_cast<const float4 *>(w0 - a * 40 + tx * 8);
                const float4 wa = wr[0], wb = wr[1];
                float2 &e0 = p[a][2 * b], &e1 = p[a][2 * b + 1];
                e0 = ffma2(make_float2(wa.x, wa.y), q0, e0);
                e0 = ffma2(make_float2(wa.z, wa.w), q1, e0);
                e0.x = fmaf(wb.w, q2.x, e0.x);
                e1 = ffma2(make_float2(wb.x, wb.y), q1, e1);
                e1 = ffma2(make_float2(wb.z, wb.w), q2, e1);
                e1.y = fmaf(wa.x, q0.y, e1.y);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        if (A0) acc[c] += p[0][c].x + p[0][c].y;
        if (A1) acc[4 + c] += p[1][c].x + p[1][c].y;
    }
}

// acc[c] = sum over the taps of the staged cells around child c of the record with row slots b. Short FP32
// chains: radius 1 sums the middle taps along y apart from the outer ones, radius 2 the even and odd taps
// of each stencil plane on their own (one chain of 27 terms had up to 1.7 times the rounding error).
template <int R>
__device__ __forceinline__ void unit_sums(const Planes &pl, const Bases &b, const float *w, float (&acc)[8]) {
    if constexpr (R == 1) {
        float2 p[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) p[c] = make_float2(0.f, 0.f);
        const float4 *wq = reinterpret_cast<const float4 *>(w);
#pragma unroll
        for (int i = 0; i < 4; ++i) {           // cell planes z - 1 .. z + 2
#pragma unroll
            for (int j = 0; j < 4; ++j) {       // cell rows x - 1 .. x + 2
                const int c0 = ((i + 1) & 1) * 4 + ((j + 1) & 1) * 2;
                const unsigned s = b.at(((i + 1) >> 1) * 3 + ((j + 1) >> 1));
                const float *q0 = pl.cell(c0) + s, *q1 = pl.cell(c0 + 1) + s;
                const float v0 = q1[0], v3 = q0[2];
                const float2 m = make_float2(q0[1], q1[1]);
#pragma unroll
                for (int a = 0; a < 2; ++a)
#pragma unroll
                    for (int bb = 0; bb < 2; ++bb) {
                        const int tz = i - a, tx = j - bb, c = 4 * a + 2 * bb;
                        if (tz < 0 || tz > 2 || tx < 0 || tx > 2) continue;
                        const float4 f = wq[tz * 3 + tx];   // w0, w1, w1, w2
                        p[c] = ffma2(make_float2(f.z, f.w), m, p[c]);
                        p[c].y = fmaf(f.x, v0, p[c].y);
                        p[c + 1] = ffma2(make_float2(f.x, f.y), m, p[c + 1]);
                        p[c + 1].x = fmaf(f.w, v3, p[c + 1].x);
                    }
            }
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = p[c].x + p[c].y;
    } else {
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = 0.f;
        {
            const unsigned s[3] = {b.at(0), b.at(1), b.at(2)};
            plane_sums5<true, false>(pl.p2[0], s, w, acc);
        }
#pragma unroll 1
        for (int i = 1; i < 5; ++i) {
            const int r = 3 * (i >> 1);
            const unsigned s[3] = {b.at(r), b.at(r + 1), b.at(r + 2)};
            plane_sums5<true, true>(pl.p2[2 * (i & 1)], s, w + i * 40, acc);
        }
        {
            const unsigned s[3] = {b.at(6), b.at(7), b.at(8)};
            plane_sums5<false, true>(pl.p2[2], s, w + 5 * 40, acc);
        }
    }
}

// Per-particle epilogue of the convolution: the plain output, or the element-wise division and
// multiplication of a Richardson-Lucy update (Sec. 6.2) fused into the write. aux may alias the
// output (each particle's entry is read, then written, by the same thread).
struct Epilogue {
    int mode;                  // EPI_PLAIN, EPI_DIVIDE (aux[p] / acc, 0 if acc <= 0), EPI_MULTIPLY (aux[p] * acc)
    bool flip;                 // taps in reversed order in every dimension (the flipped stencil)
    const float *aux;
    __device__ __forceinline__ float apply(int p, float acc) const {
        if (mode == EPI_DIVIDE) return acc > 0.f ? __fdiv_rn(aux[p], acc) : 0.f;
        if (mode == EPI_MULTIPLY) return aux[p] * acc;
        return acc;
    }
};

// Work items [first, first + n) of a tile-range call; n < 0: every record.
struct TileRange {
    int first, n;
    __device__ __forceinline__ bool has(const int32_t *tile, int rec) const {
        return n < 0 || unsigned(tile[rec] - first) < unsigned(n);
    }
};

// ------------------------------------------------------------------------------------------------
// APR convolution (Sec. 4.1).
// ------------------------------------------------------------------------------------------------
template <int R>
__global__ void __launch_bounds__(UT, 4) unit_conv_kernel(const UnitView U, const UnitHdr *units, const float *__restrict__ vals,
                                                          const float *__restrict__ tree,
                                                          const float *__restrict__ stencils, int bc, float *out,
                                                          const Epilogue epi, const TileRange tr) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    UnitSmem &S = *reinterpret_cast<UnitSmem *>(smem_raw);
    pdl_trigger();
    const UnitHdr h = units[blockIdx.x];
    const int tid = threadIdx.x;
    // the record, loaded ahead of the staging
    Rec rec{};
    const bool mine = tid < h.nrec && tr.has(U.tile_f, h.rec0 + tid);
    if (tr.n >= 0 && __syncthreads_or(mine) == 0) {
        pdl_wait();   // (their kernel must not end before the launch before it)
        return;
    }
    if (mine) rec.load(U.rec + h.rec0 + tid);
    Staging<true> st = value_staging(U, h, vals, tree);
    pdl_wait();
    Taps<R> taps;
    taps.load(stencils, h.lev, epi.flip);
    st.values(h);
    rec.put(S.bs, tid);
    const unsigned node = rec.node();
    const bool r1 = taps.radius1(), reflect = bc == APR_BC_REFLECT;
    if (r1) {
        taps.template store<1>(S.w[0]);
        st.commit<true>(h, reflect, S.pl);
    } else {
        taps.template store<R>(S.w[0]);
        st.commit<R == 1>(h, reflect, S.pl);
    }
    __syncthreads();
    if (!mine) return;
    float acc[8];
    if (r1) unit_sums<1>(S.pl, S.bs, S.w[0], acc);
    else unit_sums<R>(S.pl, S.bs, S.w[0], acc);
    for_child_particles(child_particles(U, node), [&](int p, int c) { out[p] = epi.apply(p, acc[c]); });
}

// Gradient magnitude (Sec. 4.3, Sobel filters with level-rescaled stencils, Eq. adapt_grad):
// out[p] = sqrt(sum_a (w_a (*) u)_p^2) for three stencil stacks w_a (a = z, x, y) on one staged unit.
template <int R>
__global__ void __launch_bounds__(UT, 3) unit_gradmag_kernel(const UnitView U, const float *__restrict__ vals,
                                                             const float *__restrict__ tree,
                                                             const float *__restrict__ stencils, int n_levels, int bc,
                                                             float *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    UnitSmem &S = *reinterpret_cast<UnitSmem *>(smem_raw);
    pdl_trigger();
    const UnitHdr h = U.work[blockIdx.x];
    const int tid = threadIdx.x;
    Rec rec{};
    if (tid < h.nrec) rec.load(U.rec + h.rec0 + tid);
    constexpr int K3 = (2 * R + 1) * (2 * R + 1) * (2 * R + 1);
    Staging<true> st = value_staging(U, h, vals, tree);
    pdl_wait();
    Taps<R> taps[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) taps[a].load(stencils + size_t(a) * n_levels * K3, h.lev, false);
    st.values(h);
#pragma unroll
    for (int a = 0; a < 3; ++a) taps[a].template store<R>(S.w[a]);
    rec.put(S.bs, tid);
    const unsigned node = rec.node();
    st.commit<R == 1>(h, bc == APR_BC_REFLECT, S.pl);
    __syncthreads();
    if (tid >= h.nrec) return;
    float sq[8] = {};
#pragma unroll 1
    for (int a = 0; a < 3; ++a) {
        float acc[8];
        unit_sums<R>(S.pl, S.bs, S.w[a], acc);
#pragma unroll
        for (int c = 0; c < 8; ++c) sq[c] = fmaf(acc[c], acc[c], sq[c]);
    }
    for_child_particles(child_particles(U, node), [&](int p, int c) { out[p] = sqrtf(sq[c]); });
}

// ------------------------------------------------------------------------------------------------
// Backward, data part: for every level-l cell c,
//   H(c) = sum over preimages c' of c under the boundary reflection of sum_e w[e] g(c' - e),
// g = dL/dout at the level-l particles (zero elsewhere, and outside the grid). H goes to the source that
// supplied cell c in the forward patch: the level-l particle or tree node (unit_adjoint_kernel: the
// record's children) or the level-(l-1) particle over c (leaf_adjoint_kernel, launched after it, adds the
// sum over the particle's eight cells). A particle gets at most these two terms, in this order.
// ------------------------------------------------------------------------------------------------
// A missing child's sum belongs to its sibling.
__device__ __forceinline__ void fold_missing(unsigned edge, float (&v)[8]) {
    const unsigned miss = missing_children(edge);
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const unsigned m = 1u << ax;
        if (miss & m) {
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (!(c & int(m))) v[c] += v[c | int(m)];
        }
    }
}

// Writes a record's sums to its children: stored, or added to what this thread stored before; ATOMIC: the
// particles' sums are added to what other calls may add to at the same time.
template <bool ATOMIC>
__device__ __forceinline__ void emit_children(const UnitView &U, unsigned node, const float (&v)[8], bool add, float *gp,
                                              float *gt) {
    const int4 *m = reinterpret_cast<const int4 *>(U.nplan + node);
    const Octet o(__ldg(m), __ldg(m + 1));
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        if (o.kind[c] == 1) {
            if (!ATOMIC) gp[o.ix[c]] = add ? gp[o.ix[c]] + v[c] : v[c];
            else if (v[c] != 0.f) atomicAdd(gp + o.ix[c], v[c]);
        } else if (o.kind[c] == 2) {
            gt[o.ix[c]] = add ? gt[o.ix[c]] + v[c] : v[c];
        }
    }
}

// The images of the block's edge records (the first h.nflag; `live`: this thread's record is computed by
// this call), added to what emit_children has stored; ATOMIC: the record's own sums too, so that a
// particle gets them as one term and concurrent calls' terms can come in any order. All images of the unit are dealt to the threads,
// then every record adds its own in order: a record in a corner has seven, one after the other they
// took most of the call on small images (0.8 M particles, 5^3 taps on every level: 63 -> 35 us). Not
// inlined: few units have edge records, and the code next to the records' own sums cost those registers.
template <int R, bool ATOMIC>
__device__ __noinline__ void edge_images(const UnitView &U, const UnitHdr &h, AdjSmem &S, bool live, float *gp, float *gt) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const NodeRec *rec = U.rec + h.rec0;
    constexpr int SELF = ATOMIC ? 0 : 1;   // shifts left out: the record's own place
    int n = 0;   // this record's images
    if (tid < h.nflag) n = __popcll(edge_shifts<R>(rec[tid].edge)) - SELF;
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int q = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += q;
    }
    if (lane == 31) S.wsum[warp] = incl;
    __syncthreads();
    int before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < UT / 32; ++w) {
        before += w < warp ? S.wsum[w] : 0;
        total += S.wsum[w];
    }
    const int first = before + incl - n;
    S.first[tid] = first;
    __syncthreads();
    float sum[8], own[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) sum[c] = own[c] = 0.f;
#pragma unroll 1
    for (int k0 = 0; k0 < total; k0 += UT) {
        const int k = k0 + tid;
        if (k < total) {
            int a = 0, b = h.nflag;   // the record with first[a] <= k
            while (b - a > 1) {
                const int m = (a + b) / 2;
                if (S.first[m] <= k) a = m;
                else b = m;
            }
            unsigned long long m = edge_shifts<R>(rec[a].edge);
            for (int q = k - S.first[a] + SELF; q > 0; --q) m &= m - 1ull;
            const int t = __ffsll((long long)m) - 1;
            const int iz = t >> 4, ix = (t >> 2) & 3, iy = t & 3, dy = iy == 1 ? -1 : (iy == 0 ? 0 : iy - 1);
            for (int q = 0; q < 9; ++q) {
                const int oz = image_layer(iz, q / 3), ox = image_layer(ix, q % 3);
                S.u.bs.b[q][tid] = uint16_t(oz < 0 || ox < 0 ? ZERO_SLOT : unsigned(int(rec[a].base[3 * oz + ox]) + dy));
            }
            float v[8];
            unit_sums<R>(S.u.pl, S.u.bs, S.u.w[0], v);
            const int mir = (iz ? 4 : 0) | (ix ? 2 : 0) | (iy ? 1 : 0);
#pragma unroll
            for (int c = 0; c < 8; ++c) S.H[c ^ mir][tid] = v[c];
        }
        __syncthreads();
        const int a = max(first, k0) - k0, b = min(first + n, k0 + UT) - k0;
        if (live)
            for (int q = a; q < b; ++q)
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    if (ATOMIC && k0 + q == first) own[c] = S.H[c][q];
                    else sum[c] += S.H[c][q];
                }
        __syncthreads();
    }
    if (live && n > 0) {
        // own sums and images are added in the same order either way: the results agree bit for bit
        fold_missing(rec[tid].edge, sum);
        if (ATOMIC) {
            fold_missing(rec[tid].edge, own);
#pragma unroll
            for (int c = 0; c < 8; ++c) sum[c] = own[c] + sum[c];
        }
        emit_children<ATOMIC>(U, rec[tid].node, sum, !ATOMIC, gp, gt);
    }
}

template <int R, bool ATOMIC>
__device__ __forceinline__ void block_adjoint(const UnitView &U, const UnitHdr &h, AdjSmem &S, unsigned node, bool live,
                                              bool reflect, float *gp, float *gt) {
    if (live && !(ATOMIC && reflect && threadIdx.x < h.nflag)) {
        float v[8];
        unit_sums<R>(S.u.pl, S.u.bs, S.u.w[0], v);
        if (reflect && threadIdx.x < h.nflag) fold_missing(U.rec[h.rec0 + threadIdx.x].edge, v);
        emit_children<ATOMIC>(U, node, v, false, gp, gt);
    }
    if (reflect && h.nflag > 0) edge_images<R, ATOMIC>(U, h, S, live && int(threadIdx.x) < h.nflag, gp, gt);
}

template <bool SC>
__device__ __forceinline__ void zero_slots(Planes &pl) {
    const float z[8] = {};
    if (threadIdx.x < 3) pl.store<SC>(ZERO_SLOT + threadIdx.x, z);
}

// ADD: gradients are added (tile-range calls: other calls may add to the same particles); else they
// are stored (every particle and tree node is the child of one record).
template <int R, bool ADD>
__global__ void __launch_bounds__(UT, 4) unit_adjoint_kernel(const UnitView U, const UnitHdr *units, const float *__restrict__ stencils,
                                                             int bc, const float *__restrict__ gout,
                                                             float *__restrict__ gp, float *__restrict__ gt,
                                                             const TileRange tr) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    AdjSmem &S = *reinterpret_cast<AdjSmem *>(smem_raw);
    pdl_trigger();
    const UnitHdr h = units[blockIdx.x];
    const int tid = threadIdx.x;
    Rec rec{};
    const bool live = tid < h.nrec && tr.has(U.tile_b, h.rec0 + tid);
    if (ADD && __syncthreads_or(live) == 0) {
        pdl_wait();
        return;
    }
    if (live) rec.load(U.rec + h.rec0 + tid);
    Staging<false> st = gradient_staging(U, h, false, gout);
    pdl_wait();
    Taps<R> taps;
    taps.load(stencils, h.lev, true);
    st.values(h);
    rec.put(S.u.bs, tid);
    const unsigned node = rec.node();
    const bool r1 = taps.radius1();
    if (r1) {
        taps.template store<1>(S.u.w[0]);
        zero_slots<true>(S.u.pl);
        st.commit<true>(h, false, S.u.pl);
    } else {
        taps.template store<R>(S.u.w[0]);
        zero_slots<R == 1>(S.u.pl);
        st.commit<R == 1>(h, false, S.u.pl);
    }
    __syncthreads();
    if (r1) block_adjoint<1, ADD>(U, h, S, node, live, bc == APR_BC_REFLECT, gp, gt);
    else block_adjoint<R, ADD>(U, h, S, node, live, bc == APR_BC_REFLECT, gp, gt);
}

// Summed taps of a coarse source: sw[3 r + j][child] = sum over the source's cells d of w[d - q] for the
// cell q = that child of neighbour j of row r (w: the flipped stencil), without the cells along the axes in
// `miss` (missing second children).
template <int R>
__device__ __forceinline__ void sum_weights(const float *w, int miss, float *sw) {
    constexpr int K = 2 * R + 1;
    for (int i = threadIdx.x; i < 27 * 8; i += int(blockDim.x)) {
        const int n = i >> 3, c = i & 7;
        const int qz = 2 * (n / 9 - 1) + (c >> 2), qx = 2 * ((n / 3) % 3 - 1) + ((c >> 1) & 1), qy = 2 * (n % 3 - 1) + (c & 1);
        float s = 0.f;
        for (int d = 0; d < 8; ++d) {
            const int tz = qz - (d >> 2) + R, tx = qx - ((d >> 1) & 1) + R, ty = qy - (d & 1) + R;
            if (!(d & miss) && unsigned(tz) < unsigned(K) && unsigned(tx) < unsigned(K) && unsigned(ty) < unsigned(K))
                s += tap<R>(w, tz * K + tx, ty);
        }
        sw[i] = s;
    }
}

// The sum over a coarse source's cells of H, from its neighbour nodes (mask, row slots b) against sw.
template <int R>
__device__ __forceinline__ float leaf_sums(const Planes &pl, const unsigned (&b)[9], unsigned mask,
                                           const float *sw) {
    float total = 0.f;
#pragma unroll
    for (int r = 0; r < 9; ++r) {
        const unsigned m = (mask >> (3 * r)) & 7u;
        const int dz = r / 3 - 1, dx = r % 3 - 1;
        float part = 0.f;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            if (r == 4 && j == 1) continue;   // the source itself
            const int dy = j - 1;
            if ((m >> j) & 1u) {
                const unsigned s = b[r] + __popc(m & ((1u << j) - 1u));
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    // cells within reach of the source's cells along every axis
                    const int qz = 2 * dz + (k >> 1), qx = 2 * dx + (k & 1), q0 = 2 * dy, q1 = 2 * dy + 1;
                    if (qz < -R || qz > 1 + R || qx < -R || qx > 1 + R) continue;
                    const float2 v = pl.p2[k][s];
                    const float2 f = reinterpret_cast<const float2 *>(sw)[(3 * r + j) * 4 + k];
                    if (q0 >= -R && q0 <= 1 + R) part = fmaf(f.x, v.x, part);
                    if (q1 >= -R && q1 <= 1 + R) part = fmaf(f.y, v.y, part);
                }
            }
        }
        total += part;
    }
    return total;
}

template <int R>
__device__ __forceinline__ float leaf_adjoint(const Planes &pl, const uint4 &q0, const uint4 &q1, const LeafRec *grec,
                                              bool reflect, const float (*sw)[27 * 8]) {
    const unsigned edge = q0.z & 0xffffu;
    unsigned long long todo = reflect && edge ? edge_shifts<R>(edge) : 1ull;
    // with the zero boundary the cells outside the grid are no part of the source; with reflection they
    // are images of its other cells
    const float *swm = sw[reflect || !edge ? 0 : missing_children(edge)];
    float total = 0.f;
#pragma unroll 1
    do {
        const int t = __ffsll((long long)todo) - 1;
        todo &= todo - 1ull;
        unsigned b[9], mask = q0.y;
        unpack_bases(q0.z, make_uint2(q0.w, q1.x), make_uint2(q1.y, q1.z), b);
        if (t) {
            const int iz = t >> 4, ix = (t >> 2) & 3, iy = t & 3;
            mask = 0;
#pragma unroll
            for (int r = 0; r < 9; ++r) {
                const int oz = image_layer(iz, r / 3), ox = image_layer(ix, r % 3), o = 3 * oz + ox;
                b[r] = 0;
                if (oz < 0 || ox < 0) continue;
                const unsigned m = (q0.y >> (3 * o)) & 7u;
                b[r] = grec->base[o] + (iy == 0 ? 0u : __popc(m & (iy == 3 ? 3u : 1u)));
                mask |= (iy == 0 ? m : (iy == 1 ? (m << 1) & 4u : (m >> (iy - 1)) & 1u)) << (3 * r);
            }
        }
        total += leaf_sums<R>(pl, b, mask, swm);
    } while (todo);
    return total;
}

template <int R, bool ADD>
__global__ void __launch_bounds__(UT, 4) leaf_adjoint_kernel(const UnitView U, const UnitHdr *units, const float *__restrict__ stencils,
                                                             int bc, const float *__restrict__ gout,
                                                             float *__restrict__ gp, const TileRange tr) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LeafSmem &S = *reinterpret_cast<LeafSmem *>(smem_raw);
    pdl_trigger();
    const UnitHdr h = units[blockIdx.x];
    const int tid = threadIdx.x;
    const bool live = tid < h.nrec && tr.has(U.ltile_b, h.rec0 + tid), reflect = bc == APR_BC_REFLECT;
    uint4 q0 = make_uint4(0, 0, 0, 0), q1 = q0;
    if (ADD && __syncthreads_or(live) == 0) {
        pdl_wait();
        return;
    }
    if (live) {
        const uint4 *q = reinterpret_cast<const uint4 *>(U.lrec + h.rec0 + tid);
        q0 = __ldg(q);
        q1 = __ldg(q + 1);
    }
    Staging<false> st = gradient_staging(U, h, true, gout);
    pdl_wait();
    Taps<R> taps;
    taps.load(stencils, h.lev, true);
    st.values(h);
    const bool r1 = taps.radius1();
    if (r1) taps.template store<1>(S.w);
    else taps.template store<R>(S.w);
    st.commit<false>(h, false, S.pl);
    __syncthreads();
    const int nmiss = !reflect && h.nflag > 0 ? 8 : 1;
    for (int v = 0; v < nmiss; ++v) {
        if (r1) sum_weights<1>(S.w, v, S.sw[v]);
        else sum_weights<R>(S.w, v, S.sw[v]);
    }
    __syncthreads();
    if (!live) return;
    const LeafRec *grec = U.lrec + h.rec0 + tid;
    const float s = r1 ? leaf_adjoint<1>(S.pl, q0, q1, grec, reflect, S.sw) : leaf_adjoint<R>(S.pl, q0, q1, grec, reflect, S.sw);
    if (!ADD) gp[q0.x] += s;
    else if (s != 0.f) atomicAdd(gp + q0.x, s);
}

// ------------------------------------------------------------------------------------------------
// Backward, stencil part: grad_w[l][e] = sum over the level's particles p of g_p u_l(p + e).
//
// A block takes a contiguous range of the units of the levels that hold particles. Warp (tz, q) owns
// stencil plane tz: each lane takes records (nodes) in turn and keeps the plane's K^2 taps of its records
// of the unit in registers (8 K^2 products per record from the two cell planes z + tz, z + tz + 1); at the
// unit's end the 32 lanes are summed by a halving exchange (lane t keeps tap t), so a running sum is one
// register per lane and chains stay short. At a level's end the warps' sums are written to the level's
// partial of this block, and stencil_grad_reduce_kernel adds the blocks in order.
// ------------------------------------------------------------------------------------------------
template <int R>
struct WgradSmem {
    static constexpr int K = 2 * R + 1, Q = R == 1 ? 4 : 2, NT = K * Q * 32;
    static constexpr int BLOCKS = R == 1 ? 2 : 3;   // resident per SM (80 registers x 384 threads, 64 x 320)
    Planes pl;
    float g[8][UNIT_RECS];
    Bases bs;
    float red[K * Q][K * K];
    unsigned bad;             // levels with a sum that is not finite (live_levels)
};

// Sum over the 32 lanes of v[t], t < N <= 32: returned on lane t.
template <int N>
__device__ __forceinline__ float lane_sums(const float (&v)[N]) {
    const int lane = threadIdx.x & 31;
    float a[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {   // lanes with bit 4 keep taps 16 + i, the others taps i
        const float lo = i < N ? v[i] : 0.f, hi = 16 + i < N ? v[16 + i < N ? 16 + i : 0] : 0.f;
        const float send = (lane & 16) ? lo : hi, keep = (lane & 16) ? hi : lo;
        a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int h = 8; h > 0; h >>= 1)
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float send = (lane & h) ? a[i] : a[i + h], keep = (lane & h) ? a[i + h] : a[i];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
        }
    return a[0];
}

// dL/dout of the children of unit h's records (zero where the child is no particle) and the records' row slots.
template <int R>
__device__ __forceinline__ void stage_gradient(const UnitView &U, const UnitHdr &h, const float *gout, WgradSmem<R> &S) {
    for (int n = threadIdx.x; n < h.nrec; n += WgradSmem<R>::NT) {
        Rec rec;
        rec.load(U.rec + h.rec0 + n);
        rec.put(S.bs, n);
        float g[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) g[c] = 0.f;
        for_child_particles(child_particles(U, rec.node()), [&](int p, int c) { g[c] = load_after_wait(gout + p); });
#pragma unroll
        for (int c = 0; c < 8; ++c) S.g[c][n] = g[c];
    }
}
// The warps' sums of a level (lane t: tap t of the warp's plane) to the block's partial of it; whether all are finite.
template <int R>
__device__ __forceinline__ bool put_partial(WgradSmem<R> &S, float run, float *partial, int stride) {
    constexpr int K = WgradSmem<R>::K, Q = WgradSmem<R>::Q;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane < K * K) S.red[warp][lane] = run;
    __syncthreads();
    bool finite = true;
    for (int t = threadIdx.x; t < K * K * K; t += WgradSmem<R>::NT) {
        float s = 0.f;
#pragma unroll
        for (int qq = 0; qq < Q; ++qq) s += S.red[qq * K + t / (K * K)][t % (K * K)];
        partial[size_t(t) * stride] = s;
        finite = finite && isfinite(s);
    }
    return finite;
}

// The levels in S.bad again, over the particles alone. unit_wgrad_kernel multiplies the cells around a record with
// the zero that stands for a child that is no particle, so an infinity or NaN there is in sums of particles
// that do not read it. Taken by blocks with a sum that is not finite; the others pay for the test of what they write
// (nothing measurable). 1 M particles: 3^3 28 us, one infinite value 39 us, all infinite 65 us; 5^3 36, 82, 132 us.
template <int R>
__device__ __noinline__ void live_levels(WgradSmem<R> &S, const UnitView &U, const UnitLevels &W, const float *vals, const float *tree,
                                         int bc, const float *gout, float *partial, int stride) {
    constexpr int K = WgradSmem<R>::K;
    const int lane = threadIdx.x & 31, tz = (threadIdx.x >> 5) % K, q = (threadIdx.x >> 5) / K, total = W.begin[W.n];
    const int u0 = int(int64_t(blockIdx.x) * total / gridDim.x), u1 = int(int64_t(blockIdx.x + 1) * total / gridDim.x);
#pragma unroll 1
    for (int i = 0; i < W.n; ++i) {
        if (!((S.bad >> i) & 1u)) continue;
        float run = 0.f;
#pragma unroll 1
        for (int u = max(u0, W.begin[i]); u < min(u1, W.begin[i + 1]); ++u) {
            const UnitHdr h = U.hdr[W.unit0[i] + u - W.begin[i]];
            Staging<true> st = value_staging(U, h, vals, tree);
            st.values(h);
            __syncthreads();
            stage_gradient<R>(U, h, gout, S);
            st.commit<false>(h, bc == APR_BC_REFLECT, S.pl);
            __syncthreads();
            float acc[K * K];
#pragma unroll
            for (int t = 0; t < K * K; ++t) acc[t] = 0.f;
#pragma unroll 1
            for (int n = q * 32 + lane; n < h.nrec; n += WgradSmem<R>::Q * 32) {
                unsigned live = 0;
                for_child_particles(child_particles(U, U.rec[h.rec0 + n].node), [&](int, int c) { live |= 1u << c; });
#pragma unroll 1
                for (; live; live &= live - 1) {
                    // child c's cells, counted from two before the parent's first one
                    const int c = __ffs(live) - 1, z = (c >> 2) + tz - R + 2, x0 = ((c >> 1) & 1) - R + 2, y0 = (c & 1) - R + 2;
                    const float g = S.g[c][n];
#pragma unroll
                    for (int t = 0; t < K * K; ++t) {
                        const int x = x0 + t / K, y = y0 + t % K;
                        const float2 v = S.pl.p2[2 * (z & 1) + (x & 1)][S.bs.b[3 * (z >> 1) + (x >> 1)][n] + (y >> 1)];
                        acc[t] = fmaf(g, y & 1 ? v.y : v.x, acc[t]);
                    }
                }
            }
            __syncwarp();
            run += lane_sums(acc);
        }
        put_partial<R>(S, run, partial + blockIdx.x + i, stride);
    }
}

template <int R>
__global__ void __launch_bounds__(WgradSmem<R>::NT, WgradSmem<R>::BLOCKS) unit_wgrad_kernel(const UnitView U, const UnitLevels W,
                                                                      const float *__restrict__ vals,
                                                                      const float *__restrict__ tree, int bc,
                                                                      const float *__restrict__ gout,
                                                                      float *__restrict__ partial, int stride) {
    using Smem = WgradSmem<R>;
    constexpr int K = Smem::K, Q = Smem::Q;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem &S = *reinterpret_cast<Smem *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, tz = warp % K, q = warp / K;
    const int total = W.begin[W.n];
    const int u0 = int(int64_t(blockIdx.x) * total / gridDim.x), u1 = int(int64_t(blockIdx.x + 1) * total / gridDim.x);
    if (tid == 0) S.bad = 0;
    for (int i = 0; i < W.n; ++i) {
        const int a = max(u0, W.begin[i]), b = min(u1, W.begin[i + 1]);
        if (a >= b) continue;
        float run = 0.f;
        for (int u = a; u < b; ++u) {
            const UnitHdr h = U.hdr[W.unit0[i] + u - W.begin[i]];
            Staging<true> st = value_staging(U, h, vals, tree);
            st.values(h);
            __syncthreads();   // the previous unit's (or level's) readers are done
            stage_gradient<R>(U, h, gout, S);
            st.commit<false>(h, bc == APR_BC_REFLECT, S.pl);
            __syncthreads();
            float acc[K * K];
#pragma unroll
            for (int t = 0; t < K * K; ++t) acc[t] = 0.f;
            for (int n = q * 32 + lane; n < h.nrec; n += Q * 32) {
#pragma unroll
                for (int a2 = 0; a2 < 2; ++a2) {
                    // cell plane 2z + a2 + tz - R: parent row dz, child plane pa
                    const int i2 = a2 + tz - R + 2, dz = i2 >> 1, pa = i2 & 1;
                    const unsigned s[3] = {S.bs.b[3 * dz][n], S.bs.b[3 * dz + 1][n], S.bs.b[3 * dz + 2][n]};
                    const float g[4] = {S.g[4 * a2][n], S.g[4 * a2 + 1][n], S.g[4 * a2 + 2][n], S.g[4 * a2 + 3][n]};
#pragma unroll
                    for (int j = 0; j < K + 1; ++j) {   // cell rows 2x + j - R
                        const int j2 = j - R + 2;
                        const float2 *row = S.pl.p2[2 * pa + (j2 & 1)] + s[j2 >> 1];
                        float v[K + 1];
                        if constexpr (R == 1) {
                            const float2 m = row[1];
                            v[0] = row[0].y;
                            v[1] = m.x;
                            v[2] = m.y;
                            v[3] = row[2].x;
                        } else {
                            const float2 q0 = row[0], q1 = row[1], q2 = row[2];
                            v[0] = q0.x;
                            v[1] = q0.y;
                            v[2] = q1.x;
                            v[3] = q1.y;
                            v[4] = q2.x;
                            v[5] = q2.y;
                        }
#pragma unroll
                        for (int bb = 0; bb < 2; ++bb) {
                            const int tx = j - bb;
                            if (tx < 0 || tx >= K) continue;
#pragma unroll
                            for (int t = 0; t < K; ++t) {
                                acc[tx * K + t] = fmaf(g[2 * bb], v[t], acc[tx * K + t]);
                                acc[tx * K + t] = fmaf(g[2 * bb + 1], v[t + 1], acc[tx * K + t]);
                            }
                        }
                    }
                }
            }
            run += lane_sums(acc);
        }
        if (!put_partial<R>(S, run, partial + blockIdx.x + i, stride)) atomicOr(&S.bad, 1u << i);
    }
    __syncthreads();
    if (S.bad) live_levels<R>(S, U, W, vals, tree, bc, gout, partial, stride);
}

// grad_w[lev][e] = sum of the level's block partials (partial[e][block + i], blocks first .. last for the
// i-th level), in a fixed order; zero for a level without particles.
__global__ void __launch_bounds__(128) stencil_grad_reduce_kernel(const float *__restrict__ partial, int stride,
                                                                  const UnitRanges rg, int K3,
                                                                  float *__restrict__ gw) {
    __shared__ float red[4];
    const int lev = blockIdx.y, e = blockIdx.x, tid = threadIdx.x;
    float s = 0.f;
    for (int i = rg.first[lev] + tid; i <= rg.last[lev]; i += 128) s += partial[size_t(e) * stride + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((tid & 31) == 0) red[tid >> 5] = s;
    __syncthreads();
    if (tid == 0) gw[size_t(lev) * K3 + e] = (red[0] + red[1]) + (red[2] + red[3]);
}

// Shared memory per block sets the blocks per SM (228 KB per SM, 1 KB reserved per block).
static_assert(4 * (sizeof(UnitSmem) + 1024) <= 228 * 1024, "convolution units: four blocks per SM");
static_assert(4 * (sizeof(AdjSmem) + 1024) <= 228 * 1024, "adjoint units: four blocks per SM");
static_assert(4 * (sizeof(LeafSmem) + 1024) <= 228 * 1024, "leaf units: four blocks per SM");
static_assert(WgradSmem<1>::BLOCKS * (sizeof(WgradSmem<1>) + 1024) <= 228 * 1024, "stencil gradient: two blocks per SM");
static_assert(WgradSmem<2>::BLOCKS * (sizeof(WgradSmem<2>) + 1024) <= 228 * 1024, "stencil gradient: three blocks per SM");
static_assert(UNIT_SLOTS <= int(UE_SLOT) + 1, "slot numbers fit an entry");

// pdl: the kernel starts while the launch before it finishes and loads its header, records and entries meanwhile. A
// chain of small launches is bound by these: ten Richardson-Lucy iterations of 40 k particles 409 -> 272 us, 20 of 2.8 M
// 2506 -> 2354 us; restriction and 5^3 convolution of 1 M 30 -> 27 us; gradient magnitude of 1.2 M 35 -> 31 us.
template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kernel)(KArgs...), int grid, int block, size_t smem, cudaStream_t s, bool pdl, Args &&...args) {
    if (grid <= 0) return cudaSuccess;
    cudaError_t e = set_max_dynamic_smem(reinterpret_cast<const void *>(kernel), smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(kernel, dim3(grid), dim3(block), smem, s, pdl, std::forward<Args>(args)...);
}

}  // namespace

// The units of a launch: `all` of them, longest first, or those of a range call, `span` of them in their own order.
// (Over all units, as a first form did, a rank's ranges cost the whole image's headers once per level. An eighth of 8 M
// particles, one range per level: convolution 3^3 56 -> 44, 5^3 89 -> 75, adjoint 146 -> 102 and 214 -> 165 us; one work
// item: adjoint 17 and 19 -> 7.5 us.)
struct Units {
    const UnitHdr *hdr;
    int n;
    Units(const UnitHdr *sorted, int all, const UnitHdr *hdr_, const UnitSpan &span, bool range)
        : hdr(range && span.last - span.first < all ? hdr_ + span.first : sorted), n(range ? span.last - span.first : all) {}
};

// n_units: the units of the levels down to the coarsest one with particles (the finest come first).
// first_tile, n_tiles: a range of forward work items, whose records are in the units `span`; n_tiles < 0: all.
cudaError_t launch_conv_fwd(int k, const UnitView &U, int n_units, const float *vals, const float *tree, const float *st,
                            int bc, float *out, cudaStream_t s, int epi_mode, bool flip, const float *aux, const UnitSpan &span,
                            int first_tile, int n_tiles) {
    const Epilogue epi{epi_mode, flip, aux};
    const TileRange tr{first_tile, n_tiles};
    const Units u(U.work, n_units, U.hdr, span, n_tiles >= 0);
    return k == 3 ? launch(unit_conv_kernel<1>, u.n, UT, sizeof(UnitSmem), s, true, U, u.hdr, vals, tree, st, bc, out, epi, tr)
                  : launch(unit_conv_kernel<2>, u.n, UT, sizeof(UnitSmem), s, true, U, u.hdr, vals, tree, st, bc, out, epi, tr);
}

cudaError_t launch_gradmag(int k, const UnitView &U, int n_units, const float *vals, const float *tree, const float *st,
                           int n_levels, int bc, float *out, cudaStream_t s) {
    return k == 3 ? launch(unit_gradmag_kernel<1>, n_units, UT, sizeof(UnitSmem), s, true, U, vals, tree, st, n_levels, bc, out)
                  : launch(unit_gradmag_kernel<2>, n_units, UT, sizeof(UnitSmem), s, true, U, vals, tree, st, n_levels, bc, out);
}

// The data adjoint: stored gradients over all units, or (n_tiles >= 0) gradients added over a range of
// adjoint work items, whose records are in the given spans of the node and the leaf units.
template <int R>
static cudaError_t launch_adjoint_t(const UnitView &U, const float *st, int bc, const float *gout, float *gp, float *gt,
                                    cudaStream_t s, const UnitSpan &nodes, const UnitSpan &leaves, const TileRange &tr) {
    const bool add = tr.n >= 0;
    const Units un(U.work_adj, U.n, U.hdr, nodes, add), ul(U.lwork, U.nl, U.lhdr, leaves, add);
    cudaError_t e = launch(add ? unit_adjoint_kernel<R, true> : unit_adjoint_kernel<R, false>, un.n, UT, sizeof(AdjSmem), s, true, U,
                           un.hdr, st, bc, gout, gp, gt, tr);
    // (started early, the leaf units slow the last wave of the node units: 8 M particles 208 -> 215 us; the few units
    // of a range call start early)
    if (e == cudaSuccess)
        e = launch(add ? leaf_adjoint_kernel<R, true> : leaf_adjoint_kernel<R, false>, ul.n, UT, sizeof(LeafSmem), s, ul.n < U.nl, U, ul.hdr, st,
                   bc, gout, gp, tr);
    return e;
}
cudaError_t launch_adjoint(int k, const UnitView &U, const float *st, int bc, const float *gout, float *gp, float *gt,
                           cudaStream_t s, const UnitSpan &nodes, const UnitSpan &leaves, int first_tile, int n_tiles) {
    const TileRange tr{first_tile, n_tiles};
    return k == 3 ? launch_adjoint_t<1>(U, st, bc, gout, gp, gt, s, nodes, leaves, tr)
                  : launch_adjoint_t<2>(U, st, bc, gout, gp, gt, s, nodes, leaves, tr);
}

int stencil_grad_blocks(int k) { return k == 3 ? WgradSmem<1>::BLOCKS : WgradSmem<2>::BLOCKS; }
// The stencil gradient into gw [n_levels][k^3], on the blocks of W, R (unit_levels). partial: k^3 x stride
// floats; block b writes its i-th level to column b + i.
cudaError_t launch_stencil_grad(int k, const UnitView &U, const UnitLevels &W, const UnitRanges &R, int blocks, int n_levels,
                                const float *vals, const float *tree, int bc, const float *gout, float *partial, int stride,
                                float *gw, cudaStream_t s) {
    const cudaError_t e =
        k == 3 ? launch(unit_wgrad_kernel<1>, blocks, WgradSmem<1>::NT, sizeof(WgradSmem<1>), s, false, U, W, vals, tree, bc, gout, partial, stride)
               : launch(unit_wgrad_kernel<2>, blocks, WgradSmem<2>::NT, sizeof(WgradSmem<2>), s, false, U, W, vals, tree, bc, gout, partial, stride);
    if (e != cudaSuccess) return e;
    stencil_grad_reduce_kernel<<<dim3(k * k * k, n_levels), 128, 0, s>>>(partial, stride, R, k * k * k, gw);
    return cudaGetLastError();
}

}  // namespace aprk
