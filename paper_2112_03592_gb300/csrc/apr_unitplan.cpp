// Host builder of the convolution units (apr_units.cuh), once per APR.
//
// A level-l cell lies in a parent cell of the level-(l-1) grid, and the parents of the particles and
// tree nodes of level l are tree nodes (for l = l_min, where the tree ends, "virtual" parents hold the
// same 2 x 2 x 2 child cells). All taps of a 3^3 or 5^3 stencil around a parent's eight child cells lie
// in the 3 x 3 x 3 parents around it. So the unit of work is a group of parents (records) together with
// the list of the parents around them (slots): the kernels stage one 2 x 2 x 2 octet of values per slot
// in shared memory and find a record's neighbourhood through nine slot numbers, one per (z, x) row,
// since the three parents of a row along y are consecutive slots. Parents outside the level grid are
// slots too, with the reflected octet as their source (or zeros), so records need no boundary case.
//
// Units are cut from blocks of 32^3 parents, walked in 4^3 bricks in Morton order, so that a unit is
// compact: about 3.6 slots per record at 256 records on the blob images (4.2 at 128, 5.0 at 64; the
// 8 x 8 x 64-cell tiles these units replace hold 29 parents on average at the finest level of the
// 1024 x 1024 x 512 image and stage 1224 parents' space for them).
#include <algorithm>
#include <atomic>
#include <cstring>
#include <memory>
#include <thread>

#include "apr_internal.h"

namespace aprk {

namespace {

constexpr int UB = 32;        // parents per block edge
constexpr int UW = UB + 2;    // with a one-parent halo
constexpr int Y0 = 2;         // bit of a row word that holds the block's first parent along y

// The parents of one level's cells: sorted y per row of tree nodes (or virtual parents) and, at a
// coarser particle level, of particles.
struct ParentLevel {
    int l = 0;                          // level of the child cells
    int pz = 0, px = 0, py = 0;         // parent grid
    int dz = 0, dx = 0, dy = 0;         // child grid
    const uint32_t *nrow = nullptr;     // row offsets of the nodes (into ny), row 0 = (0, 0)
    const uint16_t *ny = nullptr;
    int64_t node0 = 0;                  // node index = node0 + position in ny
    const TreeNodePlan *maps = nullptr; // child maps of the nodes, by position in ny
    const uint32_t *prow = nullptr;     // row offsets of the level-(l-1) particles, or null
    const uint16_t *py_ = nullptr;
};

struct Block {
    uint64_t N[UW][UW], L[UW][UW];      // nodes, particles: bit j = y0 - Y0 + j, with a one-parent halo
    uint32_t n0[UW][UW], l0[UW][UW];    // index of the first of each in the row's window
};

inline int popc(uint64_t v) { return __builtin_popcountll(v); }

// Source parent of an out-of-grid parent position along one axis (half-sample reflection of its two
// child cells); mirrored: its children are the source's in reversed order.
inline int source_axis(int q, int P, int d, bool &mirrored) {
    mirrored = q < 0 || q >= P;
    if (q < 0) return 0;
    if (q >= P) return d % 2 == 0 ? P - 1 : std::max(P - 2, 0);
    return q;
}

inline unsigned edge_code(int p, int d) {  // bit 0: first parent; bits 1, 2: cells left to the grid's end if <= 3
    const int left = d - 2 * p;
    return (p == 0 ? 1u : 0u) | (unsigned(left <= 3 ? left : 0) << 1);
}

struct JobOut {
    std::vector<UnitHdr> hdr, lhdr;
    std::vector<uint4> pure, lpure;
    std::vector<TreeNodePlan> nmap, lnmap;
    std::vector<uint32_t> ninfo, lninfo;
    std::vector<uint2> oth;
    std::vector<NodeRec> rec;
    std::vector<LeafRec> lrec;
    std::vector<int32_t> tf, tb, ltb;
    int64_t children[2] = {};           // particles and tree nodes among the records' children
    bool uncovered = false;
};

// f(0), ..., f(n - 1) on up to 16 threads, this one among them, and no more than one per 64 k of `work` (steps of some
// ten nanoseconds: starting a thread takes 50 to 100 us). Throws std::bad_alloc if a call threw.
template <typename F>
void parallel_for(size_t n, int64_t work_, F f) {
    std::atomic<size_t> next{0};
    std::atomic<bool> failed{false};
    auto work = [&] {
        try {
            for (size_t i = next++; i < n && !failed; i = next++) f(i);
        } catch (...) {
            failed = true;
        }
    };
    const unsigned nth = unsigned(std::min<int64_t>(std::max(1u, std::min(16u, std::thread::hardware_concurrency())),
                                                    std::min<int64_t>(int64_t(n), 1 + work_ / 65536)));
    std::vector<std::thread> threads;
    for (unsigned t = 1; t < nth; ++t) {
        try {
            threads.emplace_back(work);
        } catch (...) {
            break;  // fewer threads
        }
    }
    work();
    for (auto &t : threads) t.join();
    if (failed) throw std::bad_alloc();
}

class BlockJob {
  public:
    BlockJob(const ParentLevel &P, int l_min, int unit_recs, const int32_t *tf, const int32_t *tb, int ntx, int nty,
             JobOut &o)
        : P_(P), lev_(P.l - l_min), UN_(unit_recs), tf_(tf), tb_(tb), ntx_(ntx), nty_(nty), o_(o) {}

    void run(int bz, int bx, int by) {
        z0_ = bz * UB;
        x0_ = bx * UB;
        y0_ = by * UB;
        if (!fill()) return;
        node_units();
        if (P_.prow) leaf_units();
    }

  private:
    bool fill() {
        bool any = false;
        for (int z = 0; z < UW; ++z)
            for (int x = 0; x < UW; ++x) {
                K_.N[z][x] = K_.L[z][x] = 0;
                K_.n0[z][x] = K_.l0[z][x] = 0;
                const int gz = z0_ - 1 + z, gx = x0_ - 1 + x;
                if (gz < 0 || gx < 0 || gz >= P_.pz || gx >= P_.px) continue;
                const int64_t row = int64_t(gz) * P_.px + gx;
                const int ya = y0_ - 1, yb = y0_ + UB + 1;
                auto scan = [&](const uint32_t *rows, const uint16_t *ys, uint64_t &bits, uint32_t &first) {
                    const uint16_t *b = ys + rows[row], *e = ys + rows[row + 1];
                    const uint16_t *p = ya <= 0 ? b : std::lower_bound(b, e, uint16_t(ya));
                    first = uint32_t(p - ys);
                    for (; p < e && int(*p) < yb; ++p) bits |= 1ull << (int(*p) - y0_ + Y0);
                };
                scan(P_.nrow, P_.ny, K_.N[z][x], K_.n0[z][x]);
                if (P_.prow) scan(P_.prow, P_.py_, K_.L[z][x], K_.l0[z][x]);
                if (z > 0 && x > 0 && z <= UB && x <= UB && ((K_.N[z][x] | K_.L[z][x]) & kInner)) any = true;
            }
        return any;
    }

    // Calls f(z, x, j) for the set bits of the inner rows of `bits`, in Morton order of 4^3 bricks.
    template <typename F>
    void walk(const uint64_t (*bits)[UW], F f) {
        for (int m = 0; m < 512; ++m) {
            int bz = 0, bx = 0, by = 0;
            for (int b = 0; b < 3; ++b) {
                by |= ((m >> (3 * b)) & 1) << b;
                bx |= ((m >> (3 * b + 1)) & 1) << b;
                bz |= ((m >> (3 * b + 2)) & 1) << b;
            }
            for (int z = 4 * bz + 1; z <= 4 * bz + 4; ++z)
                for (int x = 4 * bx + 1; x <= 4 * bx + 4; ++x) {
                    unsigned w = unsigned(bits[z][x] >> (4 * by + Y0)) & 15u;
                    while (w) {
                        const int j = 4 * by + Y0 + __builtin_ctz(w);
                        w &= w - 1;
                        f(z, x, j);
                    }
                }
        }
    }

    // The unit under construction lies in rows [za_, zb_] x [xa_, xb_] (records); slots one row further.
    void reset() {
        for (int z = std::max(za_ - 1, 0); z <= zb_ + 1; ++z)
            for (int x = std::max(xa_ - 1, 0); x <= xb_ + 1; ++x) T_[z][x] = D_[z][x] = 0;
        za_ = xa_ = UW;
        zb_ = xb_ = -2;
        nrec_ = nslot_ = 0;
    }

    // Slots of one row of record y = j: its three neighbours, and (node units, at the grid's ends along y)
    // the positions outside the grid that the data adjoint reads around its mirrored images, which it
    // stages as zeros.
    uint64_t row_slots(int j, bool guards) const {
        uint64_t w = 7ull << (j - 1);
        if (guards) {
            const int y = y0_ - Y0 + j, left = P_.dy - 2 * y;
            if (y == 0) w |= 1ull << (j - 2);
            if (left == 2 || (left == 1 && y == 0)) w |= 4ull << j;
            if (left == 3) w |= 12ull << j;
        }
        return w;
    }

    // Adds parent (z, x, j) with the neighbourhood restricted to `allow` rows (null: all 27); closes the
    // current unit first when it is full.
    template <typename Close>
    void add(int z, int x, int j, const uint64_t (*allow)[UW], Close close) {
        uint64_t w[9];
        const uint64_t all = row_slots(j, !allow);
        for (int r = 0; r < 9; ++r) w[r] = allow ? all & allow[z + r / 3 - 1][x + r % 3 - 1] : all;
        int inc = 0;
        for (int pass = 0; pass < 2; ++pass) {
            inc = 0;
            for (int r = 0; r < 9; ++r) inc += popc(w[r] & ~D_[z + r / 3 - 1][x + r % 3 - 1]);
            if (nrec_ < UN_ && nslot_ + inc <= UNIT_SLOTS) break;
            close();
            reset();
        }
        for (int r = 0; r < 9; ++r) D_[z + r / 3 - 1][x + r % 3 - 1] |= w[r];
        nslot_ += inc;
        T_[z][x] |= 1ull << j;
        za_ = std::min(za_, z);
        zb_ = std::max(zb_, z);
        xa_ = std::min(xa_, x);
        xb_ = std::max(xb_, x);
        ++nrec_;
    }

    int rank(int z, int x, int j) const { return pre_[z][x] + popc(D_[z][x] & ((1ull << j) - 1ull)); }
    void prefix() {
        int n = 0;
        for (int z = za_ - 1; z <= zb_ + 1; ++z)
            for (int x = xa_ - 1; x <= xb_ + 1; ++x) {
                pre_[z][x] = n;
                n += popc(D_[z][x]);
            }
    }
    unsigned edges(int gz, int gx, int gy) const {
        return edge_code(gz, P_.dz) | (edge_code(gx, P_.dx) << 3) | (edge_code(gy, P_.dy) << 6);
    }
    // Calls f(z, x, j, edges) for the unit's records: those at the grid's edges first.
    template <typename F>
    int records(F f) {
        int nflag = 0;
        for (int pass = 0; pass < 2; ++pass)
            for (int z = za_; z <= zb_; ++z)
                for (int x = xa_; x <= xb_; ++x) {
                    uint64_t w = T_[z][x];
                    while (w) {
                        const int j = __builtin_ctzll(w);
                        w &= w - 1;
                        const unsigned e = edges(z0_ - 1 + z, x0_ - 1 + x, y0_ - Y0 + j);
                        if ((e != 0) != (pass == 0)) continue;
                        f(z, x, j, e);
                        if (e) ++nflag;
                    }
                }
        return nflag;
    }
    void bases(int z, int x, int j, uint16_t *b) const {
        for (int r = 0; r < 9; ++r) b[r] = uint16_t(rank(z + r / 3 - 1, x + r % 3 - 1, j - 1));
    }
    void tiles(int z, int x, int j, int32_t &f, int32_t &b) const {
        const int64_t k = (int64_t((z0_ - 1 + z) / (TZ / 2)) * ntx_ + (x0_ - 1 + x) / (TX / 2)) * nty_ +
                          (y0_ - Y0 + j) / (BY / 2);
        f = tf_[k];
        b = tb_[k];
    }

    // Adds the entry of node `i` (position in ny): pure if its eight children are particles and it is
    // staged as it is.
    void put_node(uint32_t i, unsigned info, std::vector<uint4> &pure, std::vector<TreeNodePlan> &nmap,
                  std::vector<uint32_t> &ninfo) const {
        const TreeNodePlan &m = P_.maps[i];
        bool all = (info >> UE_MIRROR) == 0;
        for (int k = 0; k < 4; ++k) all = all && uint32_t(m.p[k]) >> 30 == 3u;
        if (!all) {
            nmap.push_back(m);
            ninfo.push_back(info);
            return;
        }
        uint32_t w[4];
        for (int k = 0; k < 4; ++k) w[k] = (uint32_t(m.p[k]) & 0x0fffffffu) | (((info >> (4 * k)) & 15u) << 28);
        pure.push_back(uint4{w[0], w[1], w[2], w[3]});
    }

    // Whether child cell c of in-grid parent (z, x, j) has a source.
    bool covered(int z, int x, int j, int c) const {
        const uint64_t bit = 1ull << j;
        if (!(K_.N[z][x] & bit)) return (K_.L[z][x] & bit) != 0;
        const TreeNodePlan &m = P_.maps[K_.n0[z][x] + popc(K_.N[z][x] & (bit - 1ull))];
        return ((uint32_t(m.p[c >> 1]) | uint32_t(m.t[c >> 1])) >> (30 + (c & 1))) & 1u;
    }
    // Whether a cell next to a particle of the unit's records lies in the grid and has no source (possible
    // only in a layout that was not validated).
    bool any_uncovered() const {
        for (int z = za_; z <= zb_; ++z)
            for (int x = xa_; x <= xb_; ++x)
                for (uint64_t w = T_[z][x]; w; w &= w - 1) {
                    const int j = __builtin_ctzll(w);
                    const TreeNodePlan &m = P_.maps[K_.n0[z][x] + popc(K_.N[z][x] & ((1ull << j) - 1ull))];
                    for (int c = 0; c < 8; ++c) {
                        if (!((uint32_t(m.p[c >> 1]) >> (30 + (c & 1))) & 1u)) continue;
                        for (int t = 0; t < 27; ++t) {
                            const int cz = 2 * (z0_ - 1 + z) + (c >> 2) + t / 9 - 1, cx = 2 * (x0_ - 1 + x) + ((c >> 1) & 1) + (t / 3) % 3 - 1,
                                      cy = 2 * (y0_ - Y0 + j) + (c & 1) + t % 3 - 1;
                            if (cz < 0 || cx < 0 || cy < 0 || cz >= P_.dz || cx >= P_.dx || cy >= P_.dy) continue;
                            if (!covered((cz >> 1) - (z0_ - 1), (cx >> 1) - (x0_ - 1), (cy >> 1) - (y0_ - Y0),
                                         4 * (cz & 1) + 2 * (cx & 1) + (cy & 1)))
                                return true;
                        }
                    }
                }
        return false;
    }

    void close_nodes() {
        if (!nrec_) return;
        prefix();
        bool holes = false;   // in-grid slots or children without a source
        UnitHdr h{};
        h.pure0 = int32_t(o_.pure.size());
        h.node0 = int32_t(o_.nmap.size());
        h.oth0 = int32_t(o_.oth.size());
        h.rec0 = int32_t(o_.rec.size());
        h.lev = int16_t(lev_);
        std::vector<uint2> &leaf = tmp_leaf_, &zero = tmp_zero_;
        leaf.clear();
        zero.clear();
        for (int z = za_ - 1; z <= zb_ + 1; ++z)
            for (int x = xa_ - 1; x <= xb_ + 1; ++x) {
                uint64_t w = D_[z][x];
                unsigned pos = unsigned(pre_[z][x]);
                for (; w; w &= w - 1, ++pos) {
                    const int j = __builtin_ctzll(w);
                    const int y = y0_ - Y0 + j;
                    if (y < -1 || y > P_.py) {   // only the data adjoint reads it
                        zero.push_back(uint2{0u, pos});
                        continue;
                    }
                    bool mz, mx, my;
                    const int sz = source_axis(z0_ - 1 + z, P_.pz, P_.dz, mz), sx = source_axis(x0_ - 1 + x, P_.px, P_.dx, mx),
                              sy = source_axis(y, P_.py, P_.dy, my);
                    const int wz = sz - (z0_ - 1), wx = sx - (x0_ - 1), wj = sy - (y0_ - Y0);
                    const uint64_t bit = 1ull << wj, below = bit - 1ull;
                    const unsigned miss = (2 * sz + 1 >= P_.dz ? 4u : 0u) | (2 * sx + 1 >= P_.dx ? 2u : 0u) | (2 * sy + 1 >= P_.dy ? 1u : 0u);
                    const unsigned mir = (mz ? 4u : 0u) | (mx ? 2u : 0u) | (my ? 1u : 0u);
                    unsigned info = pos | (mir << UE_MIRROR) | (miss << UE_MISS);
                    if (K_.N[wz][wx] & bit) {
                        const uint32_t i = uint32_t(K_.n0[wz][wx] + popc(K_.N[wz][wx] & below));
                        const TreeNodePlan &m = P_.maps[i];
                        const uint32_t k0 = uint32_t(m.p[0]) | uint32_t(m.t[0]), k1 = uint32_t(m.p[1]) | uint32_t(m.t[1]),
                                       k2 = uint32_t(m.p[2]) | uint32_t(m.t[2]), k3 = uint32_t(m.p[3]) | uint32_t(m.t[3]);
                        if (miss || (k0 & k1 & k2 & k3) >> 30 != 3u)
                            holes = holes || popc(uint64_t(k0 >> 30 | k1 >> 30 << 2 | k2 >> 30 << 4 | k3 >> 30 << 6)) != 8 >> popc(miss);
                        put_node(i, info, o_.pure, o_.nmap, o_.ninfo);
                    } else if (K_.L[wz][wx] & bit) {
                        leaf.push_back(uint2{uint32_t(K_.l0[wz][wx] + popc(K_.L[wz][wx] & below)), info});
                    } else {
                        holes = true;
                        zero.push_back(uint2{0u, info});
                    }
                }
            }
        h.npure = int16_t(int32_t(o_.pure.size()) - h.pure0);
        h.nnode = int16_t(int32_t(o_.nmap.size()) - h.node0);
        h.nleaf = int16_t(leaf.size());
        o_.oth.insert(o_.oth.end(), leaf.begin(), leaf.end());
        o_.oth.insert(o_.oth.end(), zero.begin(), zero.end());
        h.noth = int16_t(int32_t(o_.oth.size()) - h.oth0);
        h.nflag = int16_t(records([&](int z, int x, int j, unsigned e) {
            NodeRec r{};
            const uint32_t i = uint32_t(K_.n0[z][x] + popc(K_.N[z][x] & ((1ull << j) - 1ull)));
            r.node = uint32_t(P_.node0) + i;
            for (int k = 0; k < 4; ++k) {
                const uint32_t pm = uint32_t(P_.maps[i].p[k]) >> 30, tm = uint32_t(P_.maps[i].t[k]) >> 30;
                o_.children[0] += (pm & 1u) + (pm >> 1);
                o_.children[1] += (tm & 1u) + (tm >> 1);
            }
            r.edge = uint16_t(e);
            bases(z, x, j, r.base);
            o_.rec.push_back(r);
            int32_t f, b;
            tiles(z, x, j, f, b);
            o_.tf.push_back(f);
            o_.tb.push_back(b);
        }));
        h.nrec = int16_t(nrec_);
        if (holes && any_uncovered()) o_.uncovered = true;
        o_.hdr.push_back(h);
    }

    void node_units() {
        reset();
        walk(K_.N, [&](int z, int x, int j) { add(z, x, j, nullptr, [&] { close_nodes(); }); });
        close_nodes();
    }

    void close_leaves() {
        if (!nrec_) return;
        prefix();
        UnitHdr h{};
        h.pure0 = int32_t(o_.lpure.size());
        h.node0 = int32_t(o_.lnmap.size());
        h.rec0 = int32_t(o_.lrec.size());
        h.lev = int16_t(lev_);
        for (int z = za_ - 1; z <= zb_ + 1; ++z)
            for (int x = xa_ - 1; x <= xb_ + 1; ++x) {
                uint64_t w = D_[z][x];
                unsigned pos = unsigned(pre_[z][x]);
                for (; w; w &= w - 1, ++pos) {
                    const uint64_t bit = w & ~(w - 1);
                    put_node(uint32_t(K_.n0[z][x] + popc(K_.N[z][x] & (bit - 1ull))), pos, o_.lpure, o_.lnmap, o_.lninfo);
                }
            }
        h.npure = int16_t(int32_t(o_.lpure.size()) - h.pure0);
        h.nnode = int16_t(int32_t(o_.lnmap.size()) - h.node0);
        h.nflag = int16_t(records([&](int z, int x, int j, unsigned e) {
            LeafRec r{};
            r.particle = uint32_t(K_.l0[z][x] + popc(K_.L[z][x] & ((1ull << j) - 1ull)));
            r.edge = uint16_t(e);
            bases(z, x, j, r.base);
            for (int q = 0; q < 9; ++q)
                r.mask |= uint32_t((K_.N[z + q / 3 - 1][x + q % 3 - 1] >> (j - 1)) & 7u) << (3 * q);
            o_.lrec.push_back(r);
            int32_t f, b;
            tiles(z, x, j, f, b);
            o_.ltb.push_back(b);
        }));
        h.nrec = int16_t(nrec_);
        o_.lhdr.push_back(h);
    }

    // Level-(l-1) particles with a node among their 26 neighbours: the coarse sources of level l.
    void leaf_units() {
        uint64_t A[UW][UW] = {};
        bool any = false;
        for (int z = 1; z <= UB; ++z)
            for (int x = 1; x <= UB; ++x) {
                uint64_t n = 0;
                for (int r = 0; r < 9; ++r) n |= K_.N[z + r / 3 - 1][x + r % 3 - 1];
                A[z][x] = K_.L[z][x] & (n | (n << 1) | (n >> 1)) & kInner & ~K_.N[z][x];
                any = any || A[z][x];
            }
        if (!any) return;
        reset();
        walk(A, [&](int z, int x, int j) { add(z, x, j, K_.N, [&] { close_leaves(); }); });
        close_leaves();
    }

    static constexpr uint64_t kInner = ((1ull << UB) - 1ull) << Y0;
    const ParentLevel &P_;
    int lev_, UN_;
    const int32_t *tf_, *tb_;
    int ntx_, nty_;
    JobOut &o_;
    int z0_ = 0, x0_ = 0, y0_ = 0, nrec_ = 0, nslot_ = 0;
    int za_ = 1, zb_ = UB, xa_ = 1, xb_ = UB;   // (the first reset clears everything)
    Block K_;
    uint64_t T_[UW][UW], D_[UW][UW];
    int pre_[UW][UW];
    std::vector<uint2> tmp_leaf_, tmp_zero_;
};

// Virtual parents of the cells of l_min: rows, y and child maps of the parents with at least one
// particle or tree node among their child cells.
struct VirtualRows {
    std::vector<uint32_t> count;        // of each row
    std::vector<uint16_t> y;
    std::vector<TreeNodePlan> map;
};
void virtual_rows(const HostIndex &X, int64_t row0, int64_t row1, VirtualRows &V) {
    const LevelGeo &g = X.geo[X.l_min];
    const bool tree = X.l_min < X.l_max;
    const int px = (g.dx + 1) / 2;
    for (int64_t row = row0; row < row1; ++row) {
        const int z = int(row / px), x = int(row % px);
        const size_t begin = V.y.size();
        int64_t pa[4], pe[4], ta[4], te[4];
        for (int k = 0; k < 4; ++k) {
            const int cz = 2 * z + (k >> 1), cx = 2 * x + (k & 1);
            pa[k] = pe[k] = ta[k] = te[k] = 0;
            if (cz >= g.dz || cx >= g.dx) continue;
            const int64_t r = int64_t(cz) * g.dx + cx;
            pa[k] = X.row_ptr[size_t(g.row0 + r)];
            pe[k] = X.row_ptr[size_t(g.row0 + r + 1)];
            if (tree) {
                ta[k] = X.trow_ptr[size_t(g.trow0 + r)];
                te[k] = X.trow_ptr[size_t(g.trow0 + r + 1)];
            }
        }
        for (;;) {
            int y = INT32_MAX;
            for (int k = 0; k < 4; ++k) {
                if (pa[k] < pe[k]) y = std::min(y, int(X.y[size_t(pa[k])]) >> 1);
                if (ta[k] < te[k]) y = std::min(y, int(X.ty[size_t(ta[k])]) >> 1);
            }
            if (y == INT32_MAX) break;
            TreeNodePlan p{};
            for (int k = 0; k < 4; ++k) {
                uint32_t pw = uint32_t(pa[k]), tw = uint32_t(ta[k]);
                for (int e = 0; e < 2; ++e) {
                    const int cy = 2 * y + e;
                    const bool isp = pa[k] < pe[k] && int(X.y[size_t(pa[k])]) == cy;
                    if (isp) {
                        pw |= 1u << (30 + e);
                        ++pa[k];
                    }
                    if (ta[k] < te[k] && int(X.ty[size_t(ta[k])]) == cy) {  // (a cell that is both: the particle)
                        if (!isp) tw |= 1u << (30 + e);
                        ++ta[k];
                    }
                }
                p.p[k] = int32_t(pw);
                p.t[k] = int32_t(tw);
            }
            V.y.push_back(uint16_t(y));
            V.map.push_back(p);
        }
        V.count.push_back(uint32_t(V.y.size() - begin));
    }
}
void virtual_parents(HostIndex &X) {
    const LevelGeo &g = X.geo[X.l_min];
    const int64_t total = int64_t((g.dz + 1) / 2) * ((g.dx + 1) / 2);   // rows of parents
    const int64_t rows0 = g.row0, rows1 = rows0 + int64_t(g.dz) * g.dx, work = int64_t(X.row_ptr[size_t(rows1)]) - X.row_ptr[size_t(rows0)];
    const size_t n = size_t(std::min<int64_t>(total, 64));              // groups of them
    std::vector<VirtualRows> rows(n);
    parallel_for(n, work / 4, [&](size_t i) {
        virtual_rows(X, int64_t(i) * total / int64_t(n), int64_t(i + 1) * total / int64_t(n), rows[i]);
    });
    std::vector<size_t> first(n + 1, 0);
    X.vrow_ptr.assign(1, 0);
    X.vrow_ptr.reserve(size_t(total) + 1);
    for (size_t i = 0; i < n; ++i) {
        first[i + 1] = first[i] + rows[i].y.size();
        for (uint32_t c : rows[i].count) X.vrow_ptr.push_back(X.vrow_ptr.back() + c);
    }
    X.vy.resize(first[n]);
    X.vplan.resize(first[n]);
    parallel_for(n, work / 16, [&](size_t i) {
        std::copy(rows[i].y.begin(), rows[i].y.end(), X.vy.begin() + int64_t(first[i]));
        std::copy(rows[i].map.begin(), rows[i].map.end(), X.vplan.begin() + int64_t(first[i]));
        rows[i] = VirtualRows{};
    });
}

// The units of a launch in descending order of their work (a record's sums cost about as much as staging four
// pure slots or two others), so that its last wave consists of short ones. In the order they are built (finest
// level first, along the curve) the long blocks of the second finest level still start in the last of two or
// three waves. Measured: 20 Richardson-Lucy iterations of 2.8 M particles (3 waves) 2717 -> 2506 us, gradient
// magnitude of 1.2 M 39 -> 35 us, 16-channel leaf adjoint of 1 M 90 -> 75 us and of the FP32 one of 8 M 84 -> 72 us.
// flag: what an edge record's images cost on top (16-channel data adjoint of 1 M particles, whose images take tiles of
// their own: 106 -> 96 us; FP32 of 8 M 129 -> 124 us, which makes up for the lost neighbourhood).
template <typename It>
void sort_by_work(It first, It last, int flag = 0) {
    auto work = [flag](const UnitHdr &h) { return (4 * int(h.nrec) + int(h.npure) + 2 * (int(h.nnode) + int(h.noth))) + flag * int(h.nflag); };
    std::stable_sort(first, last, [&](const UnitHdr &a, const UnitHdr &b) { return work(a) > work(b); });
}

// The span of units (headers in their own order) that hold records of each of n work items.
std::vector<UnitSpan> item_spans(const std::vector<UnitHdr> &hdr, const std::vector<int32_t> &tile, size_t n) {
    std::vector<UnitSpan> s(n, UnitSpan{0, 0});
    for (size_t u = 0; u < hdr.size(); ++u)
        for (int32_t r = hdr[u].rec0; r < hdr[u].rec0 + hdr[u].nrec; ++r)
            if (tile[size_t(r)] >= 0) {
                UnitSpan &q = s[size_t(tile[size_t(r)])];
                if (q.last == 0) q.first = int32_t(u);
                q.last = int32_t(u) + 1;
            }
    return s;
}

void widen(UnitSpan &a, const UnitSpan &b) {
    if (b.first >= b.last) return;
    a = a.first >= a.last ? b : UnitSpan{std::min(a.first, b.first), std::max(a.last, b.last)};
}

}  // namespace

void UnitSpans::set(std::vector<UnitSpan> items) {
    item_ = std::move(items);
    group_.assign((item_.size() + G - 1) / G, UnitSpan{0, 0});
    for (size_t i = 0; i < item_.size(); ++i) widen(group_[i / G], item_[i]);
}

UnitSpan UnitSpans::of(int64_t first, int64_t n) const {
    UnitSpan s{0, 0};
    for (int64_t i = first; i < first + n;) {
        const bool whole = i % G == 0 && i + G <= first + n;
        widen(s, whole ? group_[size_t(i / G)] : item_[size_t(i)]);
        i += whole ? G : 1;
    }
    return s;
}

void build_units(HostIndex &X, int sms) {
    virtual_parents(X);
    UnitPlan &U = X.units;
    U = UnitPlan{};
    const int64_t parents = X.nt + int64_t(X.vy.size());
    // Records per unit: 256 where that fills the chip (4 resident units of 128 and more per multiprocessor), fewer for small
    // APRs, whose calls are bound by the latency of one unit, not by throughput. Measured with 256, 128 and 64: 142 k
    // parents, 16-channel training step 401, 424 and 586 us, gradient magnitude (174 k) 38, 43 and 51 us; 6 k parents, 16-channel
    // training step 128, 96 and 94 us, ten Richardson-Lucy iterations 301, 284 and 278 us.
    const int UN = parents >= int64_t(sms) * 4 * 128 ? 256 : parents >= int64_t(sms) * 64 ? 128 : 64;
    std::vector<ParentLevel> levels;
    std::vector<std::vector<int32_t>> tf, tb;
    std::vector<int> ntx, nty;
    for (int l = X.l_max; l >= X.l_min; --l) {
        const LevelGeo &g = X.geo[l];
        ParentLevel P;
        P.l = l;
        P.dz = g.dz;
        P.dx = g.dx;
        P.dy = g.dy;
        P.pz = (g.dz + 1) / 2;
        P.px = (g.dx + 1) / 2;
        P.py = (g.dy + 1) / 2;
        if (l == X.l_min) {
            P.nrow = X.vrow_ptr.data();
            P.ny = X.vy.data();
            P.node0 = X.nt;
            P.maps = X.vplan.data();
        } else {
            const LevelGeo &gp = X.geo[l - 1];
            P.nrow = X.trow_ptr.data() + gp.trow0;
            P.ny = X.ty.data();
            P.maps = X.tnplan.data();
            P.prow = X.row_ptr.data() + gp.row0;
            P.py_ = X.y.data();
        }
        levels.push_back(P);
        const int ntz = (g.dz + TZ - 1) / TZ, nx = (g.dx + TX - 1) / TX;
        ntx.push_back(nx);
        nty.push_back(g.nb);
        auto ids = [&](const std::vector<Item> &items, const int64_t *begin) {
            std::vector<int32_t> m(size_t(ntz) * nx * g.nb, -1);
            for (int64_t i = begin[l]; i < begin[l + 1]; ++i) {
                const Item &it = items[size_t(i)];
                m[(size_t(it.a) * nx + it.b) * g.nb + it.yb] = int32_t(i);
            }
            return m;
        };
        tf.push_back(ids(X.fwd_items, X.fwd_level_begin));
        tb.push_back(ids(X.bwd_items, X.bwd_level_begin));
    }
    struct Job {
        int li, bz, bx, by;
    };
    std::vector<Job> jobs;
    for (size_t i = 0; i < levels.size(); ++i) {
        const ParentLevel &P = levels[i];
        for (int z = 0; z * UB < P.pz; ++z)
            for (int x = 0; x * UB < P.px; ++x)
                for (int y = 0; y * UB < P.py; ++y) jobs.push_back(Job{int(i), z, x, y});
    }
    std::vector<JobOut> out(jobs.size());
    parallel_for(jobs.size(), int64_t(jobs.size()) * 65536, [&](size_t j) {
        const Job &J = jobs[j];
        std::unique_ptr<BlockJob> B(new BlockJob(levels[size_t(J.li)], X.l_min, UN, tf[size_t(J.li)].data(), tb[size_t(J.li)].data(),
                                                 ntx[size_t(J.li)], nty[size_t(J.li)], out[j]));
        B->run(J.bz, J.bx, J.by);
    });
    // The blocks' arrays one after the other, an array per thread: it is the first touch of the memory that takes the
    // time (with the virtual parents in threads too: handle of an all-finest 256^3 image 142 -> 114 ms, of 8 M particles
    // 655 -> 637, of a 1 x 1024 x 1024 plane 13.4 -> 10.9).
    int64_t children[2] = {};
    for (const JobOut &o : out) {
        children[0] += o.children[0];
        children[1] += o.children[1];
        U.uncovered = U.uncovered || o.uncovered;
    }
    for (int l = 0; l <= MAXL; ++l) U.level_begin[l] = 0;
    auto append = [&out](auto member, auto &dst) {
        size_t n = 0;
        for (const JobOut &o : out) n += (o.*member).size();
        dst.reserve(n);
        for (JobOut &o : out) {
            dst.insert(dst.end(), (o.*member).begin(), (o.*member).end());
        }
    };
    parallel_for(14, 4 * parents, [&](size_t task) {
        switch (task) {
            case 0: append(&JobOut::rec, U.rec); break;
            case 1: append(&JobOut::pure, U.pure); break;
            case 2: append(&JobOut::lrec, U.lrec); break;
            case 3: append(&JobOut::lpure, U.lpure); break;
            case 4: append(&JobOut::nmap, U.nmap); break;
            case 5: append(&JobOut::lnmap, U.lnmap); break;
            case 6: append(&JobOut::oth, U.oth); break;
            case 7: append(&JobOut::tf, U.tile_f); break;
            case 8: append(&JobOut::tb, U.tile_b); break;
            case 9: append(&JobOut::ltb, U.ltile_b); break;
            case 10: append(&JobOut::ninfo, U.ninfo); break;
            case 11: append(&JobOut::lninfo, U.lninfo); break;
            case 12: {   // headers, their first entries and records counted over all blocks
                UnitHdr n{};
                size_t j = 0;
                for (size_t i = 0; i < levels.size(); ++i) {
                    U.level_begin[levels[i].l - X.l_min] = int32_t(U.hdr.size());   // finest level first
                    for (; j < jobs.size() && jobs[j].li == int(i); ++j) {
                        for (UnitHdr h : out[j].hdr) {
                            h.pure0 += n.pure0;
                            h.node0 += n.node0;
                            h.oth0 += n.oth0;
                            h.rec0 += n.rec0;
                            U.hdr.push_back(h);
                        }
                        n.pure0 += int32_t(out[j].pure.size());
                        n.node0 += int32_t(out[j].nmap.size());
                        n.oth0 += int32_t(out[j].oth.size());
                        n.rec0 += int32_t(out[j].rec.size());
                    }
                }
                break;
            }
            default: {
                UnitHdr n{};
                for (const JobOut &o : out) {
                    for (UnitHdr h : o.lhdr) {
                        h.pure0 += n.pure0;
                        h.node0 += n.node0;
                        h.rec0 += n.rec0;
                        U.lhdr.push_back(h);
                    }
                    n.pure0 += int32_t(o.lpure.size());
                    n.node0 += int32_t(o.lnmap.size());
                    n.rec0 += int32_t(o.lrec.size());
                }
            }
        }
    });
    parallel_for(out.size(), parents, [&](size_t j) { out[j] = JobOut{}; });
    U.fwd_units.set(item_spans(U.hdr, U.tile_f, X.fwd_items.size()));
    U.bwd_units.set(item_spans(U.hdr, U.tile_b, X.bwd_items.size()));
    U.bwd_leaves.set(item_spans(U.lhdr, U.ltile_b, X.bwd_items.size()));
    U.lwork = U.lhdr;
    sort_by_work(U.lwork.begin(), U.lwork.end());
    U.work = U.hdr;
    for (int l = X.l_max; l >= X.l_min; --l)
        if (X.fwd_level_begin[l + 1] > X.fwd_level_begin[l])
            U.n_forward = l == X.l_min ? int32_t(U.hdr.size()) : U.level_begin[l - 1 - X.l_min];
    const auto forward = U.work.begin() + U.n_forward;
    sort_by_work(U.work.begin(), forward);
    sort_by_work(forward, U.work.end());
    U.work_adj = U.hdr;
    sort_by_work(U.work_adj.begin(), U.work_adj.end(), 20);
    // whether every particle and tree node is some parent's child (each then has its own gradient
    // written by exactly one record)
    U.complete = children[0] == X.np && children[1] == X.nt;
}

}  // namespace aprk
