"""Convolution units (the parent groups the convolution kernels compute from), on the host.

The units of a host-only handle are decoded and the kernels' arithmetic is repeated from them in numpy
(octets staged per slot, taps read through the records' row slots) in FP64, against the oracle: a wrong
slot, source, mirror or missing bit gives a wrong sum. The coarse-source records are checked through
the transpose: what the forward sums read from a level-(l-1) particle is what its record lists.
"""
import numpy as np
import pytest

import aprsynth as S
import oracle
import paper_2112_03592_gb300 as G
from paper_2112_03592_gb300 import _abi

HOST = G.APR_VALIDATE | G.APR_REQUIRE_BALANCE | G.APR_HOST_ONLY
INDEX = (1 << 30) - 1

CASES = {
    "blob64": lambda: S.make_config("blob64"),
    "ragged": lambda: S.random_balanced_apr((33, 47, 70), 1, seed=3, p_fine=0.01),
    "odd_fine": lambda: S.random_balanced_apr((21, 19, 75), 2, seed=5, p_fine=0.2),
    "thin": lambda: S.random_balanced_apr((2, 3, 97), 1, seed=6, p_fine=0.05),
    "plane": lambda: S.random_balanced_apr((1, 37, 90), 1, seed=14, p_fine=0.03),
    "row": lambda: S.random_balanced_apr((1, 1, 67), 0, seed=8, p_fine=0.1),
    "uniform_fine": lambda: S.uniform_level_apr((17, 20, 33), 6),
    "uniform_coarse": lambda: S.uniform_level_apr((40, 40, 40), 4),
    "one": lambda: S.uniform_level_apr((1, 1, 1), 0),
}


def decode_pure(e):
    """Slot numbers and the eight particles of pure entries."""
    slot = sum((e[:, k] >> 28) << (4 * k) for k in range(4))
    first = e & 0x0FFFFFFF
    return slot, np.stack([first[:, k] + b for k in range(4) for b in range(2)], axis=1)


class Units:
    def __init__(self, apr):
        self.apr = apr
        lay = G.AprLayout.from_apr(apr, flags=HOST)
        self.n_p, self.n_t = lay.n_particles, lay.n_tree
        ex = lambda n: lay.export(getattr(_abi, "APR_STRUCT_" + n))
        for n in ("hdr", "pure", "node", "node_info", "rec"):
            setattr(self, n, ex("UNIT_" + n.upper()))
            setattr(self, "l" + n, ex("LEAF_" + n.upper()))
        self.other = ex("UNIT_OTHER").astype(np.int64)
        self.child = self.decode_map(np.concatenate([ex("TREE_NODE_MAP"), ex("UNIT_MAP")]))

    def decode_map(self, maps):
        """Index of every child in [particles, tree nodes, 0-value], absent children last."""
        maps = maps.astype(np.int64) & 0xFFFFFFFF
        none = self.n_p + self.n_t
        child = np.full((len(maps), 8), none)
        for k in range(4):
            pm, tm = maps[:, k] >> 30, maps[:, 4 + k] >> 30
            for e in range(2):
                p = (maps[:, k] & INDEX) + (pm & 1 if e else 0)
                t = (maps[:, 4 + k] & INDEX) + (tm & 1 if e else 0)
                child[:, 2 * k + e] = np.where((pm >> e) & 1, p, np.where((tm >> e) & 1, self.n_p + t, none))
        return child

    def octets(self, h, bc):
        """Source index (into [particles, tree, zero]) of the 8 cells of every slot of unit h."""
        pure0, node0, oth0, _, npure, nn, nl, noth = (int(v) for v in h[:8])
        none = self.n_p + self.n_t
        oth = self.other[oth0:oth0 + noth]
        src = np.full((nn + noth, 8), none)
        src[:nn] = self.decode_map(self.node[node0:node0 + nn])
        src[nn:nn + nl] = oth[:nl, 0][:, None]
        info = np.concatenate([self.node_info[node0:node0 + nn].astype(np.int64), oth[:, 1]])
        mir, miss = (info >> 16) & 7, (info >> 20) & 7
        c = np.arange(8)
        for m in (1, 2, 4):
            src = np.where(((miss & m) != 0)[:, None] & ((c & m) != 0)[None], src[:, c ^ m] if bc == 0 else none, src)
        if bc == 1:
            src[mir != 0] = none
        for m in (1, 2, 4):
            src = np.where(((mir & m) != 0)[:, None], src[:, c ^ m], src)
        out = np.full((nn + noth + npure, 8), -1)
        out[info & 0x7FF] = src
        slot, kids = decode_pure(self.pure[pure0:pure0 + npure].astype(np.int64))
        out[slot] = kids
        assert (out >= 0).all()
        return out

    def forward_sources(self, bc, R):
        """(records' children [n, 8], level [n], source index of every tap [n, 8, K, K, K])."""
        kids, lev, taps = [], [], []
        for h in self.hdr:
            slots = self.octets(h, bc)
            nrec = int(h[8])
            rec = self.rec[h[3]:h[3] + nrec].astype(np.int64)
            node = rec[:, 0] | (rec[:, 1] << 16)
            base = rec[:, 3:12]
            cells = np.empty((nrec, 6, 6, 6), np.int64)   # cells -2 .. 3 per axis around the record
            for z in range(6):
                for x in range(6):
                    for y in range(6):
                        s = base[:, (z >> 1) * 3 + (x >> 1)] + (y >> 1)
                        cells[:, z, x, y] = slots[s, (z & 1) * 4 + (x & 1) * 2 + (y & 1)]
            K = 2 * R + 1
            t = np.empty((nrec, 8, K, K, K), np.int64)
            for c in range(8):
                z, x, y = 2 + (c >> 2) - R, 2 + ((c >> 1) & 1) - R, 2 + (c & 1) - R
                t[:, c] = cells[:, z:z + K, x:x + K, y:y + K]
            kids.append(self.child[node])
            lev.append(np.full(nrec, h[10]))
            taps.append(t)
        return np.concatenate(kids), np.concatenate(lev), np.concatenate(taps)


@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("case", list(CASES))
def test_units_reproduce_the_convolution(case, bc):
    apr = CASES[case]()
    u = Units(apr)
    o = oracle.Oracle(apr)
    src = np.concatenate([apr.values.astype(np.float64), o.tree()[:, 0], [0.0]])
    rng = np.random.default_rng(0)
    for R in (1, 2):
        k = 2 * R + 1
        st = rng.normal(size=(apr.n_levels, k ** 3))
        kids, lev, taps = u.forward_sources(bc, R)
        # every particle and tree node is the child of exactly one record
        own = kids[kids < u.n_p + u.n_t]
        assert np.array_equal(np.sort(own), np.arange(u.n_p + u.n_t))
        out = np.einsum("ncabd,nabd->nc", src[taps], st[lev].reshape(-1, k, k, k))
        got = np.full(u.n_p, np.nan)
        isp = kids < u.n_p
        got[kids[isp]] = out[isp]
        ref = o.conv(st, k, bc=bc)[:, 0]
        assert np.max(np.abs(got - ref)) <= 1e-11 * np.max(np.abs(ref))


@pytest.mark.parametrize("case", ["blob64", "ragged", "odd_fine", "thin"])
def test_leaf_records_list_the_coarse_sources(case):
    """A level-(l-1) particle that forward sums read as a coarse source has one record; its slots are the
    nodes whose records read it."""
    apr = CASES[case]()
    u = Units(apr)
    readers = {}
    for h in u.hdr:
        leaf = u.other[h[2]:h[2] + h[6]]
        slot_of = {int(e[1]) & 0x7FF: int(e[0]) for e in leaf if (int(e[1]) >> 16) & 7 == 0}
        for r in u.rec[h[3]:h[3] + h[8]].astype(np.int64):
            node = int(r[0] | (r[1] << 16))
            for q in range(9):
                for j in range(3):
                    if int(r[3 + q]) + j in slot_of:
                        readers.setdefault(slot_of[int(r[3 + q]) + j], []).append((26 - (3 * q + j), node))
    got = {}
    node_of = {tuple(k): i for i, k in enumerate(u.child)}
    for h in u.lhdr:
        maps = u.decode_map(u.lnode[h[1]:h[1] + h[5]])
        node_at = {int(i) & 0x7FF: node_of[tuple(k)] for i, k in zip(u.lnode_info[h[1]:h[1] + h[5]], maps)}
        slot, kids = decode_pure(u.lpure[h[0]:h[0] + h[4]].astype(np.int64))
        node_at.update((int(s), node_of[tuple(k)]) for s, k in zip(slot, kids))
        assert sorted(node_at) == list(range(h[4] + h[5]))
        for r in u.lrec[h[3]:h[3] + h[8]].astype(np.int64):
            p, mask = int(r[0] | (r[1] << 16)), int(r[2] | (r[3] << 16))
            lst = []
            for q in range(9):
                m = (mask >> (3 * q)) & 7
                for j in range(3):
                    if (m >> j) & 1:
                        lst.append((3 * q + j, node_at[int(r[5 + q]) + bin(m & ((1 << j) - 1)).count("1")]))
            assert p not in got
            got[p] = sorted(lst)
    assert got == {p: sorted(v) for p, v in readers.items()}


# ---- on the GPU: unit boundaries (64, 128 and 256 records per unit; units cut by the slot limit) and the
# images of records and coarse sources at odd, even and one-cell grid ends, against the oracle
GPU_CASES = {
    "sparse": lambda: S.random_balanced_apr((70, 90, 110), 3, seed=31, p_fine=0.0006),      # isolated parents: slot limit
    "units_of_128": lambda: S.random_balanced_apr((64, 80, 96), 2, seed=32, p_fine=0.01),
    "odd_ends": lambda: S.random_balanced_apr((23, 45, 67), 1, seed=33, p_fine=0.02),
    "one_cell_ends": lambda: S.random_balanced_apr((1, 2, 35), 0, seed=34, p_fine=0.2),
    "three_cells": lambda: S.random_balanced_apr((3, 5, 6), 0, seed=35, p_fine=0.3),
    "one": CASES["one"],
}


@pytest.mark.gpu
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("k", [3, 5])
@pytest.mark.parametrize("case", list(GPU_CASES))
def test_unit_kernels_match_the_oracle(case, k, bc):
    """Forward, data adjoint and stencil gradient with taps on every level, to FP32 rounding: the sums have
    at most a few hundred terms of random sign (bound 1e-5 of the largest entry, as the other parity tests)."""
    import torch
    apr = GPU_CASES[case]()
    rng = np.random.default_rng(2)
    st = (rng.normal(size=(apr.n_levels, k ** 3)) / k ** 3).astype(np.float32)
    g = rng.normal(size=apr.n_particles).astype(np.float32)
    dev = lambda a: torch.as_tensor(a, device="cuda")
    lay = G.AprLayout.from_apr(apr)
    v = dev(apr.values)
    tree = G.apr_tree_restrict(lay, v)
    out = G.apr_convolve(lay, v, tree, dev(st), k, bc)
    gp, gw = G.apr_convolve_backward(lay, v, tree, dev(st), k, dev(g), bc)
    o = oracle.Oracle(apr)
    ref = o.conv(st.astype(np.float64), k, bc=bc)[:, 0]
    rp, rw = o.conv_backward(st.astype(np.float64), k, g.astype(np.float64), bc=bc)
    for got, want in ((out, ref), (gp, rp[:, 0]), (gw, rw.reshape(gw.shape))):
        assert np.max(np.abs(got.cpu().numpy() - want)) <= 1e-5 * np.max(np.abs(want))
    # the same through work-item ranges: forward outputs bit for bit, the adjoint's terms summed in halves
    items = lay.export(_abi.APR_STRUCT_FWD_ITEMS)
    part = torch.zeros_like(out)
    for a, b in ((0, len(items) // 2), (len(items) // 2, len(items))):
        G.apr_convolve_tiles(lay, v, tree, dev(st), k, a, b - a, bc, part)
    assert torch.equal(part, out)
    n = len(lay.export(_abi.APR_STRUCT_BWD_ITEMS))
    tp, tt = torch.zeros_like(v), torch.zeros(lay.n_tree, device="cuda")
    for a, b in ((0, n // 2), (n // 2, n)):
        G.apr_convolve_adjoint_tiles(lay, dev(st), k, dev(g), tp, tt, a, b - a, bc)
    G.apr_tree_restrict_adjoint(lay, tt, tp)
    assert np.max(np.abs(tp.cpu().numpy() - rp[:, 0])) <= 1e-5 * np.max(np.abs(rp))
