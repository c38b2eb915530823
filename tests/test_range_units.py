"""Work-item-range calls launch the units that hold records of the range, not those of the whole image.

CPU, from the exported arrays of host-only handles: the span of a work item is the first to the last unit with a
record in it, and no longer than the units of the 32^3 parents (64^3 cells) around the item. GPU: ranges that
start and end anywhere give the whole call's bits.
"""
import numpy as np
import pytest

import aprsynth as S
import paper_2112_03592_gb300 as G
from paper_2112_03592_gb300 import _abi
from test_units import HOST, Units

CASES = {
    "blob64": lambda: S.make_config("blob64"),
    "ragged": lambda: S.random_balanced_apr((33, 47, 70), 1, seed=3, p_fine=0.01),
    "plane": lambda: S.random_balanced_apr((1, 37, 90), 1, seed=14, p_fine=0.03),
    "no_tree": lambda: S.uniform_level_apr((70, 66, 131), 8, l_min=8),
    "blocks": lambda: S.random_balanced_apr((150, 80, 140), 2, seed=8, p_fine=0.01),
}


def particle_coords(apr):
    """(level, z, x, y) of every particle."""
    out, r = [], 0
    for l in range(apr.l_min, apr.l_max + 1):
        dz, dx, _ = apr.level_dims(l)
        n = np.diff(apr.row_ptr[r:r + dz * dx + 1])
        rows = np.repeat(np.arange(dz * dx), n)
        y = apr.y_idx[apr.row_ptr[r]:apr.row_ptr[r + dz * dx]]
        out.append(np.stack([np.full(len(rows), l), rows // dx, rows % dx, y], 1))
        r += dz * dx
    return np.concatenate(out)


def check(spans, item_of_record, unit_of_record, block_of_unit):
    """spans [items][2] against (item, unit) of every record (item -1: none)."""
    first, last = np.full(len(spans), 1 << 30), np.zeros(len(spans), np.int64)
    use = item_of_record >= 0
    np.minimum.at(first, item_of_record[use], unit_of_record[use])
    np.maximum.at(last, item_of_record[use], unit_of_record[use] + 1)
    first[last == 0] = 0
    assert np.array_equal(spans, np.stack([first, last], 1))
    for a, b in spans:      # one block of parents
        assert len({tuple(block_of_unit[u]) for u in range(a, b)}) <= 1


@pytest.mark.parametrize("case", list(CASES))
def test_spans_are_the_units_of_the_items(case):
    apr = CASES[case]()
    u = Units(apr)
    lay = G.AprLayout.from_apr(apr, flags=HOST)
    pos = particle_coords(apr)
    tree = np.full((u.n_t, 4), -1)
    cell = np.concatenate([pos, tree, [[-1] * 4]])      # child coordinates; tree nodes below

    def record_cells(hdr, rec, node_word):
        """(level of the cells, z, x, y of the parent, unit) of every record."""
        rows = []
        for i, h in enumerate(hdr):
            for r in rec[h[3]:h[3] + h[8]].astype(np.int64):
                rows.append((apr.l_min + h[10], *parent(r, node_word), i))
        return np.array(rows).reshape(-1, 5)

    where = {}

    def parent(r, node_word):
        if not node_word:       # leaf record: the level-(l-1) particle is the parent
            return tuple(pos[int(r[0] | (r[1] << 16)), 1:])
        return where[int(r[0] | (r[1] << 16))]

    # a node's place: that of its first child, or (all children nodes) half of that node's
    for n in range(len(u.child) - 1, -1, -1):
        k = u.child[n]
        c = int(np.nonzero(k < u.n_p + u.n_t)[0][0])
        z, x, y = cell[k[c], 1:]
        where[n] = (int(z) // 2, int(x) // 2, int(y) // 2)
        if n < u.n_t:
            cell[u.n_p + n] = (0, *where[n])

    for which, item_sel, hdr, rec, is_node in (("FWD_UNIT_SPANS", "FWD_ITEMS", u.hdr, u.rec, True),
                                               ("BWD_UNIT_SPANS", "BWD_ITEMS", u.hdr, u.rec, True),
                                               ("BWD_LEAF_SPANS", "BWD_ITEMS", u.lhdr, u.lrec, False)):
        spans = lay.export(getattr(_abi, "APR_STRUCT_" + which))
        items = lay.export(getattr(_abi, "APR_STRUCT_" + item_sel))
        index = {tuple(t): i for i, t in enumerate(items.tolist())}
        R = record_cells(hdr, rec, is_node)
        item = np.array([index.get((l, z // 4, x // 4, y // 32), -1) for l, z, x, y, _ in R], np.int64)
        blocks = {}
        for l, z, x, y, i in R:
            blocks.setdefault(i, (l, z // 32, x // 32, y // 32))
            assert blocks[i] == (l, z // 32, x // 32, y // 32)
        check(spans, item, R[:, 4] if len(R) else np.zeros(0, np.int64), blocks)


@pytest.mark.gpu
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("k", [3, 5])
@pytest.mark.parametrize("case", list(CASES))
def test_ranges_give_the_whole_calls_bits(case, k, bc):
    import torch
    apr = CASES[case]()
    lay = G.AprLayout.from_apr(apr)
    rng = np.random.default_rng(k)
    f = lambda *shape: torch.as_tensor(rng.normal(size=shape).astype(np.float32), device="cuda")
    v, g, st = f(apr.n_particles), f(apr.n_particles), f(apr.n_levels, k ** 3)
    tree = G.apr_tree_restrict(lay, v)
    out = G.apr_convolve(lay, v, tree, st, k, bc)
    gp, gt = G.apr_convolve_adjoint(lay, st, k, g, bc)
    cuts = lambda n: sorted({0, n, 1, max(n - 1, 0), *rng.integers(0, n + 1, size=5).tolist()})
    part = torch.full_like(out, float("nan"))
    c = cuts(len(lay.export(_abi.APR_STRUCT_FWD_ITEMS)))
    for a, b in zip(c, c[1:]):
        G.apr_convolve_tiles(lay, v, tree, st, k, a, b - a, bc, part)
    G.apr_convolve_tiles(lay, v, tree, st, k, c[-1], 0, bc, part)      # an empty range
    assert torch.equal(part, out)
    tp, tt = torch.zeros_like(v), torch.zeros(lay.n_tree, device="cuda")
    c = cuts(len(lay.export(_abi.APR_STRUCT_BWD_ITEMS)))
    for a, b in zip(c, c[1:]):
        G.apr_convolve_adjoint_tiles(lay, st, k, g, tp, tt, a, b - a, bc)
    assert torch.equal(tp, gp)      # two terms per particle, in either order
    assert torch.equal(tt, gt)
