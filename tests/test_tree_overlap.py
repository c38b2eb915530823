"""Layouts that are accepted without validation and in which a cell is a particle and a tree node at once: the
restriction still writes every node and the push-down still passes every node's gradient on, level by level, as
the child maps say (a cell that is both counts as the particle)."""
import dataclasses

import numpy as np
import pytest

import aprsynth as S
import paper_2112_03592_gb300 as G
from paper_2112_03592_gb300 import _abi

INDEX = (1 << 30) - 1


def overlapping(seed):
    """A random APR with particles added on cells that are split (tree nodes)."""
    apr = S.random_balanced_apr((24, 20, 40), 1, seed=seed, p_fine=0.02)
    lay = G.AprLayout.from_apr(apr, flags=G.APR_VALIDATE | G.APR_HOST_ONLY)
    trp, ty = lay.export(_abi.APR_STRUCT_TREE_ROW_PTR), lay.export(_abi.APR_STRUCT_TREE_Y_IDX)
    rng = np.random.default_rng(seed)
    rows = []
    for r in range(len(apr.row_ptr) - 1):
        y = apr.y_idx[apr.row_ptr[r]:apr.row_ptr[r + 1]]
        if r < len(trp) - 1 and rng.random() < 0.3:
            y = np.union1d(y, ty[trp[r]:trp[r + 1]][::2])
        rows.append(y.astype(np.int32))
    y_idx = np.concatenate(rows)
    row_ptr = np.concatenate([[0], np.cumsum([len(y) for y in rows])]).astype(np.int64)
    return dataclasses.replace(apr, row_ptr=row_ptr, y_idx=y_idx, values=rng.random(len(y_idx)).astype(np.float32))


def children(lay):
    """Per node its eight children in [particles, tree nodes], -1 where there is none."""
    m = lay.export(_abi.APR_STRUCT_TREE_NODE_MAP).astype(np.int64) & 0xFFFFFFFF
    c = np.full((len(m), 8), -1)
    for k in range(4):
        pm, tm = m[:, k] >> 30, m[:, 4 + k] >> 30
        for e in range(2):
            p = (m[:, k] & INDEX) + (pm & 1 if e else 0)
            t = (m[:, 4 + k] & INDEX) + (tm & 1 if e else 0) + lay.n_particles
            c[:, 2 * k + e] = np.where((pm >> e) & 1, p, np.where((tm >> e) & 1, t, -1))
    return c


@pytest.mark.gpu
@pytest.mark.parametrize("seed", [1, 2])
def test_every_node_is_written(seed):
    import torch
    apr = overlapping(seed)
    lay = G.AprLayout.from_apr(apr, flags=0)
    kids = children(lay)
    named = set(kids[kids >= lay.n_particles].tolist())
    dz, dx, _ = apr.level_dims(apr.l_min)
    assert len(named) < lay.n_tree - int(lay.export(_abi.APR_STRUCT_TREE_ROW_PTR)[dz * dx])   # some below l_min are no parent's child
    v = torch.as_tensor(apr.values, device="cuda")
    # the next finer level's nodes come later in tree order
    val = np.concatenate([apr.values.astype(np.float64), np.zeros(lay.n_tree)])
    for n in range(lay.n_tree - 1, -1, -1):
        val[lay.n_particles + n] = val[kids[n][kids[n] >= 0]].mean()
    tree = torch.full((lay.n_tree,), float("nan"), device="cuda")
    G.apr_tree_restrict(lay, v, tree)
    assert np.abs(tree.cpu().numpy() - val[lay.n_particles:]).max() <= 2e-6      # a few roundings of means below 1
    tb = torch.full((lay.n_tree, 16), float("nan"), dtype=torch.bfloat16, device="cuda")
    G.apr_tree_restrict_bf16(lay, v[:, None].expand(-1, 16).contiguous().to(torch.bfloat16), tb)
    assert np.abs(tb.float().cpu().numpy() - val[lay.n_particles:, None]).max() <= 0.05   # a bf16 rounding per level
    g = np.concatenate([np.zeros(lay.n_particles), np.random.default_rng(0).random(lay.n_tree)])
    gt = torch.as_tensor(g[lay.n_particles:].astype(np.float32), device="cuda")
    gp = torch.zeros_like(v)
    G.apr_tree_restrict_adjoint(lay, gt, gp)
    for n in range(lay.n_tree):
        k = kids[n][kids[n] >= 0]
        g[k] += g[lay.n_particles + n] / len(k)
    assert np.abs(gp.cpu().numpy() - g[:lay.n_particles]).max() <= 2e-5 * max(1.0, np.abs(g).max())
