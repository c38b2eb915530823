"""Multi-channel convolution on units, at the sizes and alignments where its tiles can go wrong, vs the oracle.

Features, gradients and weights are multiples of 1/8 and 1/16 below 8 and 1 (exact in bfloat16), tree values
bfloat16 averages of them: the oracle sees the GPU's inputs exactly. Products of features and weights are
multiples of 2^-7 (tree values: a few bits more) and a sum of 432 of them stays below 2^24 of these units, so
FP32 accumulation in any order is exact or within a few roundings of 2^-24; 1e-5 of the largest value, the
bound of the other multi-channel tests, is far above that and far below one missing tap (about 1e-3).
"""
import numpy as np
import pytest
import torch

import aprsynth as S
import oracle
import paper_2112_03592_gb300 as G

pytestmark = pytest.mark.gpu
FLAGS = G.APR_VALIDATE | G.APR_REQUIRE_BALANCE
C = 16
NORM = 1e-5

CASES = {
    "odd_ends": lambda: S.random_balanced_apr((21, 19, 75), 2, seed=5, p_fine=0.2),
    "plane": lambda: S.random_balanced_apr((1, 37, 90), 1, seed=14, p_fine=0.03),
    "row": lambda: S.random_balanced_apr((1, 1, 67), 0, seed=8, p_fine=0.1),
    "three_cells": lambda: S.random_balanced_apr((3, 3, 3), 0, seed=4, p_fine=0.5),
    "tiles_of_128": lambda: S.uniform_level_apr((17, 20, 33), 6),
    "units_of_128": lambda: S.random_balanced_apr((64, 56, 60), 2, seed=31, p_fine=0.6),
    "units_of_256": lambda: S.uniform_level_apr((87, 88, 86), 7),
}


def bf16(a, offset):
    """a in bfloat16 on the GPU, its first element `offset` values behind a 512-byte boundary."""
    a = np.ascontiguousarray(a, np.float32)
    buf = torch.zeros(a.size + offset, dtype=torch.bfloat16, device="cuda")
    t = buf[offset:].view(a.shape)
    t.copy_(torch.as_tensor(a))
    return t


def assert_norm(got, ref):
    ref = np.asarray(ref, np.float64)
    got = got.cpu().numpy().astype(np.float64)
    assert got.shape == ref.shape and np.isfinite(got).all()
    if ref.size:
        assert np.abs(got - ref).max() <= NORM * max(np.abs(ref).max(), 1e-30)


@pytest.mark.parametrize("case,bc,offset", [(c, bc, 0) for c in CASES for bc in (0, 1) if c != "units_of_256"] +
                         [("units_of_256", 0, 0), ("odd_ends", 0, 8), ("odd_ends", 1, 8), ("tiles_of_128", 0, 8)])
def test_mc_units_match_the_oracle(case, bc, offset):
    apr = CASES[case]()
    rng = np.random.default_rng(len(case) + bc)
    x = rng.integers(-64, 65, size=(apr.n_particles, C)) / 8.0
    w = rng.integers(-16, 17, size=(apr.n_levels, C, C, 27)) / 16.0
    g = rng.integers(-64, 65, size=(apr.n_particles, C)) / 8.0
    lay = G.AprLayout.from_apr(apr, FLAGS)
    xd, gd, wd = bf16(x, offset), bf16(g, offset), bf16(w, 0)
    tree = bf16(np.zeros((lay.n_tree, C)), offset)
    G.apr_tree_restrict_bf16(lay, xd, tree)
    out = G.apr_convolve_mc(lay, xd, tree, wd, bc)
    relu = G.apr_convolve_mc_relu_bf16(lay, xd, tree, wd, bc)
    base = torch.as_tensor(rng.normal(size=apr.n_particles).astype(np.float32), device="cuda")
    read = G.apr_convolve_mc_readout(lay, xd, tree, wd, base, 0.37, bc)
    gp, gw = G.apr_convolve_mc_backward(lay, xd, tree, wd, gd, bc)
    torch.cuda.synchronize()
    lay.sync_status()
    o = oracle.Oracle(apr, x)
    np.testing.assert_array_equal(tree.float().cpu().numpy().astype(np.float64), o.tree_bf16())
    assert_norm(out, o.conv(w, 3, bc, C_out=C))
    ref_gp, ref_gw = o.conv_backward(w, 3, g, bc, C_out=C)
    assert_norm(gp, ref_gp)
    assert_norm(gw, ref_gw)
    assert torch.equal(relu, G.apr_mc_relu_bf16(out))              # the fused writes: the same numbers
    assert torch.equal(read, G.apr_mc_readout(out, base, 0.37))


@pytest.mark.parametrize("n,offset", [(1, 0), (1001, 0), (1001, 8), (1001, 1), (70001, 0)])
def test_element_wise_layers_at_every_alignment(n, offset):
    """16-byte and single-value forms give the same bits: compared with torch's own rounding to bfloat16."""
    gen = torch.Generator().manual_seed(n + offset)

    def buf(shape, dtype):
        m = int(np.prod(shape))
        return torch.empty(m + offset, dtype=dtype, device="cuda")[offset:].view(shape)

    def rand(shape):
        t = buf(shape, torch.float32)
        t.copy_(torch.randn(shape, generator=gen) * 3)
        return t

    x, c, g = rand((n,)), rand((n, C)), rand((n, C))
    c[0, :3] = torch.tensor([float("nan"), float("inf"), -0.0])
    e = torch.zeros((n, C), dtype=torch.float32, device="cuda")
    e[:, 0] = np.float32(0.37) * x
    assert torch.equal(G.apr_mc_embed_bf16(x, float(np.float32(0.37)), buf((n, C), torch.bfloat16)), e.to(torch.bfloat16))
    assert torch.equal(G.apr_mc_readout_backward_bf16(x, float(np.float32(0.37)), buf((n, C), torch.bfloat16)), e.to(torch.bfloat16))
    ref = torch.where(c > 0, c, torch.zeros_like(c)).to(torch.bfloat16)
    assert torch.equal(G.apr_mc_relu_bf16(c, buf((n, C), torch.bfloat16)), ref)
    assert torch.equal(G.apr_mc_relu_bf16(c.view(-1)[:n * C - 5], buf((n * C - 5,), torch.bfloat16)), ref.view(-1)[:n * C - 5])
    ref = torch.where(c > 0, g, torch.zeros_like(g)).to(torch.bfloat16)
    assert torch.equal(G.apr_mc_relu_backward_bf16(c, g, buf((n, C), torch.bfloat16)), ref)


@pytest.mark.parametrize("bc", [0, 1])
def test_outputs_at_16_byte_alignment_are_the_same_bits(bc):
    """32-byte stores where the outputs allow them, 16-byte stores else: the same numbers."""
    apr = CASES["odd_ends"]()
    rng = np.random.default_rng(9)
    lay = G.AprLayout.from_apr(apr, FLAGS)
    x, g = (bf16(rng.integers(-64, 65, size=(apr.n_particles, C)) / 8.0, 0) for _ in range(2))
    w = bf16(rng.integers(-16, 17, size=(apr.n_levels, C, C, 27)) / 16.0, 0)
    tree = G.apr_tree_restrict_bf16(lay, x)

    def at(offset, dtype):
        return torch.empty(apr.n_particles * C + offset, dtype=dtype, device="cuda")[offset:].view(apr.n_particles, C)

    res = []
    for o32, o16 in ((0, 0), (4, 8)):
        res.append((G.apr_convolve_mc(lay, x, tree, w, bc, out=at(o32, torch.float32)),
                    G.apr_convolve_mc_relu_bf16(lay, x, tree, w, bc, out=at(o16, torch.bfloat16)),
                    G.apr_convolve_mc_backward(lay, x, tree, w, g, bc, need_weights=False, grad_particles=at(o32, torch.float32))[0]))
    for a, b in zip(*res):
        assert torch.equal(a, b)
