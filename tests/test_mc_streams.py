"""Multi-channel calls share nothing but the handle's read-only index: calls with different weights on two streams at
the same time, and a chain that follows itself through reused buffers, give the bits of calls one by one. (Each
block lays the weights out for itself; through a buffer of the handle one call's weights reached the other.)"""
import numpy as np
import pytest
import torch

import aprsynth as S
import paper_2112_03592_gb300 as G

pytestmark = pytest.mark.gpu
C = 16
CASES = {
    "waves": lambda: S.uniform_level_apr((87, 88, 86), 7),                                # several waves of blocks
    "levels": lambda: S.random_balanced_apr((64, 56, 60), 2, seed=31, p_fine=0.1),
}


def inputs(apr, seed):
    rng = np.random.default_rng(seed)
    bf = lambda *shape: torch.as_tensor(rng.normal(size=shape).astype(np.float32), device="cuda").to(torch.bfloat16)
    return bf(apr.n_particles, C), bf(apr.n_particles, C), bf(apr.n_levels, C, C, 27)


def step(lay, x, g, w):
    tree = G.apr_tree_restrict_bf16(lay, x)
    return (G.apr_convolve_mc(lay, x, tree, w), G.apr_convolve_mc_relu_bf16(lay, x, tree, w),
            *G.apr_convolve_mc_backward(lay, x, tree, w, g, need_weights=False)[:1])


@pytest.mark.parametrize("case", list(CASES))
def test_two_streams_with_different_weights(case):
    apr = CASES[case]()
    lay = G.AprLayout.from_apr(apr, G.APR_VALIDATE | G.APR_REQUIRE_BALANCE)
    data = [inputs(apr, 1), inputs(apr, 2)]
    ref = [step(lay, *d) for d in data]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(5):
        got = []
        for _ in range(3):
            for s, d in zip(streams, data):
                with torch.cuda.stream(s):
                    got.append(step(lay, *d))
        torch.cuda.synchronize()
        for i, res in enumerate(got):
            assert all(torch.equal(a, b) for a, b in zip(res, ref[i % 2]))
    lay.sync_status()


@pytest.mark.parametrize("offset", [0, 1, 8])
def test_weights_at_any_alignment(offset):
    apr = CASES["levels"]()
    lay = G.AprLayout.from_apr(apr, G.APR_VALIDATE | G.APR_REQUIRE_BALANCE)
    x, g, w = inputs(apr, 3)
    buf = torch.empty(w.numel() + offset, dtype=torch.bfloat16, device="cuda")
    shifted = buf[offset:].view(w.shape)
    shifted.copy_(w)
    assert all(torch.equal(a, b) for a, b in zip(step(lay, x, g, shifted), step(lay, x, g, w)))


@pytest.mark.parametrize("case", list(CASES))
def test_chained_calls_equal_synchronised_ones(case):
    """Restriction, two convolutions with different weights through the same buffers, then the backward with the first
    weights, whose gradients make the next step's features: one by one, unsynchronised, and as a CUDA graph."""
    apr = CASES[case]()
    lay = G.AprLayout.from_apr(apr, G.APR_VALIDATE | G.APR_REQUIRE_BALANCE)
    x0, g0, w1 = inputs(apr, 4)
    w2 = inputs(apr, 5)[2]
    x, g = x0.clone(), g0.clone()
    tree = torch.empty((lay.n_tree, C), dtype=torch.bfloat16, device="cuda")
    h, c = torch.empty_like(x), torch.empty((apr.n_particles, C), device="cuda")
    gp, gw = torch.empty_like(c), torch.empty(apr.n_levels, C, C, 27, device="cuda")

    def run_step(pause):
        for call in (lambda: G.apr_tree_restrict_bf16(lay, x, tree), lambda: G.apr_convolve_mc_relu_bf16(lay, x, tree, w1, out=h),
                     lambda: G.apr_tree_restrict_bf16(lay, h, tree), lambda: G.apr_convolve_mc(lay, h, tree, w2, out=c),
                     lambda: G.apr_tree_restrict_bf16(lay, x, tree),
                     lambda: G.apr_convolve_mc_backward(lay, x, tree, w1, g, grad_particles=gp, grad_weights=gw)):
            call()
            pause()
        x.copy_(gp / gp.abs().max().clamp_min(1e-20))
        g.copy_(c / c.abs().max().clamp_min(1e-20))
        w1.copy_(gw / gw.abs().max().clamp_min(1e-20))

    start = (x0.clone(), g0.clone(), w1.clone())

    def run(pause, n=4):
        for t, s in zip((x, g, w1), start):
            t.copy_(s)
        for _ in range(n):
            run_step(pause)
        torch.cuda.synchronize()
        return [t.clone() for t in (x, g, w1, gw)]

    ref = run(torch.cuda.synchronize)
    for _ in range(3):
        assert all(torch.equal(a, b) for a, b in zip(run(lambda: None), ref))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run_step(lambda: None)
    for t, s in zip((x, g, w1), start):
        t.copy_(s)
    for _ in range(4):
        graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip((x, g, w1, gw), ref))
    lay.sync_status()
