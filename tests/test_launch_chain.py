"""Kernels that start while the launch before them finishes: a chain of calls that feed one another through the same
buffers gives the same bits as the calls one by one, and as the chain captured in a CUDA graph."""
import numpy as np
import pytest
import torch

import aprsynth as S
import paper_2112_03592_gb300 as G

pytestmark = pytest.mark.gpu

CASES = {
    "tiny": lambda: S.random_balanced_apr((2, 3, 5), 0, seed=9, p_fine=0.3),
    "ragged": lambda: S.random_balanced_apr((33, 47, 70), 1, seed=3, p_fine=0.01),
    "waves": lambda: S.uniform_level_apr((120, 120, 120), 7, l_min=6),
}


@pytest.mark.parametrize("k", [3, 5])
@pytest.mark.parametrize("case", list(CASES))
def test_chained_calls_equal_synchronised_ones(case, k):
    apr = CASES[case]()
    lay = G.AprLayout.from_apr(apr, G.APR_VALIDATE | G.APR_REQUIRE_BALANCE)
    rng = np.random.default_rng(k)
    f = lambda shape: torch.as_tensor(rng.normal(size=shape).astype(np.float32), device="cuda")
    x0, st = f(apr.n_particles), f((apr.n_levels, k ** 3)) / k ** 1.5
    x = x0.clone()
    st_t, y, g = st.clone(), torch.empty_like(x), torch.empty_like(x)
    tree = torch.empty(max(lay.n_tree, 1), device="cuda")[:lay.n_tree]
    gt = torch.empty_like(tree)

    def step(pause):
        G.apr_tree_restrict(lay, x, tree)
        pause()
        G.apr_convolve(lay, x, tree, st_t, k, out=y)
        pause()
        G.apr_convolve_adjoint(lay, st_t, k, y, grad_particles=g, grad_tree=gt)
        pause()
        G.apr_tree_restrict_adjoint(lay, gt, g)
        pause()
        G.apr_tree_restrict(lay, g, tree)
        pause()
        G.apr_gradient_magnitude(lay, g, tree, torch.cat([st_t, st_t, st_t]), k, out=x)
        pause()
        x.mul_(1.0 / x.abs().max().clamp_min(1e-20))
        st_t.neg_()

    def run(pause):
        x.copy_(x0)
        st_t.copy_(st)
        for _ in range(6):
            step(pause)
        torch.cuda.synchronize()
        return x.clone()

    ref = run(torch.cuda.synchronize)
    for _ in range(3):
        assert torch.equal(run(lambda: None), ref)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step(lambda: None)
    x.copy_(x0)
    st_t.copy_(st)
    for _ in range(6):
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(x, ref)
