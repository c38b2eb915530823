"""Richardson-Lucy in one call, whose kernels start while the launch before them finishes and whose estimate is read and
overwritten by them, gives the bits of its steps called one by one with synchronisations between them, and as
a CUDA graph."""
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


@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("k", [3, 5])
@pytest.mark.parametrize("case", list(CASES))
def test_one_call_equals_its_steps(case, k, bc):
    apr = CASES[case]()
    lay = G.AprLayout.from_apr(apr, G.APR_VALIDATE | G.APR_REQUIRE_BALANCE)
    rng = np.random.default_rng(k)
    f = lambda *shape: torch.as_tensor((rng.random(size=shape) + 0.1).astype(np.float32), device="cuda")
    u, st = f(apr.n_particles), f(apr.n_levels, k ** 3) / k ** 3
    flipped = st.flip(1).contiguous()

    def conv(x, w):
        torch.cuda.synchronize()
        tree = G.apr_tree_restrict(lay, x)
        torch.cuda.synchronize()
        out = G.apr_convolve(lay, x, tree, w, k, bc)
        torch.cuda.synchronize()
        return out

    ref = u.clone()
    for _ in range(4):
        ref = ref * conv(u / conv(ref, st), flipped)
    for _ in range(3):
        assert torch.equal(G.apr_richardson_lucy(lay, u, st, k, 4, bc), ref)
    est = torch.empty_like(u)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        est.copy_(u)
        G.apr_richardson_lucy(lay, u, st, k, 4, bc, estimate=est)
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(est, ref)
