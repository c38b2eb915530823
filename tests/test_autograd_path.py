"""AprConv equals the calls it stands for, bit for bit: with and without tree nodes, on the current stream."""
import numpy as np
import pytest
import torch

import aprsynth as S
import paper_2112_03592_gb300 as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side_stream", [False, True])
@pytest.mark.parametrize("case", ["no_tree", "ragged"])
def test_autograd_equals_the_separate_calls(case, side_stream):
    apr = S.uniform_level_apr((9, 8, 10), 4, l_min=4) if case == "no_tree" else S.random_balanced_apr((21, 13, 50), 1, seed=7, p_fine=0.05)
    lay = G.AprLayout.from_apr(apr, G.APR_VALIDATE | G.APR_REQUIRE_BALANCE)
    assert (lay.n_tree == 0) == (case == "no_tree")
    rng = np.random.default_rng(3)
    st = torch.cuda.Stream() if side_stream else torch.cuda.current_stream()
    f = lambda shape: torch.as_tensor(rng.normal(size=shape).astype(np.float32), device="cuda")
    x, w, g = f(apr.n_particles), f((apr.n_levels, 3, 3, 3)), f(apr.n_particles)
    tree = G.apr_tree_restrict(lay, x)
    ref = G.apr_convolve(lay, x, tree, w, 3)
    gx, gw = G.apr_convolve_backward(lay, x, tree, w, 3, g)
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        xr, wr = x.clone().requires_grad_(), w.clone().requires_grad_()
        out = G.AprConv.apply(xr, wr, lay, 3)
        dx, dw = torch.autograd.grad(out, (xr, wr), g)
    torch.cuda.synchronize()
    assert torch.equal(out, ref) and torch.equal(dx, gx)
    assert dw.shape == w.shape and torch.equal(dw.view_as(gw), gw)
