"""Tree restriction and push-down in groups of levels: deep and shallow trees (one to nine tree levels, so
groups of one to four levels and several groups), odd grids whose nodes miss children, against the oracle."""
import numpy as np
import pytest

import aprsynth as S
import oracle
import paper_2112_03592_gb300 as G

pytestmark = pytest.mark.gpu

CASES = {
    "one_level": lambda: S.random_balanced_apr((8, 8, 8), 2, seed=1, p_fine=0.1),
    "nine_levels": lambda: S.random_balanced_apr((1, 3, 300), 0, seed=2, p_fine=0.02),
    "odd_deep": lambda: S.random_balanced_apr((33, 47, 70), 0, seed=3, p_fine=0.01),
    "split_groups": lambda: S.random_balanced_apr((96, 96, 128), 3, seed=4, p_fine=0.02),
    "no_tree": lambda: S.uniform_level_apr((9, 9, 9), 4),
}


@pytest.mark.parametrize("case", list(CASES))
def test_tree_groups(case):
    import torch
    apr = CASES[case]()
    lay = G.AprLayout.from_apr(apr)
    rng = np.random.default_rng(0)
    v = torch.as_tensor(apr.values, device="cuda")
    ref = oracle.Oracle(apr).tree()[:, 0]
    tree = G.apr_tree_restrict(lay, v)
    # each level averages eight values in FP32: a few rounding errors of 2^-24 per level
    assert np.all(np.abs(tree.cpu().numpy() - ref) <= 2e-6 * np.abs(ref))
    x = (rng.integers(-64, 65, size=(apr.n_particles, 16)) / 8.0).astype(np.float32)
    xb = torch.as_tensor(x, device="cuda").to(torch.bfloat16)
    tb = G.apr_tree_restrict_bf16(lay, xb)
    assert np.array_equal(tb.float().cpu().numpy().astype(np.float64), oracle.Oracle(apr, x.astype(np.float64)).tree_bf16())
    # push-down is the transpose: <t, restrict(x)> = <push(t), x>, summed in FP64
    t = torch.as_tensor(rng.normal(size=lay.n_tree).astype(np.float32), device="cuda")
    gp = torch.zeros_like(v)
    G.apr_tree_restrict_adjoint(lay, t.clone(), gp)
    a, b = (t.double() * torch.as_tensor(ref, device="cuda")).sum(), (gp.double() * v.double()).sum()
    scale = (t.double().abs() * torch.as_tensor(np.abs(ref), device="cuda")).sum() + 1e-30
    assert abs(float(a - b)) <= 1e-6 * float(scale)
