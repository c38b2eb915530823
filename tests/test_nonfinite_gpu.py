"""Infinities and NaN reach exactly the outputs and gradients that read them: a kernel that computes cells no
particle asks for must not multiply them into what it keeps. One value (or gradient) is not finite; the
oracle sums each target's own terms only, so its non-finite entries are the ones allowed. The other entries
agree to 1e-5 of their largest, the bound of the parity tests.
"""
import numpy as np
import pytest
import torch

import aprsynth as S
import oracle
import paper_2112_03592_gb300 as G

pytestmark = pytest.mark.gpu
C = 16
CASES = {
    "blob64": lambda: S.make_config("blob64"),
    "odd": lambda: S.random_balanced_apr((37, 42, 75), 2, seed=5, p_fine=0.05),
}


def assert_same(got, ref):
    got, ref = got.double().cpu().numpy().reshape(ref.shape), np.asarray(ref)
    fin = np.isfinite(ref)
    assert not fin.all() and fin.any()
    assert np.array_equal(np.isfinite(got), fin)
    assert np.abs(got[fin] - ref[fin]).max() <= 1e-5 * np.abs(ref[fin]).max()


def setup(case, seed):
    apr = CASES[case]()
    rng = np.random.default_rng(seed)
    at = apr.n_particles - 1 - int(rng.integers(apr.n_particles // 2))   # of the finest levels
    return apr, rng, at, G.AprLayout.from_apr(apr, G.APR_VALIDATE | G.APR_REQUIRE_BALANCE)


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, np.float32), device="cuda")


def single_channel(case, k, bc, bad):
    apr, rng, at, lay = setup(case, k + bc)
    v = rng.normal(size=apr.n_particles).astype(np.float32)
    g = rng.normal(size=apr.n_particles).astype(np.float32)
    st = (rng.normal(size=(apr.n_levels, k ** 3)) / k ** 1.5).astype(np.float32)
    vb, gb = v.copy(), g.copy()
    vb[at], gb[at] = bad, bad
    return apr, lay, v, vb, g, gb, st, oracle.Oracle(apr, vb.astype(np.float64))


SINGLE = [pytest.mark.parametrize("bad", [np.inf, np.nan]), pytest.mark.parametrize("bc", [0, 1]),
          pytest.mark.parametrize("k", [3, 5]), pytest.mark.parametrize("case", list(CASES))]


def single(test):
    for mark in SINGLE:
        test = mark(test)
    return test


@single
def test_convolution(case, k, bc, bad):
    apr, lay, v, vb, g, gb, st, o = single_channel(case, k, bc, bad)
    out = G.apr_convolve(lay, dev(vb), G.apr_tree_restrict(lay, dev(vb)), dev(st), k, bc)
    assert_same(out, o.conv(st.astype(np.float64), k, bc=bc)[:, 0])


@single
def test_stencil_gradient(case, k, bc, bad):
    apr, lay, v, vb, g, gb, st, o = single_channel(case, k, bc, bad)
    _, rw = o.conv_backward(st.astype(np.float64), k, g.astype(np.float64), bc=bc)
    assert_same(G.apr_convolve_stencil_grad(lay, dev(vb), G.apr_tree_restrict(lay, dev(vb)), k, dev(g), bc), rw)


@single
def test_data_adjoint(case, k, bc, bad):
    apr, lay, v, vb, g, gb, st, o = single_channel(case, k, bc, bad)
    rp, _ = oracle.Oracle(apr, v.astype(np.float64)).conv_backward(st.astype(np.float64), k, gb.astype(np.float64), bc=bc)
    gp, _ = G.apr_convolve_backward(lay, dev(v), G.apr_tree_restrict(lay, dev(v)), dev(st), k, dev(gb), bc)
    assert_same(gp, rp[:, 0])


def multi_channel(case, bc, bad):
    """Features, gradients and weights as in the multi-channel unit tests (exact in bfloat16)."""
    apr, rng, at, lay = setup(case, bc)
    x, g = (rng.integers(-64, 65, size=(apr.n_particles, C)) / 8.0 for _ in range(2))
    w = rng.integers(-16, 17, size=(apr.n_levels, C, C, 27)) / 16.0
    xb, gb = x.copy(), g.copy()
    xb[at, 3], gb[at, 5] = bad, bad
    bf = lambda a: dev(a).to(torch.bfloat16)
    o, good = oracle.Oracle(apr, xb), oracle.Oracle(apr, x)
    o.tree_bf16(), good.tree_bf16()
    return lay, bf, x, xb, g, gb, w, o, good


MULTI = [pytest.mark.parametrize("bad", [np.inf, -np.inf]), pytest.mark.parametrize("bc", [0, 1]),
         pytest.mark.parametrize("case", list(CASES))]


def multi(test):
    for mark in MULTI:
        test = mark(test)
    return test


@multi
def test_multi_channel_convolution(case, bc, bad):
    lay, bf, x, xb, g, gb, w, o, good = multi_channel(case, bc, bad)
    assert_same(G.apr_convolve_mc(lay, bf(xb), G.apr_tree_restrict_bf16(lay, bf(xb)), bf(w), bc), o.conv(w, 3, bc, C_out=C))


@multi
def test_multi_channel_weight_gradient(case, bc, bad):
    lay, bf, x, xb, g, gb, w, o, good = multi_channel(case, bc, bad)
    _, gw = G.apr_convolve_mc_backward(lay, bf(xb), G.apr_tree_restrict_bf16(lay, bf(xb)), bf(w), bf(g), bc)
    assert_same(gw, o.conv_backward(w, 3, g, bc, C_out=C)[1])


@multi
def test_multi_channel_data_adjoint(case, bc, bad):
    lay, bf, x, xb, g, gb, w, o, good = multi_channel(case, bc, bad)
    gp, _ = G.apr_convolve_mc_backward(lay, bf(x), G.apr_tree_restrict_bf16(lay, bf(x)), bf(w), bf(gb), bc)
    assert_same(gp, good.conv_backward(w, 3, gb, bc, C_out=C)[0])
