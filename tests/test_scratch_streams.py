"""The scratch that the Python calls bring belongs to the call and its stream: calls with different inputs on two
streams at the same time give the bits of calls one by one, and memory dropped by a call on another stream
(stream=...) is not handed out on the current one while the call still runs."""
import numpy as np
import pytest
import torch

import aprsynth as S
import paper_2112_03592_gb300 as G

pytestmark = pytest.mark.gpu
K = 3


def setup():
    apr = S.random_balanced_apr((64, 56, 60), 2, seed=31, p_fine=0.1)
    lay = G.AprLayout.from_apr(apr, G.APR_VALIDATE | G.APR_REQUIRE_BALANCE)
    rng = np.random.default_rng(0)
    f = lambda *shape: torch.as_tensor(rng.random(size=shape).astype(np.float32) + 0.1, device="cuda")
    st = f(apr.n_levels, K ** 3) / K ** 3
    w = f(apr.n_levels, 16, 16, 27).to(torch.bfloat16)
    data = []
    for _ in range(2):
        v = f(apr.n_particles)
        x = f(apr.n_particles, 16).to(torch.bfloat16)
        data.append((v, G.apr_tree_restrict(lay, v), f(apr.n_particles), x, G.apr_tree_restrict_bf16(lay, x)))
    torch.cuda.synchronize()
    return lay, st, w, data


CALLS = {
    "auto": lambda lay, st, w, v, tree, g, x, tb, s: [G.apr_convolve_auto(lay, v, st, K, stream=s)],
    "richardson_lucy": lambda lay, st, w, v, tree, g, x, tb, s: [G.apr_richardson_lucy(lay, v, st, K, 3, stream=s)],
    "backward": lambda lay, st, w, v, tree, g, x, tb, s: list(G.apr_convolve_backward(lay, v, tree, st, K, g, stream=s)),
    "stencil_grad": lambda lay, st, w, v, tree, g, x, tb, s: [G.apr_convolve_stencil_grad(lay, v, tree, K, g, stream=s)],
    "mc_backward": lambda lay, st, w, v, tree, g, x, tb, s: list(G.apr_convolve_mc_backward(lay, x, tb, w, x, stream=s)),
}


@pytest.mark.parametrize("name", list(CALLS))
def test_two_streams(name):
    lay, st, w, data = setup()
    ref = [CALLS[name](lay, st, w, *d, None) for d in data]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = []
    for _ in range(8):
        for s, d in zip(streams, data):
            with torch.cuda.stream(s):
                got.append(CALLS[name](lay, st, w, *d, None))
    torch.cuda.synchronize()
    for i, res in enumerate(got):
        assert all(torch.equal(a, b) for a, b in zip(res, ref[i % 2]))


@pytest.mark.parametrize("name", list(CALLS))
def test_stream_argument(name):
    lay, st, w, data = setup()
    ref = CALLS[name](lay, st, w, *data[0], None)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        torch.cuda._sleep(2000000)      # the call waits behind this, about a millisecond
    got = CALLS[name](lay, st, w, *data[0], s)
    for nbytes in {t for n in (lay.n_tree, lay.n_particles, 64 * lay.n_tree) for t in (n, 4 * n, 8 * n)}:
        torch.empty(max(nbytes // 4, 1), device="cuda").fill_(float("nan"))     # what the current stream can get hold of
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, ref))


def test_workspaces_are_apart():
    lay, *_ = setup()
    a, b = lay.workspace(K)[0], lay.workspace(K)[0]
    assert a.data_ptr() != b.data_ptr() and a.numel() >= lay.workspace(K)[1]
