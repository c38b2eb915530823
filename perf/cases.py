"""Workloads of the APR convolution framework, as its users run them.

Every case is one call chain over one APR image: a forward filter, a layer's training step, an
iterated filter, a gradient map, or a multi-channel bf16 layer or network. An APR is drawn on the GPU
from a seeded image of Gaussian blobs: cells are split where the blobs are steep, down to the requested
number of particles, with touching cells at most one level apart; a particle holds the shot-noisy mean
of its pixels. The blobs, and with them the cells, follow from the case; the seed gives the noise and
every other value (as the frames or channels of one acquisition, or the steps of a training, differ). ``exact`` repeats a pass in float64 with plain torch gathers and scatters over the same
cells.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2112_03592_gb300 as apr
from paper_2112_03592_gb300.surrogate import AprCnn

REFLECT, ZERO = apr.APR_BC_REFLECT, apr.APR_BC_ZERO
C = 16           # channels of the multi-channel layers
N_LAYERS = 4     # layers of the network


# ------------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------------
def listed():
    def case(name, kind, dims, particles, blobs, sigma, l_min, **kw):
        return dict(name=name, kind=kind, dz=dims[0], dx=dims[1], dy=dims[2], particles=particles, blobs=blobs,
                    sigma_lo=sigma[0], sigma_hi=sigma[1], l_min=l_min, **kw)

    return [
        # the smallest call: one 3^3 filter of a 64^3 crop (a preview, a tile of a large image)
        case("filter3_64", "filter", (64, 64, 64), 16500, 20, (2.0, 6.0), 2, k=3, stack="plain", bc=REFLECT),
        # one 5^3 smoothing of a mid-size volume (a frame of a time lapse), level-restricted stencils
        case("filter5_256", "filter", (256, 256, 256), 1000000, 400, (2.0, 12.0), 2, k=5, stack="restricted", bc=REFLECT),
        # the same smoothing of a full light-sheet volume: the paper's forward pipeline
        case("filter5_1024", "filter", (512, 1024, 1024), 8000000, 2000, (2.0, 20.0), 3, k=5, stack="restricted",
             bc=REFLECT),
        # a training step of a small learned 3^3 layer on a ragged crop with zero padding
        case("train3_ragged", "train", (61, 93, 130), 45000, 24, (2.0, 7.0), 2, k=3, stack="learned", bc=ZERO),
        # a training step of a learned 5^3 layer (taps on every level) on a mid-size odd volume
        case("train5_odd", "train", (201, 333, 411), 800000, 200, (2.0, 12.0), 2, k=5, stack="learned", bc=REFLECT),
        # forward and backward of the 5^3 layer on the full volume: the repository's default benchmark
        case("train5_1024", "train", (512, 1024, 1024), 8000000, 2000, (2.0, 20.0), 3, k=5, stack="restricted", bc=REFLECT),
        # deconvolution of a small crop: a chain of short dependent calls
        case("rl3_crop", "rl", (70, 96, 131), 40000, 20, (2.0, 7.0), 2, k=3, stack="restricted", bc=ZERO, iters=10),
        # 20 Richardson-Lucy iterations on a 512^3 volume
        case("rl5_512", "rl", (512, 512, 512), 2870000, 200, (2.0, 20.0), 3, k=5, stack="restricted", bc=REFLECT, iters=20),
        # gradient magnitude (segmentation input) of an odd-sized volume, level-rescaled Sobel filters
        case("gradient_odd", "gradient", (301, 277, 390), 1200000, 300, (2.0, 14.0), 3, k=3, stack="sobel", bc=REFLECT),
        # a training step of one 16 -> 16-channel bf16 layer: small ragged crop, and the 1 M-particle volume
        case("mctrain_ragged", "mctrain", (61, 93, 130), 45000, 24, (2.0, 7.0), 2, bc=ZERO),
        case("mctrain_256", "mctrain", (256, 256, 256), 1000000, 400, (2.0, 12.0), 2, bc=REFLECT),
        # inference of the four-layer network, a whole call
        case("cnn_384", "cnn", (384, 512, 512), 2400000, 300, (2.0, 16.0), 3, bc=REFLECT),
    ]


# largest volume and particle count of each kind, as listed
_CAP = {"filter": (512 * 1024 * 1024, 8000000), "train": (512 * 1024 * 1024, 8000000), "rl": (512 ** 3, 2800000),
        "gradient": (301 * 277 * 390, 1200000), "mctrain": (256 ** 3, 1000000), "cnn": (384 * 512 * 512, 2400000)}


def draw(rng):
    kind = rng.choice(["filter", "filter", "train", "train", "rl", "gradient", "mctrain", "mctrain", "cnn"])
    vcap, pcap = _CAP[kind]
    vol = math.exp(rng.uniform(math.log(48 ** 3), math.log(vcap)))
    edge = vol ** (1.0 / 3.0)
    a, b = math.exp(rng.uniform(-0.35, 0.35)), math.exp(rng.uniform(-0.35, 0.35))
    dims = [max(24, int(edge * f)) for f in (a, b, 1.0 / (a * b))]
    dims = [d + (rng.random() < 0.5) * (1 - d % 2) for d in dims]    # odd in half of the draws
    while dims[0] * dims[1] * dims[2] > vcap:
        dims[dims.index(max(dims))] -= 2
    frac = math.exp(rng.uniform(math.log(0.012), math.log(0.08)))
    particles = max(2000, min(pcap, int(frac * dims[0] * dims[1] * dims[2])))
    hi = max(4.0, min(20.0, min(dims) / 10.0))
    case = dict(kind=kind, dz=dims[0], dx=dims[1], dy=dims[2], particles=particles,
                blobs=max(8, min(2000, particles // 4000)), sigma_lo=2.0, sigma_hi=hi, l_min=rng.choice([2, 3]),
                bc=rng.choice([REFLECT, REFLECT, ZERO]))
    if kind == "filter":
        case.update(k=rng.choice([3, 5]), stack=rng.choice(["plain", "restricted"]))
    elif kind == "train":
        case.update(k=rng.choice([3, 5]), stack=rng.choice(["restricted", "learned"]))
    elif kind == "rl":
        case.update(k=rng.choice([3, 5]), stack="restricted", iters=rng.choice([5, 10, 20]))
    elif kind == "gradient":
        case.update(k=3, stack="sobel")
    return case


# ------------------------------------------------------------------------------------------------
# an APR from a blob image
# ------------------------------------------------------------------------------------------------
def _level_dims(dims, l_max, l):
    s = 1 << (l_max - l)
    return tuple(-(-d // s) for d in dims)


def _pad_even(a, fill):
    pz, px, py = (s % 2 for s in a.shape)
    return torch.nn.functional.pad(a, (0, py, 0, px, 0, pz), value=fill) if pz or px or py else a


def _blocks(a, fill):
    a = _pad_even(a, fill)
    z, x, y = a.shape
    return a.view(z // 2, 2, x // 2, 2, y // 2, 2)


def _dilate(b):
    for ax in range(3):
        n = b.shape[ax]
        out = b.clone()
        if n > 1:
            out.narrow(ax, 1, n - 1).logical_or_(b.narrow(ax, 0, n - 1))
            out.narrow(ax, 0, n - 1).logical_or_(b.narrow(ax, 1, n - 1))
        b = out
    return b


def _upsample(b, shape):
    z, x, y = b.shape
    u = b.view(z, 1, x, 1, y, 1).expand(z, 2, x, 2, y, 2).reshape(2 * z, 2 * x, 2 * y)
    return u[:shape[0], :shape[1], :shape[2]]


def _in_grid_counts(dims, l_max, l, device):
    """Pixels along each axis under the cells of level l."""
    s = 1 << (l_max - l)
    return [torch.tensor([min(s, d - i * s) for i in range(-(-d // s))], dtype=torch.float32, device=device) for d in dims]


class _Apr:
    """Cells of one image: per level the particles' and the tree nodes' coordinates, in storage order
    (level, z, x, y), and the particle values."""


def _make_apr(case, seed):
    dev = torch.device("cuda")
    dims = (case["dz"], case["dx"], case["dy"])
    l_max, l_min = max(1, math.ceil(math.log2(max(dims)))), case["l_min"]
    rng = np.random.default_rng([case["dz"], case["dx"], case["dy"], case["particles"]])
    lam = torch.full(dims, 100.0, device=dev)
    amp = torch.full(dims, 10.0, device=dev)
    centres = rng.uniform(0.0, 1.0, (case["blobs"], 3)) * np.array(dims)
    sigmas = rng.uniform(case["sigma_lo"], case["sigma_hi"], case["blobs"])
    amps = rng.uniform(200.0, 1000.0, case["blobs"])
    for c, s, a in zip(centres, sigmas, amps):
        h = math.ceil(3.5 * s)
        lo = [max(0, int(c[i]) - h) for i in range(3)]
        hi = [min(dims[i], int(c[i]) + h + 1) for i in range(3)]
        g = [torch.from_numpy(np.exp(-0.5 * ((np.arange(lo[i], hi[i]) - c[i]) / s) ** 2).astype(np.float32)).to(dev)
             for i in range(3)]
        box = tuple(slice(lo[i], hi[i]) for i in range(3))
        lam[box] += (float(a) * g[0])[:, None, None] * (g[1][:, None] * g[2][None, :])[None]
        amp[box].clamp_(min=float(a))
    steep = torch.zeros(dims, device=dev)
    for ax in range(3):
        d = torch.zeros(dims, device=dev)
        n = dims[ax]
        d.narrow(ax, 1, n - 2).copy_(0.5 * (lam.narrow(ax, 2, n - 2) - lam.narrow(ax, 0, n - 2)))
        d.narrow(ax, 0, 1).copy_(lam.narrow(ax, 1, 1) - lam.narrow(ax, 0, 1))
        d.narrow(ax, n - 1, 1).copy_(lam.narrow(ax, n - 1, 1) - lam.narrow(ax, n - 2, 1))
        steep.addcmul_(d, d)
    del d
    # a cell of level l is split where log2(local amplitude / slope) < (l_max - l) - log2(error bound)
    t = torch.log2_(amp.div_(steep.sqrt_()))
    del steep
    tmin, sums = {}, {l_max: lam}
    for l in range(l_max - 1, l_min - 1, -1):
        t = _blocks(t, float("inf")).amin(dim=(1, 3, 5))
        tmin[l] = t
        sums[l] = _blocks(sums[l + 1], 0.0).sum(dim=(1, 3, 5))
    del t, amp

    def split_masks(e):
        split = {}
        for l in range(l_max - 1, l_min - 1, -1):
            s = tmin[l] < (l_max - l) - e
            if l + 1 < l_max:
                s |= _blocks(_dilate(split[l + 1]), False).any(5).any(3).any(1)
            split[l] = s
        return split

    def children(l):     # in-grid children of every cell of level l along each axis
        dn = _level_dims(dims, l_max, l + 1)
        return [torch.tensor([min(2, n - 2 * i) for i in range(-(-n // 2))], dtype=torch.float64, device=dev) for n in dn]

    cz = {l: children(l) for l in tmin}

    def count(split):
        n = float(np.prod(_level_dims(dims, l_max, l_min)))
        for l in range(l_min, l_max):
            per_z = torch.einsum("zxy,x,y->z", split[l].to(torch.float32), cz[l][1].float(), cz[l][2].float()).double()
            n += float((per_z * cz[l][0]).sum()) - float(split[l].sum())
        return n

    lo, hi = -14.0, 14.0        # log2 of the error bound; fewer particles for a larger one
    for _ in range(14):
        mid = 0.5 * (lo + hi)
        n = count(split_masks(mid))
        if abs(n / case["particles"] - 1.0) < 0.01:
            break
        lo, hi = (mid, hi) if n > case["particles"] else (lo, mid)
    split = split_masks(mid)
    gen = torch.Generator(device=dev).manual_seed(seed + 77)
    A = _Apr()
    A.dims, A.l_min, A.l_max = dims, l_min, l_max
    A.part, A.node, counts, ys, vals = {}, {}, [], [], []
    for l in range(l_min, l_max + 1):
        shape = _level_dims(dims, l_max, l)
        leaf = torch.ones(shape, dtype=torch.bool, device=dev) if l == l_min else _upsample(split[l - 1], shape).clone()
        if l < l_max:
            leaf &= ~split[l]
            A.node[l] = split[l].nonzero()
        idx = leaf.nonzero()
        A.part[l] = idx
        counts.append(leaf.sum(dim=2).reshape(-1))
        ys.append(idx[:, 2].to(torch.int32))
        pix = _in_grid_counts(dims, l_max, l, dev)
        z, x, y = idx.unbind(1)
        npix = pix[0][z] * pix[1][x] * pix[2][y]
        mean = sums[l][z, x, y] / npix
        noise = torch.randn(mean.shape, generator=gen, device=dev)
        vals.append((mean + torch.sqrt(mean / npix) * noise).clamp_(min=1.0))
        del leaf
    row_ptr = torch.cat([torch.zeros(1, dtype=torch.int64, device=dev), torch.cumsum(torch.cat(counts), 0)])
    A.row_ptr, A.y_idx = row_ptr.cpu().numpy(), torch.cat(ys).cpu().numpy()
    A.values = torch.cat(vals)
    A.n = int(A.values.numel())
    A.nt = sum(int(v.shape[0]) for v in A.node.values())
    A.n_levels = l_max - l_min + 1
    return A


# ------------------------------------------------------------------------------------------------
# stencils, features, weights
# ------------------------------------------------------------------------------------------------
def _gaussian(k, sigma):
    t = np.arange(-(k // 2), k // 2 + 1, dtype=np.float64)
    g = np.exp(-0.5 * (t / sigma) ** 2)
    w = g[:, None, None] * g[None, :, None] * g[None, None, :]
    return (w / w.sum()).astype(np.float32)


def _stencils(case, A, seed):
    """The stack [L][k^3] (or [3][L][k^3]) a program hands to the convolution."""
    k, L = case["k"], A.n_levels
    w = _gaussian(k, 1.0 if k == 3 else 1.5)
    if case["stack"] == "plain":
        st = np.repeat(w.reshape(1, -1), L, 0)
    elif case["stack"] == "restricted":
        st = apr.apr_restrict_stencil(w, A.l_max, A.l_min)
    elif case["stack"] == "learned":
        rng = np.random.default_rng(seed + 5)
        st = (w.reshape(1, -1) + 0.02 * rng.standard_normal((L, k ** 3))).astype(np.float32)
    else:
        st = np.stack([apr.apr_rescale_stencil(s, A.l_max, A.l_min) for s in apr.sobel_stencils(k)])
    return torch.from_numpy(np.ascontiguousarray(st, np.float32)).cuda()


def _randn(shape, seed, scale=1.0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda") * scale


def _inputs(case, seed):
    A = _make_apr(case, seed)
    S = dict(case=case, apr=A)
    kind = case["kind"]
    if kind in ("filter", "train", "rl", "gradient"):
        S["stencils"] = _stencils(case, A, seed)
    if kind == "train":
        S["grad"] = _randn((A.n,), seed + 11)
    if kind == "mctrain":
        S["x"] = _randn((A.n, C), seed + 12).to(torch.bfloat16)
        S["grad"] = _randn((A.n, C), seed + 13).to(torch.bfloat16)
        S["weights"] = _randn((A.n_levels, C, C, 27), seed + 14, math.sqrt(1.0 / (27 * C))).to(torch.bfloat16)
    if kind == "cnn":
        S["scale"] = float(np.float32(1.0 / float(A.values.double().mean())))
        # the network's own initial scales: the last layer is a small correction to the residual
        S["weights"] = [_randn((A.n_levels, C, C, 27), seed + 20 + i,
                               math.sqrt(2.0 / (27 * C)) * (0.1 if i == N_LAYERS - 1 else 1.0)).to(torch.bfloat16)
                        for i in range(N_LAYERS)]
    return S


def prepare(case, seed):
    S = _inputs(case, seed)
    A = S["apr"]
    S["layout"] = apr.AprLayout(A.dims, A.l_min, A.l_max, A.row_ptr, A.y_idx)
    S["particles"] = A.values
    if case["kind"] == "train":
        S["particles"] = A.values.clone().requires_grad_()
        S["stencils"].requires_grad_()
    if case["kind"] == "cnn":
        S["net"] = AprCnn(n_layers=N_LAYERS)
    del S["apr"]
    return S


def run(state):
    case, lay, v = state["case"], state["layout"], state["particles"]
    kind = case["kind"]
    if kind == "filter":
        return apr.apr_convolve_auto(lay, v, state["stencils"], case["k"], case["bc"])
    if kind == "train":
        out = apr.AprConv.apply(v, state["stencils"], lay, case["k"], case["bc"])
        gv, gw = torch.autograd.grad(out, (v, state["stencils"]), state["grad"])
        return out.detach(), gv, gw
    if kind == "rl":
        return apr.apr_richardson_lucy(lay, v, state["stencils"], case["k"], case["iters"], case["bc"])
    if kind == "gradient":
        tree = apr.apr_tree_restrict(lay, v)
        return apr.apr_gradient_magnitude(lay, v, tree, state["stencils"], case["k"], case["bc"])
    if kind == "mctrain":
        tree = apr.apr_tree_restrict_bf16(lay, state["x"])
        out = apr.apr_convolve_mc(lay, state["x"], tree, state["weights"], case["bc"])
        gx, gw = apr.apr_convolve_mc_backward(lay, state["x"], tree, state["weights"], state["grad"], case["bc"])
        return out, gx, gw
    return state["net"].forward(lay, v, state["scale"], weights=state["weights"])


def work(case):
    """Bytes and FLOPs of one pass. A particle has an index entry (2 bytes) beside its values, and
    there is one tree node per seven particles (index entry only: its value is no input or output)."""
    n = case["particles"]
    nt = n // 7
    kind = case["kind"]
    index = 2 * n + 2 * nt
    if kind in ("mctrain", "cnn"):
        mac = 27 * C * C * n
        if kind == "mctrain":
            return {"bytes": index + n * C * (2 + 2 + 4 + 4), "flops": 3 * 2 * mac}
        return {"bytes": index + n * (4 + 4), "flops": N_LAYERS * 2 * mac}
    k3 = case["k"] ** 3
    # restricted 5^3 stencils keep 27 taps below the finest level, which holds about a fifth of the particles
    taps = 27 + (k3 - 27) // 5 if case["stack"] == "restricted" and case["k"] == 5 else k3
    if kind == "filter":
        return {"bytes": index + 8 * n, "flops": 2 * taps * n}
    if kind == "train":
        return {"bytes": index + 16 * n, "flops": 2 * (2 * taps + k3) * n}
    if kind == "rl":
        return {"bytes": index + 8 * n, "flops": case["iters"] * 2 * 2 * taps * n}
    return {"bytes": index + 8 * n, "flops": 3 * 2 * k3 * n}


# ------------------------------------------------------------------------------------------------
# the same in float64
# ------------------------------------------------------------------------------------------------
class _Exact:
    """Sources of every level's cells: a particle, a tree node, or the next coarser particle over the
    cell, as indices into the concatenation [particles, tree nodes]."""

    def __init__(self, A, bc):
        self.A, self.bc = A, bc
        dev = A.values.device
        self.p0, self.t0, self.src, self.parent = {}, {}, {}, {}
        o = t = 0
        for l in range(A.l_min, A.l_max + 1):
            self.p0[l] = o
            o += A.part[l].shape[0]
        for l in range(A.l_min, A.l_max):
            self.t0[l] = t
            t += A.node[l].shape[0]
        prev = None
        for l in range(A.l_min, A.l_max + 1):
            shape = _level_dims(A.dims, A.l_max, l)
            m = torch.zeros(shape, dtype=torch.int32, device=dev) if prev is None else _upsample(prev, shape).clone()
            i = A.part[l]
            m[i[:, 0], i[:, 1], i[:, 2]] = torch.arange(self.p0[l], self.p0[l] + i.shape[0], dtype=torch.int32, device=dev)
            if l < A.l_max:
                i = A.node[l]
                m[i[:, 0], i[:, 1], i[:, 2]] = A.n + torch.arange(self.t0[l], self.t0[l] + i.shape[0], dtype=torch.int32,
                                                                  device=dev)
            self.src[l] = m
            prev = m
        # parent node of every particle and node above l_min, children per node
        self.cnt = torch.zeros(A.nt, dtype=torch.float64, device=dev)
        for l in range(A.l_min + 1, A.l_max + 1):
            for what in ("part", "node"):
                if what == "node" and l == A.l_max:
                    continue
                i = getattr(A, what)[l] >> 1
                par = self.src[l - 1][i[:, 0], i[:, 1], i[:, 2]].long() - A.n
                self.parent[what, l] = par
                self.cnt.index_add_(0, par, torch.ones(par.shape[0], dtype=torch.float64, device=dev))

    def restrict(self, v, rnd=None):
        A = self.A
        tree = torch.zeros((A.nt,) + v.shape[1:], dtype=torch.float64, device=v.device)
        for l in range(A.l_max - 1, A.l_min - 1, -1):
            a, b = self.t0[l], self.t0[l] + A.node[l].shape[0]
            tree.index_add_(0, self.parent["part", l + 1], v[self.p0[l + 1]:self.p0[l + 1] + A.part[l + 1].shape[0]])
            if l + 1 < A.l_max:
                tree.index_add_(0, self.parent["node", l + 1], tree[self.t0[l + 1]:self.t0[l + 1] + A.node[l + 1].shape[0]].clone())
            c = self.cnt[a:b].view((-1,) + (1,) * (v.dim() - 1))
            tree[a:b] /= c
            if rnd is not None:
                tree[a:b] = rnd(tree[a:b])
        return tree

    def push_down(self, gv, gt):
        A = self.A
        for l in range(A.l_min, A.l_max):
            share = gt / self.cnt.view((-1,) + (1,) * (gt.dim() - 1))
            gv[self.p0[l + 1]:self.p0[l + 1] + A.part[l + 1].shape[0]] += share[self.parent["part", l + 1]]
            if l + 1 < A.l_max:
                gt[self.t0[l + 1]:self.t0[l + 1] + A.node[l + 1].shape[0]] += share[self.parent["node", l + 1]]
        return gv

    def taps(self, l, k):
        """(tap, source index, inside) of every tap of the particles of level l."""
        A, r = self.A, k // 2
        d = _level_dims(A.dims, A.l_max, l)
        p = A.part[l]
        if p.shape[0] == 0:
            return
        for e in range(k ** 3):
            off = (e // (k * k) - r, (e // k) % k - r, e % k - r)
            q, ok = [], None
            for ax in range(3):
                c = p[:, ax] + off[ax]
                if self.bc == REFLECT:
                    c = torch.remainder(c, 2 * d[ax])
                    c = torch.where(c >= d[ax], 2 * d[ax] - 1 - c, c)
                elif off[ax]:
                    inside = (c >= 0) & (c < d[ax])
                    ok = inside if ok is None else ok & inside
                    c = c.clamp(0, d[ax] - 1)
                q.append(c)
            yield e, self.src[l][q[0], q[1], q[2]].long(), ok

    def levels(self):
        for l in range(self.A.l_min, self.A.l_max + 1):
            yield l, l - self.A.l_min, slice(self.p0[l], self.p0[l] + self.A.part[l].shape[0])

    def conv(self, v, tree, st, k):
        u = torch.cat([v, tree])
        out = torch.zeros_like(v)
        for l, i, s in self.levels():
            for e, src, ok in self.taps(l, k):
                t = u[src]
                if ok is not None:
                    t = t * ok
                out[s] += float(st[i, e]) * t
        return out

    def backward(self, v, tree, st, k, g):
        u = torch.cat([v, tree])
        gu, gw = torch.zeros_like(u), torch.zeros(st.shape, dtype=torch.float64, device=v.device)
        for l, i, s in self.levels():
            for e, src, ok in self.taps(l, k):
                t = g[s] if ok is None else g[s] * ok
                gu.index_add_(0, src, float(st[i, e]) * t)
                gw[i, e] = (t * u[src]).sum()
        return self.push_down(gu[:self.A.n], gu[self.A.n:]), gw

    def conv_mc(self, v, tree, W):
        u = torch.cat([v, tree])
        out = torch.zeros_like(v)
        for l, i, s in self.levels():
            for e, src, ok in self.taps(l, 3):
                t = u[src]
                if ok is not None:
                    t = t * ok[:, None]
                out[s] += t @ W[i, :, :, e].T
        return out

    def backward_mc(self, v, tree, W, g):
        u = torch.cat([v, tree])
        gu, gw = torch.zeros_like(u), torch.zeros(W.shape, dtype=torch.float64, device=v.device)
        for l, i, s in self.levels():
            for e, src, ok in self.taps(l, 3):
                t = g[s] if ok is None else g[s] * ok[:, None]
                gu.index_add_(0, src, t @ W[i, :, :, e])
                gw[i, :, :, e] = t.T @ u[src]
        return self.push_down(gu[:self.A.n], gu[self.A.n:]), gw


def _bf16(t):
    return t.to(torch.float32).to(torch.bfloat16).to(torch.float64)


def exact(case, seed):
    with torch.no_grad():
        S = _inputs(case, seed)
        A = S["apr"]
        X = _Exact(A, case["bc"])
        v = A.values.double()
        kind = case["kind"]
        if kind in ("filter", "train", "rl", "gradient"):
            k = case["k"]
            st = S["stencils"].double().cpu()
        if kind == "filter":
            return X.conv(v, X.restrict(v), st, k)
        if kind == "train":
            tree = X.restrict(v)
            gv, gw = X.backward(v, tree, st, k, S["grad"].double())
            return X.conv(v, tree, st, k), gv, gw
        if kind == "rl":
            est = v.clone()
            flip = st.flip(1)
            for _ in range(case["iters"]):
                den = X.conv(est, X.restrict(est), st, k)
                ratio = torch.where(den > 0, v / den, torch.zeros_like(v))
                est = est * X.conv(ratio, X.restrict(ratio), flip, k)
            return est
        if kind == "gradient":
            tree = X.restrict(v)
            return torch.sqrt(sum(X.conv(v, tree, st[a], k) ** 2 for a in range(3)))
        if kind == "mctrain":
            x, W = S["x"].double(), S["weights"].double()
            tree = X.restrict(x, _bf16)
            gx, gw = X.backward_mc(x, tree, W, S["grad"].double())
            return X.conv_mc(x, tree, W), gx, gw
        h = torch.zeros((A.n, C), dtype=torch.float64, device=v.device)
        h[:, 0] = (A.values * S["scale"]).to(torch.bfloat16).double()
        for i, W in enumerate(S["weights"]):
            c = X.conv_mc(h, X.restrict(h, _bf16), W.double())
            if i + 1 < N_LAYERS:
                h = _bf16(c.clamp(min=0.0))
        return v + c[:, 0] / S["scale"]
