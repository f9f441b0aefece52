"""The calls that a user of the framework makes, over the sizes and options they make them at.

A radiation-hydrodynamics code that uses the library builds the radiation tree from its
gas particles and sources at every time step and asks for the flux at its particles, so
most cases are a tree build followed by a flux. The others keep a tree and ask it for
more (the sinks on the current time step, the vector flux), differentiate the flux, run
many boxes in one launch, or sort particles along the Morton curve. Inputs are seeded
and generated on the GPU with the distributions of `workloads`: uniform particles,
lognormal absorption, lognormal luminosities, sources uniform or in Gaussian clumps.

A case is a dict: "call" names the entry points (see `run`), the rest are sizes and
options. `exact` restates the method in plain torch: the discrete decisions in fp32 in
the order that the method defines, the values in FP64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1902_08083_gb300 import trevr

ONE_BELOW = float(np.nextafter(np.float32(1.0), np.float32(0.0)))
BG_RADIUS = 0.45
GRID = 1 << 21
EXACT_FLOPS = 2e10  # larger cases would take the plain restatement too long


def _flux(name, n, s, theta=0.75, tau_ref=0.1, sigma=1.0, alpha=1.0, clumps=0, **more):
    return dict(name=name, call="step", n=n, s=s, theta=theta, tau_ref=tau_ref, sigma=sigma,
                alpha=alpha, clumps=clumps, **more)


def listed():
    return [
        # one time step of a small test box: launches and host work count
        _flux("step_uniform_4k", 4096, 64, sigma=0.0),
        # the Stromgren test: one source in a uniform medium, a build and one ray per sink
        _flux("step_stromgren_256k", 1 << 18, 1, sigma=0.0, alpha=20.0),
        # one time step of the benchmark: clumped sources, a dense occluder
        _flux("step_clumpy_4m", 1 << 22, 1 << 14, theta=0.6, sigma=2.0, clumps=16),
        # an ordinary box at a fine refinement threshold, odd sizes
        _flux("step_lognormal_100k", 100003, 1999, tau_ref=0.01),
        # background radiation from a sphere of sources
        _flux("step_background_32k", 1 << 15, 20000, theta=0.6, sigma=0.0, alpha=3.0,
              background=True),
        # buckets traced through their particles; build, neighbour lists and flux
        _flux("step_sub_bucket_64k", 1 << 16, 256, theta=0.6, tau_ref=0.05, sigma=1.5, alpha=2.0,
              sub_bucket=True),
        # three bands of radiation that share one walk
        dict(_flux("bands3_200k", 200003, 1024), call="bands", bands=3),
        # the particles on the shortest time step, one in ten, from a kept tree
        dict(_flux("active_100k_of_1m", 1 << 20, 4096), call="active", m=104857),
        # flux, vector flux and radiation pressure from a kept tree
        dict(_flux("moments_256k", 1 << 18, 1024), call="moments"),
        # a differentiable forward model: flux, then gradients of a loss
        dict(_flux("gradient_1m", 1 << 20, 1024), call="gradient"),
        # many boxes of uneven size in one persistent launch
        dict(call="batch", name="batch_64_boxes", boxes=64, lo=12, hi=17, theta=0.75, tau_ref=0.1),
        # Morton keys and order into the caller's buffers, without allocation
        dict(call="sort", name="sort_1m", n=(1 << 20) - 3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    top = max(_cost(c) for c in listed())
    while True:
        call = rng.choice(["step"] * 6 + ["bands", "active", "moments", "gradient", "batch", "sort"])
        if call == "sort":
            return dict(call=call, n=_log_int(rng, 1000, (1 << 20) - 1))
        if call == "batch":
            lo = rng.randint(8, 13)
            return dict(call=call, boxes=_log_int(rng, 2, 96), lo=lo,
                        hi=min(17, lo + rng.randint(1, 5)), theta=rng.choice([0.6, 0.75, 0.9]),
                        tau_ref=rng.choice([0.05, 0.1, 0.5]))
        n = _log_int(rng, 2000, 1 << 22)
        c = dict(call=call, n=n, s=min(_log_int(rng, 1, 1 << 14), max(1, n // 16)),
                 theta=rng.choice([0.45, 0.6, 0.75, 1.0]), tau_ref=rng.choice([0.01, 0.1, 0.5]),
                 sigma=rng.choice([0.0, 1.0, 1.5, 2.0]), alpha=rng.choice([0.25, 1.0, 4.0]),
                 clumps=rng.choice([0, 0, 0, 16]))
        if call == "step":
            kind = rng.choice(["plain"] * 4 + ["background", "sub_bucket", "topdown", "stop"])
            if kind == "background":
                c.update(background=True, sigma=0.0, clumps=0, s=_log_int(rng, 500, 20000),
                         n=_log_int(rng, 2000, 1 << 18))
            elif kind == "sub_bucket":
                c.update(sub_bucket=True, n=_log_int(rng, 2000, 1 << 18), tau_ref=0.05, sigma=1.5,
                         alpha=2.0)
                c["s"] = min(c["s"], max(1, c["n"] // 16), 1024)
            elif kind == "topdown":
                c.update(topdown=True)
            elif kind == "stop":
                c.update(tau_stop=rng.choice([8.0, 10.0]), alpha=rng.choice([4.0, 16.0]))
        elif call == "bands":
            c["bands"] = rng.randint(2, 4)
        elif call == "active":
            c["m"] = max(1, int(c["n"] * rng.choice([0.01, 0.1, 0.3])))
        if _cost(c) <= top:
            return c


# ------------------------------------------------------------------------------ work
def _rays_segments(c):
    """Rays per sink and segments per ray of this kind of box, from counted runs."""
    s = c["s"]
    rays = max(min(0.65 * s, 41.0), 33.5 * (math.log2(s + 1) - 5.7) * (0.75 / c["theta"]) ** 1.75)
    rays = min(float(s), max(1.0, rays)) * (0.25 if c.get("clumps") else 1.0)
    fine = {0.01: 1.5, 0.05: 1.2, 0.1: 1.0}.get(c["tau_ref"], 0.7)
    segments = 6.0 if not c.get("sigma") else 13.0 * fine
    return rays, segments


def _box_sizes(c):
    rng = np.random.default_rng(1000)
    return np.floor(2.0 ** rng.uniform(c["lo"], c["hi"], c["boxes"])).astype(int)


def work(c):
    """The least a pass can move and compute: inputs read and outputs written once; per ray
    an exponential and a sum (40 operations), per segment the cut with the cell's planes and
    the optical depth (12)."""
    call = c["call"]
    if call == "sort":
        return {"bytes": 24.0 * c["n"], "flops": 0.0}
    if call == "batch":
        n = float(_box_sizes(c).sum())
        rays, seg = _rays_segments(dict(s=max(1, int(n / c["boxes"] / 64)), theta=c["theta"],
                                        tau_ref=c["tau_ref"], sigma=1.0))
        return {"bytes": 20.0 * n, "flops": n * rays * (40 + 12 * seg)}
    n, s, m = c["n"], c["s"], c.get("m", c["n"])
    rays, seg = _rays_segments(c)
    flops = m * rays * (40 + 12 * seg)
    bands = c.get("bands", 1)
    nbytes = (12 + 4 * bands) * (n + s) + 4 * bands * m
    if call == "active":
        nbytes = 20.0 * m
    elif call == "moments":
        nbytes = 16.0 * (n + s) + 40.0 * n
        flops += n * rays * 18
    elif call == "gradient":
        nbytes = 16.0 * (n + s) + 12.0 * n + 4.0 * s
        flops += n * rays * (60 + 12 * seg)
    elif c.get("sub_bucket"):
        nbytes += 4.0 * n
        flops += n * rays * 1.5 * 40 * 20  # traced chords, neighbours on each, operations
    return {"bytes": float(nbytes), "flops": float(flops)}


def _cost(c):
    if c["call"] == "sort":
        return 0.0
    w = work(c)["flops"]
    return w * {"bands": 2.0, "gradient": 1.2, "active": 4.0}.get(c["call"], 1.0) * (
        1.5 if c.get("sub_bucket") else 1.0)


# ---------------------------------------------------------------------------- inputs
def _uniform(g, n):
    x = torch.rand(3, n, device="cuda", generator=g)
    return x.clamp_(max=ONE_BELOW)


def _lognormal(g, xyz, alpha, sigma, corr=0.05, modes=256):
    """alpha exp(sigma f - sigma^2/2) with f a unit Gaussian field of the correlation length."""
    k = torch.randn(modes, 3, device="cuda", generator=g) / corr
    phase = torch.rand(modes, device="cuda", generator=g) * (2.0 * math.pi)
    f = torch.empty(xyz.shape[1], device="cuda")
    step = 1 << 18
    for i in range(0, xyz.shape[1], step):
        f[i:i + step] = torch.cos(xyz[:, i:i + step].T @ k.T + phase).sum(1)
    f *= math.sqrt(2.0 / modes)
    return alpha * torch.exp(sigma * f - 0.5 * sigma * sigma)


def _sources(g, s, clumps):
    if not clumps:
        return _uniform(g, s)
    centre = 0.1 + 0.8 * torch.rand(3, clumps, device="cuda", generator=g)
    which = torch.arange(s, device="cuda") % clumps
    x = centre[:, which] + 0.02 * torch.randn(3, s, device="cuda", generator=g)
    return x.clamp_(0.0, ONE_BELOW)


def _ball(g, n, radius):
    """Uniform points in a ball around the box centre."""
    v = torch.randn(3, n, device="cuda", generator=g)
    r = radius * torch.rand(n, device="cuda", generator=g) ** (1.0 / 3.0)
    return 0.5 + v / v.norm(dim=0) * r


def _spiral(s, radius):
    k = torch.arange(s, device="cuda", dtype=torch.float64)
    z = 1.0 - (2.0 * k + 1.0) / s
    rho = (1.0 - z * z).clamp(min=0.0).sqrt()
    phi = k * (math.pi * (3.0 - math.sqrt(5.0)))
    return (0.5 + radius * torch.stack([rho * phi.cos(), rho * phi.sin(), z])).float()


def _inputs(c, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    n, s = c["n"], c["s"]
    d = {"weight": None}
    if c.get("background"):
        d["gas"], d["src"] = _ball(g, n, 0.95 * BG_RADIUS), _spiral(s, BG_RADIUS)
        d["lum"] = torch.full((s,), 1.0 / s, device="cuda")
    else:
        d["gas"] = _uniform(g, n)
        d["src"] = _sources(g, s, c["clumps"])
        if s == 1:
            d["src"].fill_(0.5)
        d["lum"] = torch.randn(s, device="cuda", generator=g).exp()
    if c["sigma"]:
        d["alpha"] = _lognormal(g, d["gas"], c["alpha"], c["sigma"])
    else:
        d["alpha"] = torch.full((n,), float(c["alpha"]), device="cuda")
    if c["clumps"]:  # the dense cube of the benchmark's box
        d["alpha"][((d["gas"] >= 0.45) & (d["gas"] <= 0.55)).all(dim=0)] *= 1e3
    if c.get("bands"):
        f = torch.tensor([1.0, 0.5, 0.25, 2.0][:c["bands"]], device="cuda")[:, None]
        d["alpha"] = (f * d["alpha"]).contiguous()
        d["lum"] = (f.reciprocal() * d["lum"]).contiguous()
    if c.get("sub_bucket"):
        # half the distance to the 32nd neighbour of a uniform set: the sphere that reaches it
        # has a Gamma(32) volume (a sum of 32 exponentials) in units of 1/n
        d["weight"] = torch.full((n,), 1.0 / n, device="cuda")
        u = torch.rand(32, n, device="cuda", generator=g, dtype=torch.float64).clamp(min=1e-12)
        volume = -u.log().sum(0) / n
        d["hsml"] = (0.5 * (volume * (3.0 / (4.0 * math.pi))) ** (1.0 / 3.0)).float()
    if c["call"] == "active":
        pick = torch.randperm(n, device="cuda", generator=g)[:c["m"]]
        d["sinks"] = pick.sort().values
    if c["call"] == "gradient":
        d["grad"] = torch.randn(n, device="cuda", generator=g)
    return d


def _options(c):
    o = {}
    if c.get("background"):
        o["bg_radius"] = BG_RADIUS
    if c.get("sub_bucket"):
        o["sub_bucket"] = 1
    if c.get("topdown"):
        o["ray_walk"] = 1
    if c.get("tau_stop"):
        o["tau_stop"] = c["tau_stop"]
    return o


def _batch_boxes(c, seed):
    boxes = []
    for b, n in enumerate(_box_sizes(c)):
        n = int(n)
        box = dict(call="step", n=n, s=max(1, n // 64), theta=c["theta"], tau_ref=c["tau_ref"],
                   sigma=float(b % 2), alpha=1.0, clumps=0)
        boxes.append((box, _inputs(box, 100003 * (seed % 9973) + b)))
    return boxes


def _build(d):
    return trevr.build_tree(d["gas"], d["alpha"], d["src"], d["lum"], d["weight"])


def prepare(c, seed):
    if c["call"] == "sort":
        g = torch.Generator("cuda").manual_seed(seed)
        n = c["n"]
        return dict(case=c, gas=_uniform(g, n), keys=torch.empty(n, dtype=torch.int64, device="cuda"),
                    perm=torch.empty(n, dtype=torch.int32, device="cuda"))
    if c["call"] == "batch":
        trees = [_build(d) for _, d in _batch_boxes(c, seed)]
        batch = trevr.Batch(trees)
        batch.run(c["theta"], c["tau_ref"])  # lays out the work items
        return dict(case=c, batch=batch)
    d = _inputs(c, seed)
    d["case"] = c
    if c["call"] in ("active", "moments"):
        d["tree"] = _build(d)
    if c["call"] == "gradient":
        d["alpha"].requires_grad_(True)
        d["lum"].requires_grad_(True)
    return d


def run(d):
    c = d["case"]
    call = c["call"]
    if call == "sort":
        return trevr.morton_sort_noalloc(d["gas"], keys_out=d["keys"], perm_out=d["perm"])
    if call == "batch":
        d["batch"].run(c["theta"], c["tau_ref"])
        return torch.cat(d["batch"].flux)
    theta, tau_ref = c["theta"], c["tau_ref"]
    if call == "step":
        tree = _build(d)
        if c.get("sub_bucket"):
            tree.set_smoothing(d["hsml"])
        return trevr.compute_flux(tree, theta, tau_ref, **_options(c))
    if call == "bands":
        return trevr.compute_flux_bands(_build(d), theta, tau_ref)
    if call == "active":
        return trevr.compute_flux(d["tree"], theta, tau_ref, sink_idx=d["sinks"])
    if call == "moments":
        return trevr.compute_flux_moments(d["tree"], theta, tau_ref)
    flux = trevr.trevr_flux(d["gas"], d["alpha"], d["src"], d["lum"], theta, tau_ref)
    ga, gl = torch.autograd.grad(flux, (d["alpha"], d["lum"]), grad_outputs=d["grad"])
    return flux.detach(), ga, gl


# ------------------------------------------------------------------ the method in 64 bits
def _spread_bits(v):
    """Bits of v moved three apart (21 bits)."""
    out = torch.zeros_like(v)
    for b in range(21):
        out |= ((v >> b) & 1) << (3 * b)
    return out


def _grid(x):
    """Grid coordinates of points in the unit box: fp32 scaling, truncation, clamping."""
    return (x * float(GRID)).to(torch.int64).clamp_(0, GRID - 1)


def _highest_bit(x):
    b = torch.zeros_like(x)
    for step in (32, 16, 8, 4, 2, 1):
        big = (x >> step) > 0
        x, b = torch.where(big, x >> step, x), b + big * step
    return b


class _ExactTree:
    """The radiation tree: topology by Morton prefixes, FP64 moments (of alpha (B, N) and
    lum (B, S), with one weight per particle)."""

    def __init__(self, gas, alpha, src, lum, weight, bucket=8):
        dev, n = gas.device, gas.shape[1]
        f64 = torch.float64
        grid = _grid(gas)
        key = (_spread_bits(grid[0]) << 2) | (_spread_bits(grid[1]) << 1) | _spread_bits(grid[2])
        self.key, self.perm = torch.sort(key, stable=True)
        grid = grid[:, self.perm]
        # cells level by level: particle range, box, split axis, child, code (path bits)
        first = torch.zeros(1, dtype=torch.int64, device=dev)
        count = first + n
        lo = torch.zeros(1, 3, dtype=torch.int64, device=dev)
        hi = lo + GRID
        code = first + 1
        parent = first - 1
        parts, total, self.levels = [], 0, []
        while first.numel():
            m = first.numel()
            self.levels.append((total, total + m))
            k0, k1 = self.key[first], self.key[first + count - 1]
            inner = (count > bucket) & (k0 != k1)
            bit = _highest_bit(torch.where(inner, k0 ^ k1, torch.ones_like(k0)))
            split = torch.searchsorted(self.key, ((k0 >> bit) | 1) << bit)
            axis = (62 - bit) % 3
            shift = 20 - torch.div(62 - bit, 3, rounding_mode="floor")
            plane = ((grid[axis, first] >> shift) | 1) << shift
            rank = torch.cumsum(inner, 0) - 1
            child = torch.where(inner, total + m + 2 * rank, torch.full_like(rank, -1))
            parts.append((first, count, lo, hi, code, parent, child,
                          torch.where(inner, axis, torch.full_like(axis, -1)), plane))
            i = torch.nonzero(inner)[:, 0]
            own = torch.arange(total, total + m, device=dev)[i]
            lo1, hi1, lo2, hi2 = lo[i].clone(), hi[i].clone(), lo[i].clone(), hi[i].clone()
            hi1.scatter_(1, axis[i, None], plane[i, None])
            lo2.scatter_(1, axis[i, None], plane[i, None])
            both = lambda a, b: torch.stack([a, b], 1).flatten(0, 1)  # noqa: E731
            new_first = both(first[i], split[i])
            count = both(split[i] - first[i], first[i] + count[i] - split[i])
            first, lo, hi = new_first, both(lo1, lo2), both(hi1, hi2)
            code, parent = both(2 * code[i], 2 * code[i] + 1), both(own, own)
            total += m
        cat = [torch.cat(p) for p in zip(*parts)]
        self.first, self.count, glo, ghi, self.code, self.parent, self.child, self.axis, plane = cat
        self.plane = plane
        self.glo, self.ghi = glo, ghi
        self.lo = glo.to(torch.float32) * (1.0 / GRID)
        self.hi = ghi.to(torch.float32) * (1.0 / GRID)
        self.depth = torch.cat([torch.full((b - a,), d, device=dev)
                                for d, (a, b) in enumerate(self.levels)])
        leaves = torch.nonzero(self.child < 0)[:, 0]
        order = torch.argsort(self.first[leaves])
        leaves = leaves[order]
        self.leaf_of = torch.repeat_interleave(leaves, self.count[leaves])  # sorted particles
        self.pos = gas[:, self.perm]
        # sources in their leaves, ordered by leaf
        src_leaf = self.locate(_grid(src))
        self.src_order = torch.argsort(self.first[src_leaf], stable=True)
        self.src = src[:, self.src_order]
        self.lum = lum.to(f64)[:, self.src_order]
        self.src_leaf = src_leaf[self.src_order]
        f = self.first[self.src_leaf]
        self.src_first = torch.searchsorted(f, self.first)
        self.src_count = torch.searchsorted(f, self.first + self.count) - self.src_first
        # moments: leaf sums, then children into parents
        w = torch.ones(n, dtype=f64, device=dev) if weight is None else weight.to(f64)[self.perm]
        a = alpha.to(f64)[:, self.perm]
        nb, nc = a.shape[0], self.first.numel()
        W = torch.zeros(nc, dtype=f64, device=dev).index_add(0, self.leaf_of, w)
        WA = torch.zeros(nb, nc, dtype=f64, device=dev).index_add(1, self.leaf_of, a * w)
        L = torch.zeros(nb, nc, dtype=f64, device=dev).index_add(1, self.src_leaf, self.lum)
        single = self.lum.sum(0).to(torch.float32).to(f64)
        if nb == 1:
            single = self.lum[0]
        self.single = single
        LY = torch.zeros(4, nc, dtype=f64, device=dev).index_add(
            1, self.src_leaf, torch.cat([single[None], single * self.src.to(f64)]))
        low = [(WA.detach()[b] / W.clamp(min=1e-300)).expand(3, nc).clone() for b in range(nb)]
        high = [x.clone() for x in low]
        width = (ghi - glo).T.to(f64)
        for a0, b0 in reversed(self.levels):
            X = torch.arange(a0, b0, device=dev)[self.child[a0:b0] >= 0]
            c = self.child[X]
            W = W.index_add(0, X, W[c] + W[c + 1])
            WA = WA.index_add(1, X, WA[:, c] + WA[:, c + 1])
            L = L.index_add(1, X, L[:, c] + L[:, c + 1])
            LY = LY.index_add(1, X, LY[:, c] + LY[:, c + 1])
            for d in range(3):
                along = self.axis[X] == d
                for x, pick in [(v, torch.minimum) for v in low] + [(v, torch.maximum) for v in high]:
                    x1, x2 = x[d, c], x[d, c + 1]
                    mean = (x1 * width[d, c] + x2 * width[d, c + 1]) / width[d, X]
                    x[d, X] = torch.where(along, mean, pick(x1, x2))
        self.abar = WA / W
        spread = [(high[b].amax(0) - low[b].amin(0)).to(torch.float32) for b in range(nb)]
        self.spread = torch.stack(spread).amax(0)
        self.bandL = L
        self.L = LY[0]
        self.cen = torch.where(LY[0] > 0, LY[1:] / LY[0].clamp(min=1e-300), torch.zeros_like(LY[1:]))
        c32 = self.cen.detach().to(torch.float32)
        far = torch.maximum(c32 - self.lo.T, self.hi.T - c32)
        self.l2 = (far[0] * far[0] + far[1] * far[1]) + far[2] * far[2]

    def locate(self, grid):
        X = torch.zeros(grid.shape[1], dtype=torch.int64, device=grid.device)
        while True:
            c = self.child[X]
            inner = c >= 0
            if not bool(inner.any()):
                return X
            g = grid.gather(0, self.axis[X].clamp(min=0)[None])[0]
            X = torch.where(inner, c + (g >= self.plane[X]).long(), X)


def _gap2(T, X, p):
    e = torch.maximum(T.lo[X].T - p, p - T.hi[X].T).clamp(min=0.0)
    return (e[0] * e[0] + e[1] * e[1]) + e[2] * e[2]


def _pairs(T, sinks, theta):
    """Every (sink, cell, source) that a ray goes to; source is -1 for a merged cell."""
    th = np.float32(theta)
    theta2 = float(th * th)
    who, X, out = sinks, torch.zeros_like(sinks), []
    while who.numel():
        keep = T.L[X] > 0
        who, X = who[keep], X[keep]
        merged = T.l2[X] < theta2 * _gap2(T, X, T.pos[:, who])
        out.append((who[merged], X[merged], torch.full_like(X[merged], -1)))
        who, X = who[~merged], X[~merged]
        leaf = T.child[X] < 0
        lw, lx = who[leaf], X[leaf]
        reps = T.src_count[lx]
        start = torch.cumsum(reps, 0) - reps
        j = torch.arange(int(reps.sum()), device=X.device) - torch.repeat_interleave(start, reps)
        j = j + torch.repeat_interleave(T.src_first[lx], reps)
        lw, lx = torch.repeat_interleave(lw, reps), torch.repeat_interleave(lx, reps)
        lit = T.single[j] > 0
        out.append((lw[lit], lx[lit], j[lit]))
        who, c = who[~leaf], T.child[X[~leaf]]
        who, X = torch.cat([who, who]), torch.cat([c, c + 1])
    return [torch.cat(v) for v in zip(*out)]


def _slabs(lo, hi, p, inv, d):
    """The ray's entry and exit parameters in a box; a still axis is half-open."""
    ta, tb = (lo - p) * inv, (hi - p) * inv
    still = d == 0
    near = torch.where(still, torch.zeros_like(ta), torch.minimum(ta, tb))
    far = torch.where(still, torch.ones_like(ta), torch.maximum(ta, tb))
    out = (still & ((p < lo) | (p >= hi))).any(0)
    t0 = near.amax(0).clamp(min=0.0)
    t1 = far.amin(0).clamp(max=1.0)
    return t0, torch.where(out, t0, t1)


def _trace(T, c, who, C, src, moments):
    """Fluxes (bands, sinks' slots summed by the caller) of these rays: values, per ray."""
    f64 = torch.float64
    p32 = T.pos[:, who]
    merged = src < 0
    j = src.clamp(min=0)
    q = torch.where(merged, T.cen[:, C], T.src[:, j].to(f64))
    q32 = torch.where(merged, T.cen[:, C].detach().to(torch.float32), T.src[:, j])
    band_lum = torch.where(merged, T.bandL[:, C], T.lum[:, j])
    if c.get("background"):
        v = q32 - 0.5
        s = ((v[0] * v[0] + v[1] * v[1]) + v[2] * v[2]).sqrt()
        moved = 0.5 + v * (torch.full_like(s, BG_RADIUS) / s)
        q32 = torch.where(merged & (s > 0), moved, q32)
        q = q32.to(f64)
        C = torch.where(merged, T.locate(_grid(q32)), C)
    S = T.leaf_of[who]
    d32 = q32 - p32
    s2 = (d32[0] * d32[0] + d32[1] * d32[1]) + d32[2] * d32[2]
    live = s2 >= 1e-24
    len32 = s2.sqrt()
    inv32 = torch.where(d32 != 0, d32.reciprocal(), torch.zeros_like(d32))
    p = p32.to(f64)
    d = q - p
    dist2 = (d * d).sum(0)
    length = dist2.sqrt()
    inv = 1.0 / torch.where(d32 != 0, d, torch.ones_like(d))
    nb, nr = T.abar.shape[0], who.numel()
    tau = torch.zeros(nb, nr, dtype=f64, device=who.device)
    ray = torch.nonzero(live)[:, 0]
    X = torch.zeros_like(ray)
    common = None
    if c.get("topdown"):  # the ray starts as the common ancestor of its two ends
        a, b = T.code[S], T.code[C]
        dep = torch.minimum(T.depth[S], T.depth[C])
        a, b = a >> (T.depth[S] - dep), b >> (T.depth[C] - dep)
        x = a ^ b
        common = dep - torch.where(x > 0, _highest_bit(x.clamp(min=1)) + 1, torch.zeros_like(x))
    while ray.numel():
        dX = T.depth[X]

        def above(Y):  # X is a proper ancestor of Y
            e = T.depth[Y] - dX
            return (e > 0) & ((T.code[Y] >> e.clamp(min=0)) == T.code[X])

        if common is None:
            forced = above(S[ray]) | above(C[ray])
        else:
            forced = above(S[ray]) & (dX < common[ray])
        t0, t1 = _slabs(T.lo[X].T, T.hi[X].T, p32[:, ray], inv32[:, ray], d32[:, ray])
        l32 = torch.where(t1 > t0, (t1 - t0) * len32[ray], torch.zeros_like(t0))
        hit = l32 > 0
        split = forced | (hit & (T.child[X] >= 0) &
                          ((T.spread[X] * l32 > np.float32(c["tau_ref"])) |
                           torch.tensor(c["tau_ref"] <= 0, device=X.device)))
        seg = hit & ~split
        r, x = ray[seg], X[seg]
        u0, u1 = _slabs(T.lo[x].T.to(f64), T.hi[x].T.to(f64), p[:, r], inv[:, r], d32[:, r])
        tau = tau.index_add(1, r, T.abar[:, x] * ((u1 - u0).clamp(min=0.0) * length[r]))
        ray, X = ray[split], T.child[X[split]]
        ray, X = torch.cat([ray, ray]), torch.cat([X, X + 1])
    f = band_lum * torch.exp(-tau) / (4.0 * math.pi * torch.where(live, dist2, torch.ones_like(dist2)))
    f = torch.where(live, f, torch.zeros_like(f))
    if c.get("tau_stop"):
        f = torch.where(tau > c["tau_stop"], torch.zeros_like(f), f)
    if moments:
        u = -d / torch.where(live, length, torch.ones_like(length))
        f = f[0]
        return torch.stack([f, *(f * u), f * u[0] * u[0], f * u[1] * u[1], f * u[2] * u[2],
                            f * u[0] * u[1], f * u[0] * u[2], f * u[1] * u[2]])
    return f


def _exact_flux(T, c, sinks, moments=False, chunk=None):
    """Flux rows at the sorted sinks, in their order."""
    rays, _ = _rays_segments(c)
    chunk = chunk or max(256, int(2e6 / max(1.0, rays)))
    rows = []
    for i in range(0, sinks.numel(), chunk):
        own = sinks[i:i + chunk]
        who, C, src = _pairs(T, own, c["theta"])
        f = _trace(T, c, who, C, src, moments)
        slot = torch.full((T.pos.shape[1],), 0, dtype=torch.int64, device=own.device)
        slot[own] = torch.arange(own.numel(), device=own.device)
        rows.append(torch.zeros(f.shape[0], own.numel(), dtype=f.dtype, device=f.device)
                    .index_add(1, slot[who], f))
    return torch.cat(rows, 1)


def exact(c, seed):
    if c["call"] == "sort" or c.get("sub_bucket"):
        return None  # whole numbers; the particle trace has its own quadrature
    if c["call"] == "batch":
        boxes = _batch_boxes(c, seed)
        if sum(work(b)["flops"] for b, _ in boxes) > EXACT_FLOPS:
            return None
        return torch.cat([_exact_one(b, d) for b, d in boxes])
    slow = 12.0 if c.get("background") else 6.0 if c["call"] == "gradient" else 1.0
    if work(c)["flops"] * slow > EXACT_FLOPS:
        return None
    return _exact_one(c, _inputs(c, seed))


def _exact_one(c, d):
    call = c["call"]
    if call == "step" and c["s"] == 1 and not c["sigma"] and not c.get("background") and \
            not c["clumps"] and not c.get("tau_stop"):
        r = (d["gas"].double() - d["src"].double()).norm(dim=0)
        return d["lum"].double() * torch.exp(-c["alpha"] * r) / (4.0 * math.pi * r * r)
    alpha, lum = d["alpha"].double(), d["lum"].double()
    if call == "gradient":
        alpha.requires_grad_(True)
        lum.requires_grad_(True)
    as2 = lambda v: v if v.dim() == 2 else v[None]  # noqa: E731
    T = _ExactTree(d["gas"], as2(alpha), d["src"], as2(lum), d["weight"])
    rank = torch.empty_like(T.perm)
    rank[T.perm] = torch.arange(rank.numel(), device=rank.device)
    if call == "gradient":
        # gradients of each part of the sinks are added up, so that one graph is held at a time
        flux = torch.empty(c["n"], dtype=torch.float64, device=alpha.device)
        ga, gl = torch.zeros_like(alpha), torch.zeros_like(lum)
        step = max(256, int(1e6 / _rays_segments(c)[0]))
        for i in range(0, c["n"], step):
            own = torch.arange(i, min(i + step, c["n"]), device=rank.device)
            f = _exact_flux(T, c, own, chunk=step)[0]
            flux[T.perm[own]] = f.detach()
            a, b = torch.autograd.grad(f, (alpha, lum), d["grad"].double()[T.perm[own]],
                                       retain_graph=True)
            ga += a
            gl += b
        return flux, ga, gl
    if call == "active":
        return _exact_flux(T, c, rank[d["sinks"]])[0]
    rows = _exact_flux(T, c, torch.arange(c["n"], device=rank.device), call == "moments")
    rows = rows[:, rank]
    if call == "moments":
        return rows[0], rows[1:4], rows[4:]
    return rows if call == "bands" else rows[0]
