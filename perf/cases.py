"""Performance cases of the spatial join: what a program that uses this package has it do.

A case names an entry point ("op"), a layer, a grid, a number of points, an
arithmetic form and, for polylines, the window:

  pip   api.pip_join     points against a resident polygon layer
  p2p   api.p2p_join     points against a resident polyline layer, within D (or a window below it)
  host  api.p2p_join_host / api.pip_join_host, points and results in pinned host memory
  round api.Engine.round, many requests of both kinds at once
  once  api.pip_join_once / api.p2p_join_once: build the layer, join, free it

Layers have the structure of paper_1403_0802_gb300/synth.py: a lattice of star
polygons, exact tilings with uneven vertex counts (with or without holes whose
rings are polygons of their own), and random walks.  Tilings and points are
made on the GPU from the seed; walks and stars come from synth itself.
"""
import math

import numpy as np
import torch

from paper_1403_0802_gb300 import api, synth

EXTENT = synth.EXTENT
DEV = "cuda"


# --------------------------------------------------------------------------- cases

def listed():
    return [
        # The smallest serving request (1,000 points) against the serving tiling's grid: latency and launches.
        dict(name="pip_request_1k", op="pip", layer="tiles", n=1_003, grid=1024, form="fp32x", cloud="mixture"),
        # The same for polylines, in the form that serving uses.
        dict(name="p2p_request_1k", op="p2p", layer="lognormal", lines=150_000, n=1_003, grid=512, form="fp32x",
             D=100.0, window=-1.0, cloud="mixture"),
        # A request of the middle of the serving range, in the default form, within a window below the layer's D.
        dict(name="p2p_window_60k_fp64", op="p2p", layer="lognormal", lines=150_000, n=60_007, grid=512, form="fp64",
             D=200.0, window=75.0, cloud="mixture"),
        # The small oracle-checked workload: 1 M uniform points, 1,024 stars, in the default (plain FP64) form.
        dict(name="pip_stars_1m_fp64", op="pip", layer="stars", n=1_000_000, grid=256, form="fp64", cloud="uniform"),
        # The multi-ring layer (holes and the islands in them) from host buffers, default form, an odd number of points.
        dict(name="pip_host_islands_5m_fp64", op="host", layer="islands", n=4_999_999, grid=1280, form="fp64",
             cloud="mixture"),
        # Polygons of hundreds to a hundred thousand vertices: long edge lists per cell.
        dict(name="pip_heavy_10m", op="pip", layer="heavy", n=10_000_000, grid=1536, form="fp32x", cloud="mixture"),
        # The tiling at scale: 100 M points against 40,000 tiles.
        dict(name="pip_tiles_100m", op="pip", layer="tiles", n=100_000_000, grid=1536, form="fp32x", cloud="mixture"),
        # The benchmark's headline: 10 M points, 100,000 walks, D = 100 m.
        dict(name="p2p_walks_10m", op="p2p", layer="walks", lines=100_000, n=10_000_000, grid=448, form="fp32x",
             D=100.0, window=-1.0, cloud="mixture"),
        # The same walks in the default form.
        dict(name="p2p_walks_3m_fp64", op="p2p", layer="walks", lines=100_000, n=3_000_001, grid=448, form="fp64",
             D=100.0, window=-1.0, cloud="mixture"),
        # The polyline join at scale, the largest workload of all.
        dict(name="p2p_lognormal_170m", op="p2p", layer="lognormal", lines=150_000, n=170_000_000, grid=512,
             form="fp32x", D=100.0, window=-1.0, cloud="mixture"),
        # One round of continuous batching: 48 requests of 1,000 to 250,000 points, 70 % polygons, some with windows.
        dict(name="round_48_requests", op="round", requests=48, n_max=250_000, pip_grid=1024, p2p_grid=512,
             lines=150_000, form="fp32x", D=100.0),
        # A program that joins once: the layer's build is most of it.
        dict(name="pip_once_1m", op="once", layer="tiles", n=1_000_000, grid=768, form="fp64", cloud="mixture"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["pip"] * 4 + ["p2p"] * 4 + ["round", "once", "host"])
    form = rng.choice(["fp64", "fp32x"])
    if op == "round":
        return dict(op=op, requests=rng.randint(2, 96), n_max=_log(rng, 20_000, 300_000),
                    pip_grid=rng.choice([512, 768, 1024]), p2p_grid=rng.randint(320, 640),
                    lines=_log(rng, 20_000, 150_000), form=form, D=rng.choice([50.0, 100.0, 200.0]))
    if op == "once":
        op2 = rng.choice(["pip", "p2p"])
        if op2 == "pip":
            return dict(op="once", layer=rng.choice(["tiles", "stars", "islands"]), n=_log(rng, 1_000, 3_000_000),
                        grid=rng.randint(256, 1280), form=form, cloud="mixture")
        return dict(op="once", layer="walks", lines=_log(rng, 5_000, 100_000), n=_log(rng, 1_000, 3_000_000),
                    grid=rng.randint(256, 640), form=form, D=rng.choice([50.0, 100.0]), window=-1.0, cloud="mixture")
    if op == "pip" or (op == "host" and rng.random() < 0.5):
        layer = rng.choice(["stars", "tiles", "islands", "heavy"])
        grid = {"stars": rng.randint(128, 512), "tiles": rng.randint(768, 1536), "islands": rng.randint(768, 1536),
                "heavy": rng.randint(1024, 1536)}[layer]
        top = 10_000_000 if op == "host" or layer == "heavy" else 100_000_000
        return dict(op=op, layer=layer, n=_log(rng, 1_000, top), grid=grid, form=form,
                    cloud=rng.choice(["mixture", "uniform"]))
    D = rng.choice([50.0, 100.0, 200.0])
    layer = rng.choice(["walks", "lognormal"])
    top = 10_000_000 if op == "host" else (20_000_000 if form == "fp64" or layer == "walks" else 100_000_000)
    return dict(op=op, layer=layer, lines=_log(rng, 20_000, 100_000 if layer == "walks" else 150_000),
                n=_log(rng, 1_000, top), grid=rng.randint(384, 640), form=form, D=D,
                window=rng.choice([-1.0, -1.0, round(D * rng.uniform(0.2, 1.0), 3)]), cloud="mixture")


# --------------------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def points(n, cloud, seed):
    """n points: uniform on the extent, or 80 % from 64 Gaussian clusters (sigma = 2,000 m) and 20 % uniform, in
    random order.  Cluster samples outside the extent are drawn once more; the few still outside stay (fixes
    beyond the layer, answered -1)."""
    g = _gen(seed)
    if cloud == "uniform":
        return _rand(g, n, 2).mul_(EXTENT)
    centres = _rand(g, 64, 2).mul_(EXTENT)
    which = torch.randint(0, 80, (n,), generator=g, device=DEV)      # 64..79: the uniform 20 %
    p = _randn(g, n, 2).mul_(0.02 * EXTENT).add_(centres[which.clamp(max=63)])
    out = ((p < 0) | (p >= EXTENT)).any(1).nonzero().squeeze(1)
    p[out] = centres[which[out].clamp(max=63)] + _randn(g, out.numel(), 2) * (0.02 * EXTENT)
    flat = (which >= 64).nonzero().squeeze(1)
    p[flat] = _rand(g, flat.numel(), 2) * EXTENT
    return p


def _starts(counts):
    return torch.cumsum(counts, 0) - counts


def _lognormal(g, n, median, sigma, lo, hi):
    return torch.exp(math.log(median) + sigma * _randn(g, n)).round().clamp(lo, hi).to(torch.int64)


def tiling(seed, nx, ny, side_median, side_cap, giants=3, islands=False):
    """(verts, ring_off, poly_ring_off) on the GPU: an exact tiling of the extent by nx x ny polygons that share
    their sides' vertices, side vertex counts lognormal (sigma 1) up to side_cap, `giants` tiles with side_cap on
    every side.  With islands, 30 % of the tiles have one to four holes, each also a polygon of its own."""
    g = _gen(seed)
    cw, ch = EXTENT / nx, EXTENT / ny
    i = torch.arange(nx + 1, device=DEV, dtype=torch.float64)
    j = torch.arange(ny + 1, device=DEV, dtype=torch.float64)
    jit = (_rand(g, nx + 1, ny + 1, 2) - 0.5) * 0.2
    jit[0, :, 0] = jit[-1, :, 0] = 0.0
    jit[:, 0, 1] = jit[:, -1, 1] = 0.0
    P = torch.stack([(i[:, None] + jit[..., 0]) * cw, (j[None, :] + jit[..., 1]) * ch], -1).clamp_(0.0, EXTENT)
    # sides: horizontal (nx x (ny + 1)) then vertical ((nx + 1) x ny), from a to b
    nh, nv = nx * (ny + 1), (nx + 1) * ny
    a = torch.cat([P[:-1, :].reshape(-1, 2), P[:, :-1].reshape(-1, 2)])
    b = torch.cat([P[1:, :].reshape(-1, 2), P[:, 1:].reshape(-1, 2)])
    hid = torch.arange(nh, device=DEV).view(nx, ny + 1)
    vid = nh + torch.arange(nv, device=DEV).view(nx + 1, ny)
    k = _lognormal(g, nh + nv, side_median, 1.0, 0, side_cap)
    gt = torch.randint(0, nx * ny, (giants,), generator=g, device=DEV)
    gi, gj = gt // ny, gt % ny
    k[torch.cat([hid[gi, gj], hid[gi, gj + 1], vid[gi, gj], vid[gi + 1, gj]])] = side_cap
    edge = torch.zeros(nh + nv, dtype=torch.bool, device=DEV)       # on the extent's boundary: straight
    edge[hid[:, 0]] = edge[hid[:, -1]] = edge[vid[0]] = edge[vid[-1]] = True
    own = torch.repeat_interleave(torch.arange(nh + nv, device=DEV), k)
    t = torch.sort(own + _rand(g, own.numel()).clamp_(1e-6, 1 - 1e-6))[0] - own
    d = b - a
    nrm = torch.stack([-d[:, 1], d[:, 0]], 1) / torch.hypot(d[:, 0], d[:, 1])[:, None]
    off = (_rand(g, own.numel()) * 2 - 1) * (0.1 * min(cw, ch)) * torch.sin(math.pi * t) * (~edge[own])
    Q = a[own] + t[:, None] * d[own] + off[:, None] * nrm[own]
    src = torch.cat([P.reshape(-1, 2), Q]).clamp_(0.0, EXTENT)
    q0 = (nx + 1) * (ny + 1) + _starts(k)
    # pieces of each tile's ring, counterclockwise: corner, side, corner, side, ... ; tile id = row * nx + column
    ti = torch.arange(nx, device=DEV).repeat(ny)
    tj = torch.arange(ny, device=DEV).repeat_interleave(nx)
    corner = lambda u, v: u * (ny + 1) + v
    one = torch.ones_like(ti)
    s0, s1, s2, s3 = hid[ti, tj], vid[ti + 1, tj], hid[ti, tj + 1], vid[ti, tj]
    start = torch.stack([corner(ti, tj), q0[s0], corner(ti + 1, tj), q0[s1], corner(ti + 1, tj + 1),
                         q0[s2] + k[s2] - 1, corner(ti, tj + 1), q0[s3] + k[s3] - 1], 1)
    size = torch.stack([one, k[s0], one, k[s1], one, k[s2], one, k[s3]], 1)
    step = torch.tensor([1, 1, 1, 1, 1, -1, 1, -1], device=DEV).expand_as(start)
    poly = torch.arange(nx * ny, device=DEV)
    ring = [start.reshape(-1), size.reshape(-1), step.reshape(-1), poly.repeat_interleave(8),
            torch.zeros(8 * nx * ny, dtype=torch.int64, device=DEV)]   # start, size, step, polygon, ring in it
    if islands:
        T = nx * ny
        nh_ = torch.where(_rand(g, T) < 0.3, torch.randint(1, 5, (T,), generator=g, device=DEV), 0)
        tile = torch.repeat_interleave(poly, nh_)
        H = tile.numel()
        q = torch.arange(H, device=DEV) - _starts(nh_)[tile]            # which quarter of the tile
        hk = _lognormal(g, H, 12.0, 0.8, 5, 400)
        ho = torch.repeat_interleave(torch.arange(H, device=DEV), hk)
        m = torch.arange(ho.numel(), device=DEV) - _starts(hk)[ho]
        ang = (m + _rand(g, ho.numel())) / hk[ho] * (2 * math.pi)       # one vertex per equal sector: star-shaped
        r = 0.05 + 0.05 * _rand(g, ho.numel())
        cx = (tile % nx + 0.375 + 0.25 * (q % 2) + (_rand(g, H) - 0.5) * 0.04) * cw
        cy = (tile // nx + 0.375 + 0.25 * (q // 2) + (_rand(g, H) - 0.5) * 0.04) * ch
        hv = torch.stack([cx[ho] + r * cw * torch.cos(ang), cy[ho] + r * ch * torch.sin(ang)], 1)
        hs = src.shape[0] + _starts(hk)
        src = torch.cat([src, hv])
        up = torch.ones_like(hs)
        isl = T + torch.arange(H, device=DEV)
        ring = [torch.cat(x) for x in ((ring[0], hs, hs), (ring[1], hk, hk), (ring[2], up, up),
                                       (ring[3], tile, isl), (ring[4], 1 + q, torch.zeros_like(q)))]
    order = torch.sort(ring[3] * 8 + ring[4], stable=True)[1]
    start, size, step, poly, sub = (x[order] for x in ring)
    own = torch.repeat_interleave(torch.arange(size.numel(), device=DEV), size)
    verts = src[start[own] + step[own] * (torch.arange(own.numel(), device=DEV) - _starts(size)[own])]
    rid = torch.unique_consecutive(poly * 8 + sub, return_inverse=True)[1]
    R = int(rid[-1]) + 1
    rsize = torch.zeros(R, dtype=torch.int64, device=DEV).scatter_add_(0, rid, size)
    rpoly = torch.empty(R, dtype=torch.int64, device=DEV).scatter_(0, rid, poly)
    psize = torch.bincount(rpoly)
    offsets = lambda c: torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(c, 0)])
    return verts.contiguous(), offsets(rsize), offsets(psize)


def polygons(layer, seed):
    if layer == "stars":
        s = synth.star_polygons(np.random.default_rng(seed))
        return tuple(torch.as_tensor(x, device=DEV) for x in (s.verts, s.ring_off, s.poly_ring_off))
    if layer == "heavy":
        return tiling(seed, 140, 100, 90.0, 25_000)
    return tiling(seed, 200, 200, 2.6, 1_250, islands=layer == "islands")


def polylines(layer, lines, seed):
    rng = np.random.default_rng(seed)
    if layer == "walks":
        sizes = rng.integers(2, 41, size=lines)
    else:
        sizes = np.clip(np.round(rng.lognormal(math.log(8.0), 0.8, size=lines)), 2, 200).astype(np.int64)
    w = synth.random_walks(rng, sizes)
    return torch.as_tensor(w.verts, device=DEV), torch.as_tensor(w.line_off, device=DEV)


def _is_p2p(case):
    return "D" in case and case["op"] != "round"


def _round_sizes(case):
    """(polygons?, points, window or None) of each request: sizes spread evenly over the logarithm from 1,000 to
    n_max in a fixed order, 70 % polygons, a third of the polyline requests with a window below D."""
    rng = np.random.default_rng(case["requests"])
    out = []
    for u in (rng.permutation(case["requests"]) + 0.5) / case["requests"]:
        pip = bool(rng.random() < 0.7)
        win = float(case["D"] * rng.uniform(0.2, 1.0)) if not pip and rng.random() < 1 / 3 else None
        out.append((pip, int(round(1_000 * (case["n_max"] / 1_000) ** u)), win))
    return out


def _round_requests(case, seed):
    return [(pip, points(n, "mixture", seed * 1000 + k), win)
            for k, (pip, n, win) in enumerate(_round_sizes(case))]


def _arena(reqs):
    """First element of each request's block in the result arena, and the arena's size."""
    size = [-(-p.shape[0] // 64) * 64 for _, p, _ in reqs]
    return [sum(size[:k]) for k in range(len(size))], sum(size)


def _outputs(n, p2p, pinned=False):
    kw = dict(pin_memory=True) if pinned else dict(device=DEV)
    return (torch.empty(n, dtype=torch.int32, **kw), torch.empty(n, dtype=torch.float64, **kw) if p2p else None)


def prepare(case, seed):
    s = {"case": case}
    if case["op"] == "round":
        s["pip"] = api.pip_layer(*polygons("tiles", seed), synth.grid(case["pip_grid"]))
        s["p2p"] = api.p2p_layer(*polylines("lognormal", case["lines"], seed), case["D"], synth.grid(case["p2p_grid"]))
        reqs = _round_requests(case, seed)
        # results in one arena, each request's block at a multiple of 64 elements
        at, total = _arena(reqs)
        s["out"] = (torch.full((total,), -1, dtype=torch.int32, device=DEV),
                    torch.full((total,), math.inf, dtype=torch.float64, device=DEV))
        s["requests"] = []
        for (pip, p, win), b in zip(reqs, at):
            oid, od = (x[b:b + p.shape[0]] for x in s["out"])
            s["requests"].append((s["pip"], p, oid, None) if pip else
                                 (s["p2p"], p, oid, od) + (() if win is None else (win,)))
        s["engine"] = api.Engine(max_points=max(1, sum(p.shape[0] for _, p, _ in reqs)),
                                 max_requests=case["requests"], form=case["form"])
        s["stream"] = torch.cuda.Stream()
        torch.cuda.synchronize()
        # a server has each layer's workspace before its first request: one round of one point each
        one = torch.zeros(1, 2, dtype=torch.float64, device=DEV)
        oid, od = _outputs(1, True)
        s["engine"].round([(s["pip"], one, oid, None), (s["p2p"], one, oid, od)], s["stream"])
        torch.cuda.synchronize()
        return s
    grid = synth.grid(case["grid"])
    p2p = _is_p2p(case)
    geo = polylines(case["layer"], case["lines"], seed) if p2p else polygons(case["layer"], seed)
    s["points"] = points(case["n"], case["cloud"], seed + 1)
    if case["op"] == "once":
        s["geometry"], s["grid"] = geo, grid
        return s
    s["layer"] = api.p2p_layer(*geo, case["D"], grid) if p2p else api.pip_layer(*geo, grid)
    if case["op"] == "host":
        host = torch.empty(case["n"], 2, dtype=torch.float64, pin_memory=True)
        s["points"] = host.copy_(s["points"])
    s["out"] = _outputs(case["n"], p2p, pinned=case["op"] == "host")
    return s


# --------------------------------------------------------------------------- one pass

def run(state):
    c = state["case"]
    if c["op"] == "round":
        state["engine"].round(state["requests"], state["stream"])
        return list(state["out"])
    p, form, p2p = state["points"], c["form"], _is_p2p(c)
    if c["op"] == "once":
        if p2p:
            return list(api.p2p_join_once(p, *state["geometry"], c["D"], state["grid"], form=form))
        return [api.pip_join_once(p, *state["geometry"], state["grid"], form=form)]
    oid, od = state["out"]
    if p2p:
        join = api.p2p_join_host if c["op"] == "host" else api.p2p_join
        win = None if c["window"] < 0 else c["window"]
        return list(join(state["layer"], p, oid, od, form=form, window=win))
    join = api.pip_join_host if c["op"] == "host" else api.pip_join
    return [join(state["layer"], p, oid, form=form)]


# --------------------------------------------------------------------------- work and 64-bit results

# mean vertices of the layers, for the bytes of reading each layer once
_VERTICES = {"stars": 36 * 1_024, "tiles": 760_000, "islands": 1_850_000, "heavy": 9_000_000}


def work(case):
    """Bytes: the points once (16 B), their ids (4 B) and distances (8 B) once, the layer's vertices once (few points
    need few of them: 8 a point at most).  Flops: per point two compares and one orientation against a polygon, or
    the distance to one segment."""
    if case["op"] == "round":
        sizes = _round_sizes(case)
        n_pip = sum(n for pip, n, _ in sizes if pip)
        n_p2p = sum(n for pip, n, _ in sizes if not pip)
        return {"bytes": 20 * n_pip + 28 * n_p2p + 16 * min(8 * n_pip, _VERTICES["tiles"]) +
                16 * min(8 * n_p2p, 11 * case["lines"]),
                "flops": 9 * n_pip + 12 * n_p2p}
    n = case["n"]
    if _is_p2p(case):
        V = case["lines"] * (21 if case["layer"] == "walks" else 11)
        return {"bytes": 28 * n + 16 * min(8 * n, V), "flops": 12 * n}
    return {"bytes": 20 * n + 16 * min(8 * n, _VERTICES[case["layer"]]), "flops": 9 * n}


def _nearest(p, verts, line_off, D, nx):
    """Distance of each point to the nearest segment within D (else inf), plain torch FP64: segments listed under
    the cells that their box widened by D meets, points expanded against their cell's list in chunks."""
    cw = EXTENT / nx
    V = verts.shape[0]
    last = torch.zeros(V, dtype=torch.bool, device=DEV)
    last[line_off[1:] - 1] = True
    i = (~last).nonzero().squeeze(1)
    A, E = verts[i], verts[i + 1] - verts[i]
    L2 = (E * E).sum(1)
    lo = ((torch.minimum(A, A + E) - D - 1e-6) / cw).floor().clamp(0, nx - 1).to(torch.int64)
    hi = ((torch.maximum(A, A + E) + D + 1e-6) / cw).floor().clamp(0, nx - 1).to(torch.int64)
    w = hi - lo + 1
    cnt = w[:, 0] * w[:, 1]
    own = torch.repeat_interleave(torch.arange(i.numel(), device=DEV), cnt)
    k = torch.arange(own.numel(), device=DEV) - _starts(cnt)[own]
    cell = (lo[own, 1] + k // w[own, 0]) * nx + lo[own, 0] + k % w[own, 0]
    cell, order = torch.sort(cell)
    own = own[order]
    c0 = torch.searchsorted(cell, torch.arange(nx * nx + 1, device=DEV))
    inside = ((p >= 0) & (p < EXTENT)).all(1)
    pc = (p / cw).floor().clamp(0, nx - 1).to(torch.int64)
    pc = pc[:, 1] * nx + pc[:, 0]
    n_of = torch.where(inside, c0[pc + 1] - c0[pc], 0)
    best = torch.full((p.shape[0],), math.inf, dtype=torch.float64, device=DEV)
    ends = torch.cumsum(n_of, 0)
    at, N = 0, p.shape[0]
    while at < N:
        base = int(ends[at - 1]) if at else 0
        to = max(at + 1, int(torch.searchsorted(ends, torch.tensor(base + 60_000_000, device=DEV), right=True)))
        to = min(to, N)
        cn = n_of[at:to]
        q = torch.repeat_interleave(torch.arange(at, to, device=DEV), cn)
        s = own[c0[pc[q]] + (torch.arange(q.numel(), device=DEV) - _starts(cn)[q - at])]
        d = p[q] - A[s]
        t = ((d * E[s]).sum(1) / L2[s]).nan_to_num_(0.0).clamp_(0.0, 1.0)
        r = d - t[:, None] * E[s]
        best.scatter_reduce_(0, q, (r * r).sum(1), "amin")
        at = to
    best = best.sqrt()
    return torch.where(best <= D, best, math.inf)


def exact(case, seed):
    """Distances of the polyline joins in 64 bits; polygon ids are whole numbers and have none."""
    if case["op"] == "round":
        verts, off = polylines("lognormal", case["lines"], seed)
        reqs = _round_requests(case, seed)
        at, total = _arena(reqs)
        out = torch.full((total,), math.inf, dtype=torch.float64, device=DEV)
        for (pip, p, win), b in zip(reqs, at):
            if not pip:
                out[b:b + p.shape[0]] = _nearest(p, verts, off, case["D"] if win is None else win, case["p2p_grid"])
        return [None, out]
    if not _is_p2p(case):
        return None
    verts, off = polylines(case["layer"], case["lines"], seed)
    win = case["D"] if case["window"] < 0 else case["window"]
    return [None, _nearest(points(case["n"], case["cloud"], seed + 1), verts, off, win, case["grid"])]
