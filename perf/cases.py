"""Performance cases: what a user of the shortest-path query library has it do.

Every case goes through the public binding (`paper_1503_07192_gb300`), on synthetic
planar graphs made on the GPU from a seed: a 4-neighbour grid, a grid with one random
diagonal per cell, a triangulation of jittered points (a grid with one diagonal per cell,
weighted by Euclidean length: the degrees, uneven component boundaries and weights of a
Delaunay triangulation), and a grid with 10% of its vertices removed (pockets cut off from
the rest: unreachable pairs).  Components are square blocks or kd-tree leaves.

Paths and the ranges that `draw` covers (the listed cases lie inside them):

  step       spq_build + spq_query + spq_free       2^8 .. 2^20 vertices, 1 .. 10M pairs
  pairs      spq_query on a resident handle, device pairs    2^10 .. 2^18 vertices, 1 .. 2M
  host       spq_query with host arrays (a served request)   2^10 .. 2^18 vertices, 1 .. 4,096
  matrix     spq_query_matrix                       1 .. 64 sources, 1,000 .. all vertices
  grad       spq_query_saved + spq_query_backward   2^10 .. 2^18 vertices, 100 .. 1M pairs
  autograd   ShortestPathDistance forward + backward, build included   2^8 .. 2^16 vertices
  paths      spq_query_saved + spq_query_paths      2^10 .. 2^16 vertices, 100 .. 50k pairs
  batch      spq_build_many + spq_query_many        2 .. 48 instances of 1,000 .. 65,536 vertices
  replan     SpqBuildPlan.run (new weights) + SpqQueryPlan.run         the same instances

Weights: "int" (int32, distances below 2^24), "long" (int32 distances above 2^24, which the
library computes in int32 arithmetic), "f32" (float32).
"""

import math

import numpy as np
import torch

import paper_1503_07192_gb300 as spq


# ---------------- cases ----------------


def listed():
    return [
        # the smallest whole use: a 64 x 64 grid in 16 blocks, build and 10,000 pairs
        {"name": "step_grid64", "path": "step", "graph": "grid", "w": 64, "h": 64, "leaf": 256, "weights": "int",
         "pairs": 10_000},
        # travel times in fine units: distances past 2^24, int32 arithmetic throughout
        {"name": "step_long64k", "path": "step", "graph": "tri", "w": 256, "h": 256, "leaf": 512, "weights": "long",
         "pairs": 200_000},
        # the benchmark's size: 2^20 vertices, 1,024 components, 10M pairs, build included
        {"name": "step_grid1m", "path": "step", "graph": "diag", "w": 1024, "h": 1024, "leaf": 1024, "weights": "int",
         "pairs": 10_000_000},
        # a handful of lookups against a resident map: latency
        {"name": "pairs_256", "path": "pairs", "graph": "tri", "w": 512, "h": 512, "leaf": 1024, "weights": "int",
         "pairs": 256},
        # a bulk lookup against a resident map
        {"name": "pairs_1m", "path": "pairs", "graph": "tri", "w": 512, "h": 512, "leaf": 1024, "weights": "int",
         "pairs": 1_000_000},
        # one served request, host arrays in and out, on a float graph of odd size
        {"name": "host_2k", "path": "host", "graph": "tri", "w": 251, "h": 263, "leaf": 700, "weights": "f32",
         "pairs": 2_048},
        # distances from 64 depots to every vertex
        {"name": "matrix_64", "path": "matrix", "graph": "tri", "w": 512, "h": 512, "leaf": 1024, "weights": "int",
         "sources": 64, "targets": 262_144},
        # gradients of a million distances with respect to the edge weights, tables resident
        {"name": "grad_256k", "path": "grad", "graph": "tri", "w": 512, "h": 512, "leaf": 1024, "weights": "f32",
         "pairs": 1_000_000},
        # one training step that learns edge weights: build, distances, gradients
        {"name": "autograd_16k", "path": "autograd", "graph": "tri", "w": 128, "h": 128, "leaf": 512, "weights": "f32",
         "pairs": 100_000},
        # routes themselves (vertex sequences), on a grid with holes: unreachable pairs too
        {"name": "paths_50k", "path": "paths", "graph": "holes", "w": 256, "h": 256, "leaf": 700, "weights": "int",
         "pairs": 50_000, "max_len": 640},
        # many small maps of uneven size at once
        {"name": "batch_48", "path": "batch", "count": 48, "n_lo": 1_000, "n_hi": 65_536, "leaf_lo": 128,
         "leaf_hi": 2_048, "weights": "int", "pairs": 50_000},
        # the same maps again with new weights: a build plan and a query plan replayed
        {"name": "replan_48", "path": "replan", "count": 48, "n_lo": 1_000, "n_hi": 65_536, "leaf_lo": 128,
         "leaf_hi": 2_048, "weights": "int", "pairs": 50_000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides(rng, lo, hi):
    """Sides of a grid of about lo .. hi vertices (hi not passed), up to 3:1."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    r = math.exp(rng.uniform(-0.55, 0.55))
    w = max(8, int(math.sqrt(n * r)))
    return w, max(8, int(n / w))


def draw(rng):
    path = rng.choice(["step", "step", "pairs", "pairs", "host", "matrix", "grad", "autograd", "paths", "batch",
                       "replan"])
    if path in ("batch", "replan"):
        lo = _log(rng, 1_000, 8_000)
        leaf = _log(rng, 128, 512)
        return {"path": path, "count": rng.randint(2, 48), "n_lo": lo, "n_hi": _log(rng, lo, 65_536), "leaf_lo": leaf,
                "leaf_hi": _log(rng, leaf, 2_048), "weights": "int", "pairs": _log(rng, 100, 50_000)}
    graph = rng.choice(["grid", "diag", "tri", "tri", "holes"])
    top = {"step": 1 << 20, "autograd": 1 << 16, "paths": 1 << 16}.get(path, 1 << 18)
    w, h = _sides(rng, 1 << (8 if path in ("step", "autograd") else 10), top)
    case = {"path": path, "graph": graph, "w": w, "h": h}
    # components of 128 .. 2,048 vertices, near the square root of the graph (the paper's
    # choice) and never so small that the boundary graph outgrows the listed cases'
    case["leaf"] = max(_log(rng, 128, 1_024), 1_024 if w * h > 300_000 else 256 if w * h > 40_000 else 128)
    if path in ("grad", "autograd"):
        case["graph"], case["weights"] = "tri", "f32"
    elif path == "paths":
        case["weights"] = "int"
    else:
        case["weights"] = rng.choice(["int", "int", "f32", "long"]) if w * h <= 300_000 else "int"
        if case["weights"] != "int":
            case["graph"] = "tri"
    if path == "matrix":
        case["sources"] = rng.randint(1, 64)
        case["targets"] = _log(rng, 1_000, w * h)
        case["graph"] = "tri" if case["graph"] == "holes" else case["graph"]
    elif path == "paths":
        case["max_len"] = 2 * (w + h)
        case["pairs"] = _log(rng, 100, 50_000)
    else:
        hi = {"step": 10_000_000 if w * h > 300_000 else 1_000_000, "pairs": 2_000_000, "host": 4_096,
              "grad": 1_000_000, "autograd": 100_000}[path]
        case["pairs"] = _log(rng, 100 if path in ("grad", "autograd") else 1, hi)
    return case


# ---------------- inputs (on the GPU, from the seed alone) ----------------


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _kdtree(xy, leaf):
    """Median splits along the longer side of the bounding box while a node holds more than
    `leaf` vertices: (part int32[n], k)."""
    n = xy.shape[0]
    dev = xy.device
    perm = torch.arange(n, device=dev)
    sizes = [n]
    while max(sizes) > leaf:
        t = torch.tensor(sizes, device=dev)
        node = torch.repeat_interleave(torch.arange(len(sizes), device=dev), t)
        p = xy[perm]
        idx = node[:, None].expand(-1, 2)
        lo = torch.full((len(sizes), 2), math.inf, device=dev, dtype=xy.dtype).scatter_reduce(0, idx, p, "amin")
        hi = torch.full((len(sizes), 2), -math.inf, device=dev, dtype=xy.dtype).scatter_reduce(0, idx, p, "amax")
        span = hi - lo
        axis = (span[:, 1] > span[:, 0]).long()
        split = t > leaf
        coord = p.gather(1, axis[node][:, None])[:, 0]
        coord = torch.where(split[node], coord, torch.zeros_like(coord))
        by = torch.sort(coord, stable=True).indices
        by = by[torch.sort(node[by], stable=True).indices]
        perm = perm[by]
        nxt = []
        for s in sizes:
            nxt += [s // 2, s - s // 2] if s > leaf else [s]
        sizes = nxt
    part = torch.empty(n, dtype=torch.int32, device=dev)
    part[perm] = torch.repeat_interleave(torch.arange(len(sizes), device=dev), torch.tensor(sizes, device=dev)).int()
    return part, len(sizes)


def _graph(kind, w, h, leaf, weights, g):
    """dict(n, rp, col, w, part, k) on the GPU."""
    dev = "cuda"
    n = w * h
    ids = torch.arange(n, device=dev).view(h, w)
    u = [ids[:, :-1].reshape(-1), ids[:-1, :].reshape(-1)]
    v = [ids[:, 1:].reshape(-1), ids[1:, :].reshape(-1)]
    if kind in ("diag", "tri"):
        a = ids[:-1, :-1].reshape(-1)
        flip = torch.randint(0, 2, a.shape, generator=g, device=dev)
        u.append(a + flip)
        v.append(a + w + 1 - flip)
    u, v = torch.cat(u), torch.cat(v)
    y, x = torch.div(torch.arange(n, device=dev), w, rounding_mode="floor"), torch.arange(n, device=dev) % w
    xy = torch.stack([x, y], 1).double()
    if kind == "tri":
        xy = xy + 0.7 * (torch.rand(n, 2, generator=g, device=dev, dtype=torch.float64) - 0.5)
    if kind == "holes":
        gone = torch.zeros(n, dtype=torch.bool, device=dev)
        gone[torch.randperm(n, generator=g, device=dev)[: n // 10]] = True
        new = torch.cumsum((~gone).long(), 0) - 1
        ok = ~gone[u] & ~gone[v]
        u, v, xy = new[u[ok]], new[v[ok]], xy[~gone]
        n = n - n // 10
    if kind == "tri":
        length = (xy[u] - xy[v]).square().sum(1).sqrt() / max(w, h)
        if weights == "f32":
            wt = (length * torch.exp(0.25 * torch.randn(length.shape, generator=g, device=dev, dtype=torch.float64)))
            wt = wt.float()
        else:
            wt = torch.round(length * (1e6 if weights == "int" else 2e8)).clamp(min=1).int()
    else:
        wt = torch.randint(1, 101 if kind == "grid" else 1001, u.shape, generator=g, device=dev, dtype=torch.int32)
    s, d, ww = torch.cat([u, v]), torch.cat([v, u]), torch.cat([wt, wt])
    by = torch.sort(s * n + d).indices
    rp = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    rp[1:] = torch.cumsum(torch.bincount(s, minlength=n), 0)
    if kind in ("grid", "diag"):  # square blocks of about `leaf` vertices
        b = max(1, int(math.sqrt(leaf)))
        nbx, nby = -(-w // b), -(-h // b)
        part, k = (torch.div(y, b, rounding_mode="floor") * nbx + torch.div(x, b, rounding_mode="floor")).int(), nbx * nby
    else:
        part, k = _kdtree(xy, leaf)
    return {"n": n, "rp": rp, "col": d[by].int(), "w": ww[by].contiguous(), "part": part, "k": k}


def _pairs(n, q, g):
    return torch.randint(0, n, (q, 2), generator=g, device="cuda", dtype=torch.int32)


def _instances(case, g):
    """Half grids with holes, half triangulations; sizes and leaves log-uniform, the sizes
    spread evenly from n_lo to n_hi so that every seed costs about the same."""
    out = []
    c = case["count"]
    for i in range(c):
        n = case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** ((i + 0.5) / c)
        leaf = int(case["leaf_lo"] * (case["leaf_hi"] / case["leaf_lo"]) ** (((i * 7) % c + 0.5) / c))
        kind = "holes" if i % 2 == 0 else "tri"
        w = max(4, int(math.sqrt(n / (0.9 if kind == "holes" else 1.0))))
        out.append(_graph(kind, w, max(4, int(n / (0.9 if kind == "holes" else 1.0) / w)), leaf, case["weights"], g))
    return out


def _new_weights(gr, g):
    """New int32 weights in [1, 1000], one per undirected edge, in CSR slot order."""
    n, m = gr["n"], gr["col"].shape[0]
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), gr["rp"].diff())
    dst = gr["col"].long()
    key = torch.minimum(src, dst) * n + torch.maximum(src, dst)
    _, inv = torch.unique(key, return_inverse=True)
    return torch.randint(1, 1001, (m,), generator=g, device="cuda", dtype=torch.int32)[inv]


def _inputs(case, seed):
    g = _gen(seed)
    path = case["path"]
    if path in ("batch", "replan"):
        s = {"graphs": _instances(case, g)}
        s["pairs"] = [_pairs(gr["n"], case["pairs"], g) for gr in s["graphs"]]
        if path == "replan":
            s["weights"] = [_new_weights(gr, g) for gr in s["graphs"]]
        return s
    gr = _graph(case["graph"], case["w"], case["h"], case["leaf"], case["weights"], g)
    s = {"graph": gr}
    if path == "matrix":
        s["sources"] = torch.randint(0, gr["n"], (case["sources"],), generator=g, device="cuda", dtype=torch.int32)
        t = torch.arange(gr["n"], device="cuda", dtype=torch.int32)
        if case["targets"] < gr["n"]:
            t = t[torch.randperm(gr["n"], generator=g, device="cuda")[: case["targets"]]].contiguous()
        s["targets"] = t
    else:
        s["pairs"] = _pairs(gr["n"], case["pairs"], g)
    if path in ("grad", "autograd"):
        s["g"] = torch.randn(case["pairs"], generator=g, device="cuda", dtype=torch.float32)
    return s


def _build(gr):
    return spq.spq_build(gr["n"], gr["rp"], gr["col"], gr["w"], gr["part"], gr["k"])


def _tuple(gr):
    return (gr["n"], gr["rp"], gr["col"], gr["w"], gr["part"], gr["k"])


def prepare(case, seed):
    s = _inputs(case, seed)
    path = s["path"] = case["path"]
    if path in ("pairs", "host", "matrix", "grad", "paths"):
        s["h"] = _build(s["graph"])
    if path == "host":
        s["pairs"] = s["pairs"].cpu().numpy()
    if path == "paths":
        s["max_len"] = case["max_len"]
    if path == "replan":
        s["plan"] = spq.spq_build_plan([_tuple(gr) for gr in s["graphs"]])
        s["qplan"] = spq.spq_query_plan(s["plan"].handles, s["pairs"])
    return s


# ---------------- one pass ----------------


def run(s):
    path = s["path"]
    if path == "step":
        h = _build(s["graph"])
        d = spq.spq_query(h, s["pairs"])
        spq.spq_free(h)
        return d
    if path in ("pairs", "host"):
        return spq.spq_query(s["h"], s["pairs"])
    if path == "matrix":
        return spq.spq_query_matrix(s["h"], s["sources"], s["targets"])
    if path == "grad":
        d, saved = spq.spq_query_saved(s["h"], s["pairs"])
        gw = torch.zeros(s["graph"]["col"].shape[0], dtype=torch.float32, device="cuda")
        spq.spq_query_backward(s["h"], s["pairs"], saved, s["g"], gw)
        return [d, saved, gw]
    if path == "autograd":
        gr = s["graph"]
        w = gr["w"].detach().requires_grad_()
        d = spq.ShortestPathDistance.apply(w, gr["rp"], gr["col"], gr["part"], gr["k"], s["pairs"])
        d.backward(s["g"])
        return [d.detach(), w.grad]
    if path == "paths":
        d, saved = spq.spq_query_saved(s["h"], s["pairs"])
        verts, lens = spq.spq_query_paths(s["h"], s["pairs"], saved, s["max_len"])
        # (rows are written up to their length only: padded with -1, as for a ragged batch)
        pad = torch.arange(s["max_len"], device="cuda", dtype=torch.int32)[None, :] >= lens[:, None]
        return [d, verts.masked_fill_(pad, -1), lens]
    if path == "batch":
        hs = spq.spq_build_many([_tuple(gr) for gr in s["graphs"]])
        outs = spq.spq_query_many(hs, s["pairs"])
        for h in hs:
            spq.spq_free(h)
        return outs
    s["plan"].run(s["weights"])  # replan
    return s["qplan"].run()


# ---------------- what a pass cannot do without ----------------


def _shape(n, leaf):
    """(components, boundary vertices of one, |BG|) of n vertices in components of `leaf`."""
    k = max(1.0, n / leaf)
    nb = 4.0 * math.sqrt(leaf) if k > 1.5 else 0.0
    return k, nb, k * nb


def _build_work(n, leaf):
    """The CSR (6 slots a vertex), partition and tables once; updates of the eliminations:
    per table, half the entries times a frontier of about 1.4 sqrt(order) columns."""
    k, nb, nbg = _shape(n, leaf)
    tables = 4.0 * (n * leaf + nbg * nbg)
    upd = 0.7 * (n * leaf * math.sqrt(leaf) + nbg * nbg * math.sqrt(max(nbg, 1.0)))
    return n * (8 + 6 * 8 + 4) + tables, 2.0 * upd


def _query_work(n, leaf, q):
    """Per pair its two table rows, ids and answer; of the boundary matrix each component
    pair's block once; |B1||B2| additions and minima a pair."""
    k, nb, nbg = _shape(n, leaf)
    blocks = k * (k + 1) / 2.0
    hit = blocks * (1.0 - math.exp(-q / blocks))
    return q * (8.0 * nb + 12.0) + hit * 4.0 * nb * nb, 2.0 * q * nb * nb


def work(case):
    path = case["path"]
    if path in ("batch", "replan"):
        b = f = 0.0
        c = case["count"]
        for i in range(c):
            n = case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** ((i + 0.5) / c)
            leaf = case["leaf_lo"] * (case["leaf_hi"] / case["leaf_lo"]) ** (((i * 7) % c + 0.5) / c)
            x, y = _build_work(n, leaf), _query_work(n, leaf, case["pairs"])
            b, f = b + x[0] + y[0], f + x[1] + y[1]
        return {"bytes": b, "flops": f}
    n, leaf = case["w"] * case["h"] * (0.9 if case["graph"] == "holes" else 1.0), case["leaf"]
    k, nb, nbg = _shape(n, leaf)
    hops = 0.6 * (case["w"] + case["h"])  # edges of a typical shortest path
    if path == "step":
        x, y = _build_work(n, leaf), _query_work(n, leaf, case["pairs"])
        return {"bytes": x[0] + y[0], "flops": x[1] + y[1]}
    if path == "matrix":
        ns, nt = case["sources"], case["targets"]
        t1 = min(ns, k) * nb * nbg  # the sources' block rows of the boundary matrix
        return {"bytes": 4.0 * (ns * nt + nt * nb + t1 + ns + nt), "flops": 2.0 * ns * (nb * nbg + nt * nb)}
    x = _query_work(n, leaf, case["pairs"])
    if path in ("pairs", "host"):
        return {"bytes": x[0], "flops": x[1]}
    q = case["pairs"]
    if path == "paths":  # one vertex written a hop
        return {"bytes": x[0] + q * (8.0 + 4.0 + 4.0 * hops), "flops": x[1] + 2.0 * q * hops}
    if path == "grad":
        return {"bytes": x[0] + q * 12.0 + 6.0 * n * 4.0, "flops": x[1] + 2.0 * q * hops}
    y = _build_work(n, leaf)  # autograd
    return {"bytes": x[0] + y[0] + q * 12.0 + 6.0 * n * 4.0, "flops": x[1] + y[1] + 2.0 * q * hops}


# ---------------- 64-bit values ----------------


def _slots(gr):
    """Padded slot table: idx[n, deg] CSR slots (0 where absent), there[n, deg]."""
    deg = gr["rp"].diff()
    j = torch.arange(int(deg.max()), device="cuda")
    there = j[None, :] < deg[:, None]
    return torch.where(there, gr["rp"][:-1, None] + j[None, :], torch.zeros_like(j)[None, :]), there


def _distances(gr, src):
    """Distances from the vertices src to every vertex, [n, len(src)], by Bellman-Ford
    sweeps over the slots in 64 bits (float64; int64 for whole weights)."""
    whole = not gr["w"].is_floating_point()
    inf = (1 << 60) if whole else math.inf
    idx, there = _slots(gr)
    nbr = gr["col"].long()[idx]
    w = gr["w"].to(torch.int64 if whole else torch.float64)[idx]
    w = torch.where(there, w, torch.full_like(w, (1 << 59) if whole else math.inf))
    d = torch.full((gr["n"], src.shape[0]), inf, dtype=w.dtype, device="cuda")
    d[src, torch.arange(src.shape[0], device="cuda")] = 0
    while True:
        e = d
        for j in range(nbr.shape[1]):
            e = torch.minimum(e, d[nbr[:, j]] + w[:, j : j + 1])
        if torch.equal(e, d):
            return d
        d = e


def exact(case, seed):
    path = case["path"]
    if path in ("batch", "replan"):
        return None
    n = case["w"] * case["h"]
    if path == "matrix":
        ns = case["sources"]
    else:
        ns = min(n, case["pairs"])
    hops = case["w"] + case["h"]
    if float(n) * ns * hops > 1.2e11 or n * ns > 1 << 29:  # (the sweeps would take too long)
        return None
    s = _inputs(case, seed)
    gr = s["graph"]
    far = (1 << 29) if case["weights"] != "f32" else math.inf
    if path == "matrix":
        d = _distances(gr, s["sources"].long())[s["targets"].long()].t()
        return torch.where(d < 1 << 50, d, torch.full_like(d, far)).contiguous()
    p = s["pairs"].long()
    src, at = torch.unique(p[:, 0], return_inverse=True)
    dist = _distances(gr, src)
    d = dist[p[:, 1], at]
    out = torch.where(d < (1 << 50), d, torch.full_like(d, far))
    if path in ("step", "pairs", "host"):
        return out
    if path == "paths":
        return [out, None, None]  # (which of several shortest paths is not a computed number)
    # gradients: every pair's path walked back from its target, the slot towards the target
    # taking the pair's upstream gradient
    idx, there = _slots(gr)
    nbr = gr["col"].long()[idx]
    w = torch.where(there, gr["w"].double()[idx], torch.full(idx.shape, math.inf, dtype=torch.float64, device="cuda"))
    owner = torch.repeat_interleave(torch.arange(gr["n"], device="cuda"), gr["rp"].diff())
    fwd = owner * gr["n"] + gr["col"].long()
    rev = torch.searchsorted(fwd, gr["col"].long() * gr["n"] + owner)  # the slot of the opposite direction
    grad = torch.zeros(gr["col"].shape[0], dtype=torch.float64, device="cuda")
    cur, up = p[:, 1].clone(), s["g"].double()
    live = torch.isfinite(d) & (cur != p[:, 0])
    cur, at, up, home = cur[live], at[live], up[live], p[:, 0][live]
    while cur.numel():
        j = (dist[nbr[cur], at[:, None]] + w[cur]).argmin(1)
        grad.index_add_(0, rev[idx[cur, j]], up)
        cur = nbr[cur, j]
        go = cur != home
        cur, at, up, home = cur[go], at[go], up[go], home[go]
    return [out, None, grad] if path == "grad" else [out, grad]
