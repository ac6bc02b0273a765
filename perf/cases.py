"""The work this framework is timed on, through its public entry points.

A case names a call, its graphs, the exponential parameter of each shift
vector, and where the caller's buffers live:

  call      single   one decomposition and its cut count (decompose, cut_edges)
            batch    pipelined decompositions of one graph, with cut counts
            union    one decomposition of a disjoint union, with cut counts
            blocks   blocks by repeated decomposition
            ranked   the permutation variant and its cut count
            serve    a burst of requests to the request server
  graphs    space-separated specifications:
              grid2d:NXxNY  grid3d:NXxNYxNZ  rmat:SCALE  rgg:N
            and, for a union, rgg:LO-HI*COUNT (sizes spread over a range) or
            any of the above with *COUNT (copies of one graph)
  betas     space-separated, one per shift vector (cycled), or LO-HI for a
            union of graphs that each have their own
  buffers   device, or host (page-locked)
  replay    the graph's captured-graph replay is on

Graphs are the resident part of a program's state; the shift vectors are the
input that changes from call to call, so they come from the seed.  R-MAT
graphs have 16 edges per vertex drawn with (a, b, c, d) = (.57, .19, .19, .05),
random geometric graphs a mean degree of 8, as in the repository's own workloads.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import ldd_gen
import paper_1307_3692_gb300 as ldd

_DEV = "cuda:0"


def listed():
    return [
        # the smallest request a server sees: launches and latency, replayed
        dict(name="grid2d_64", call="single", graphs="grid2d:64x64", betas="0.1",
             buffers="device", replay=True),
        # one small request with the caller's buffers on the host
        dict(name="rmat14_host", call="batch", graphs="rmat:14", betas="0.1", buffers="host",
             replay=False),
        # a thin-frontier graph that fits the caches, once
        dict(name="grid2d_256", call="single", graphs="grid2d:256x256", betas="0.1",
             buffers="device", replay=False),
        # one panel of the paper's figure: a million vertices, hundreds of levels
        dict(name="grid2d_1000", call="single", graphs="grid2d:1000x1000", betas="0.01",
             buffers="device", replay=False),
        # integer shifts and a tie-break permutation, odd size
        dict(name="rgg_150001_ranked", call="ranked", graphs="rgg:150001", betas="0.1",
             buffers="device", replay=False),
        # tree-embedding and sweep callers: several shift vectors of one graph, copied in and
        # out over the host link
        dict(name="rmat20_host", call="batch", graphs="rmat:20", betas="0.02 0.1 0.5",
             buffers="host", replay=False),
        # the large skewed graph, data resident: a sweep over beta
        dict(name="rmat22", call="batch", graphs="rmat:22", betas="0.02 0.1 0.5",
             buffers="device", replay=False),
        # the large regular graph: hundreds of levels with thin frontiers
        dict(name="grid3d_256", call="single", graphs="grid3d:256x256x256", betas="0.01",
             buffers="device", replay=False),
        # many uneven graphs in one call, each with its own beta
        dict(name="rgg_union_64", call="union", graphs="rgg:1000-200000*64", betas="0.02-0.5",
             buffers="device", replay=True),
        # many seeds of one graph in one call
        dict(name="rmat20_union_64", call="union", graphs="rmat:20*64", betas="0.1",
             buffers="device", replay=False),
        # repeated decomposition until no edge is left
        dict(name="rmat20_blocks", call="blocks", graphs="rmat:20", betas="0.5",
             buffers="device", replay=False),
        # a burst of mixed requests: continuous batching, host buffers
        dict(name="serve_burst", call="serve",
             graphs="rmat:14 grid2d:64x64 rmat:16 grid2d:256x256 rmat:18 grid2d:512x512 rmat:20 "
                    "grid2d:1024x1024",
             betas="0.02 0.05 0.1 0.2 0.5", buffers="host", replay=False, requests=24),
    ]


def draw(rng):
    """One more case of the same calls and ranges, sizes spread over their logarithm."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def graph(top):
        kind = rng.choice(("grid2d", "grid3d", "rmat", "rgg"))
        if kind == "grid2d":
            side = size(48, math.isqrt(min(top, 1 << 22)))
            return f"grid2d:{side}x{max(16, int(side * rng.uniform(0.5, 1.0)))}"
        if kind == "grid3d":
            side = size(12, int(top ** (1 / 3)))
            return f"grid3d:{side}x{max(8, int(side * rng.uniform(0.5, 1.0)))}x{side}"
        if kind == "rmat":
            return f"rmat:{rng.randint(11, min(22, top.bit_length() - 1))}"
        return f"rgg:{size(1000, 200000)}"

    def beta():
        return "%.3g" % math.exp(rng.uniform(math.log(0.01), math.log(0.5)))

    call = rng.choice(("single", "single", "batch", "batch", "union", "blocks", "ranked", "serve"))
    c = dict(call=call, buffers="device", replay=False, betas=beta())
    if call == "single":
        c.update(graphs=graph(1 << 24), buffers=rng.choice(("device", "host")),
                 replay=rng.random() < 0.5)
    elif call == "batch":
        c.update(graphs=graph(1 << 22), betas=" ".join(beta() for _ in range(rng.randint(1, 5))),
                 buffers=rng.choice(("device", "host")))
    elif call == "union":
        if rng.random() < 0.5:
            hi = size(2000, 200000)
            c.update(graphs=f"rgg:{max(500, hi // 50)}-{hi}*{rng.randint(2, 64)}",
                     betas="0.02-0.5")
        else:
            c.update(graphs=f"rmat:{rng.randint(11, 18)}*{rng.randint(2, 64)}")
        c["replay"] = rng.random() < 0.5
    elif call == "blocks":
        c.update(graphs=graph(1 << 20), betas="0.5")
    elif call == "ranked":
        c.update(graphs=graph(1 << 20))
    else:
        c.update(graphs=" ".join(graph(1 << 19) for _ in range(rng.randint(2, 6))),
                 betas="0.02 0.05 0.1 0.2 0.5", buffers="host", requests=rng.randint(1, 24))
    return c


# ---------------------------------------------------------------- inputs
def _rmat(scale):
    """(row_ptr, col) on the GPU: symmetric, no loops or repeats, rows ascending."""
    g = torch.Generator(device=_DEV)
    g.manual_seed(7)
    n, m = 1 << scale, 16 << scale
    u = torch.zeros(m, dtype=torch.int64, device=_DEV)
    v = torch.zeros(m, dtype=torch.int64, device=_DEV)
    for _ in range(scale):
        x = torch.rand(m, generator=g, device=_DEV)
        right = (x >= 0.57) & (x < 0.76) | (x >= 0.95)
        u = (u << 1) | (x >= 0.76)
        v = (v << 1) | right
    keep = u != v
    u, v = u[keep], v[keep]
    arcs = torch.unique(torch.cat((u * n + v, v * n + u)))
    row = torch.zeros(n + 1, dtype=torch.int64, device=_DEV)
    row[1:] = torch.bincount(arcs // n, minlength=n).cumsum(0)
    return row.to(torch.int32), (arcs % n).to(torch.int32)


def _csr(spec, seed=11):
    kind, dims = spec.split(":")
    if kind == "rmat":
        return _rmat(int(dims))
    if kind == "rgg":
        g = ldd_gen.rgg(int(dims), seed)
    elif kind == "grid2d":
        g = ldd_gen.grid2d(*map(int, dims.split("x")))
    else:
        g = ldd_gen.grid3d(*map(int, dims.split("x")))
    return torch.from_numpy(g.row_ptr).to(_DEV), torch.from_numpy(g.col).to(_DEV)


def _members(case):
    """[(row_ptr, col)] of the case's distinct graphs, and for each shift vector or request its
    graph's index."""
    specs = case["graphs"].split()
    if case["call"] == "union":
        spec, count = specs[0].split("*")
        if "-" in spec:
            lo, hi = map(int, spec.split(":")[1].split("-"))
            sizes = [s[0] for s in ldd_gen.batch_members(int(count), lo, hi, 0.02, 0.5, 11)]
            return [_csr(f"rgg:{n}", 11 + i) for i, n in enumerate(sizes)], \
                list(range(int(count)))
        return [_csr(spec)], [0] * int(count)
    csrs = [_csr(s) for s in specs]
    if case["call"] == "serve":
        return csrs, [i % len(csrs) for i in range(case["requests"])]
    return csrs, [0] * (48 if case["call"] == "blocks" else len(case["betas"].split()))


def _betas(case, k):
    if "-" in case["betas"]:
        lo, hi = map(float, case["betas"].split("-"))
        return [s[1] for s in ldd_gen.batch_members(k, 1000, 2000, lo, hi, 11)]
    given = [float(b) for b in case["betas"].split()]
    return [given[i % len(given)] for i in range(k)]


def _inputs(case, seed):
    """The graphs, which graph each vector belongs to, the betas, and the vectors on the host."""
    csrs, which = _members(case)
    betas = _betas(case, len(which))
    ns = [csrs[w][0].numel() - 1 for w in which]
    base = (seed % (1 << 30)) * 64
    if case["call"] == "ranked":
        return csrs, which, betas, [ldd_gen.ranked_inputs(ns[0], betas[0], base)]
    return csrs, which, betas, [ldd_gen.shifts(n, b, base + i)
                                for i, (n, b) in enumerate(zip(ns, betas))]


def prepare(case, seed):
    csrs, which, betas, vectors = _inputs(case, seed)
    host = case["buffers"] == "host"

    def place(a):
        t = torch.from_numpy(a)
        return t.pin_memory() if host else t.to(_DEV)

    def out(n):
        t = torch.empty(n, dtype=torch.int32)
        return t.pin_memory() if host else t.to(_DEV)

    state = dict(call=case["call"], betas=betas)
    if case["call"] == "serve":  # before the graphs: it is closed first
        state["server"] = ldd.LddServer(16 << 30)
    graphs = [ldd.LddGraph(rp, col, validate=False) for rp, col in csrs]
    state["graphs"] = graphs
    state["of"] = [graphs[w] for w in which]
    if case["call"] == "ranked":
        state["levels"], state["perm"] = map(place, vectors[0])
    elif case["call"] == "union":
        state["union"] = ldd.LddUnion(state["of"])
        state["shifts"] = place(np.concatenate(vectors))
    else:
        state["shifts"] = [place(v) for v in vectors]
    if case["call"] == "union":
        state["center"], state["dist"] = (out(state["union"].total) for _ in range(2))
    elif case["call"] == "blocks":
        state["arc_block"] = out(graphs[0].nnz)
    else:
        state["center"] = [out(g.n) for g in state["of"]]
        state["dist"] = [out(g.n) for g in state["of"]]
    if case["replay"]:
        (state["union"] if case["call"] == "union" else graphs[0]).set_graph_replay(True)
    return state


def run(state):
    call, betas = state["call"], state["betas"]
    g = state["graphs"][0]
    if call == "union":
        cut = state["union"].decompose(betas, state["shifts"], state["center"], state["dist"])
        return dict(center=state["center"], dist=state["dist"],
                    cut=np.asarray(cut, dtype=np.int64))
    if call == "blocks":
        _, left = g.block_decompose(betas, state["shifts"], out_arc_block=state["arc_block"])
        remaining = np.zeros(len(betas) + 1, dtype=np.int64)
        remaining[:len(left)] = left
        return dict(arc_block=state["arc_block"], remaining=remaining)
    center, dist = state["center"], state["dist"]
    if call == "batch":
        cut = g.decompose_batch(betas, state["shifts"], center, dist)
    elif call == "serve":
        cuts = [np.zeros(1, dtype=np.int64) for _ in betas]
        server = state["server"]
        tickets = [server.submit(*a) for a in zip(state["of"], betas, state["shifts"], center,
                                                  dist, cuts)]
        for t in tickets:
            server.wait(t)
        cut = [int(c[0]) for c in cuts]
    else:
        if call == "ranked":
            g.decompose_ranked(state["levels"], state["perm"], center[0], dist[0])
        else:
            g.decompose(betas[0], state["shifts"][0], center[0], dist[0])
        cut = [g.cut_edges(center[0])]
    return dict(center=center, dist=dist, cut=np.asarray(cut, dtype=np.int64))


def work(case):
    """Every graph, shift vector and result once.  Integer comparisons only: no flops."""
    csrs, which = _members(case)
    total = sum(4 * (rp.numel() + col.numel()) for rp, col in csrs)
    if case["call"] == "union":  # every member is read, the copies too
        total = sum(4 * (csrs[w][0].numel() + csrs[w][1].numel()) for w in which)
    if case["call"] == "blocks":  # the first vector decides nearly every edge
        return dict(bytes=total + 8 * csrs[0][0].numel() + 4 * csrs[0][1].numel(), flops=0)
    return dict(bytes=total + sum(16 * (csrs[w][0].numel() - 1) for w in which), flops=0)


# ---------------------------------------------------------------- the same by plain torch
def _decompose(src, col, a, rank, order):
    """Every vertex joins the u minimising (dist - a_u, rank_u): relaxation to the fixed point."""
    key = ((a.max() - a) << 32) | rank
    while src.numel():
        new = key.scatter_reduce(0, col, key[src] + (1 << 32), "amin")
        if torch.equal(new, key):
            break
        key = new
    center = order[key & 0xffffffff]
    return center, (key >> 32) - (key[center] >> 32)


def _of_shifts(src, col, shifts):
    a = shifts.floor()
    order = torch.sort(shifts - a, descending=True, stable=True).indices
    rank = torch.empty_like(order)
    rank[order] = torch.arange(order.numel(), device=_DEV)
    return _decompose(src, col, a.to(torch.int64), rank, order)


def _arcs(csr):
    rp, col = csr
    n = rp.numel() - 1
    return torch.repeat_interleave(torch.arange(n, device=_DEV), rp.diff().to(torch.int64)), \
        col.to(torch.int64)


def exact(case, seed):
    csrs, which, _, vectors = _inputs(case, seed)
    arcs = [_arcs(c) for c in csrs]
    if case["call"] == "blocks":
        src, col = arcs[0]
        block = torch.full_like(src, -1)
        live, remaining = torch.arange(src.numel(), device=_DEV), np.zeros(len(vectors) + 1, int)
        remaining[0] = int((src < col).sum())
        for i, v in enumerate(vectors):
            center, _ = _of_shifts(src[live], col[live], torch.from_numpy(v).to(_DEV))
            same = center[src[live]] == center[col[live]]
            block[live[same]] = i
            live = live[~same]
            remaining[i + 1] = int((src[live] < col[live]).sum())
            if not live.numel():
                break
        return dict(arc_block=block.to(torch.int32), remaining=remaining)
    centers, dists, cuts = [], [], []
    for w, v in zip(which, vectors):
        src, col = arcs[w]
        if case["call"] == "ranked":
            a, rank = (torch.from_numpy(x).to(_DEV, torch.int64) for x in v)
            order = torch.empty_like(rank)
            order[rank] = torch.arange(rank.numel(), device=_DEV)
            center, dist = _decompose(src, col, a, rank, order)
        else:
            center, dist = _of_shifts(src, col, torch.from_numpy(v).to(_DEV))
        cuts.append(int((center[src] != center[col]).sum()) // 2)
        centers.append(center.to(torch.int32))
        dists.append(dist.to(torch.int32))
    if case["call"] == "union":
        centers, dists = torch.cat(centers), torch.cat(dists)
    return dict(center=centers, dist=dists, cut=np.asarray(cuts, dtype=np.int64))
