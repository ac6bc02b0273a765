"""Padded neighbour rows of the low-degree rounds: exact at every row length
around the chunk of eight, for thin frontiers (eight lanes per vertex) and thick
ones (a thread per vertex), in unions of members with different row widths and where a
server has no room for them."""
from __future__ import annotations

import re

import numpy as np
import pytest
import torch

import ldd_gen as gen
import oracle

pytestmark = pytest.mark.gpu


def _graph(n, degrees, seed):
    """Vertices want degrees taken from `degrees` in turn; vertex 0 gets the largest exactly."""
    rng = np.random.default_rng(seed)
    want = np.resize(np.asarray(degrees), n)
    want[0] = max(degrees)
    have = np.zeros(n, int)
    edges = set()
    order = np.argsort(-want, kind="stable")
    for v in order:
        for w in rng.permutation(n):
            if have[v] >= want[v]:
                break
            if v != w and have[w] < want[w] and (min(v, w), max(v, w)) not in edges:
                edges.add((min(v, w), max(v, w)))
                have[v] += 1
                have[w] += 1
    assert have[0] == max(degrees)
    return gen.from_edges(n, sorted((int(a), int(b)) for a, b in edges))


DEGREES = [(0,), (1, 0), (2, 1), (7, 1, 2), (8, 2, 1), (9, 2, 8), (16, 1, 3, 8), (17, 4, 2),
           (24, 25, 7, 1), (32, 8, 1, 31, 9)]


@pytest.mark.parametrize("levels", [1, 8])
@pytest.mark.parametrize("degrees", DEGREES)
def test_row_lengths(ldd, cuda, degrees, levels):
    G = _graph(300, degrees, len(degrees))
    g = ldd.LddGraph(G.row_ptr, G.col)
    g.set_tuning(window_levels=levels)
    for seed, beta in enumerate((0.02, 0.2, 0.8)):
        s = gen.shifts(G.n, beta, seed)
        c, d = np.empty(G.n, np.int32), np.empty(G.n, np.int32)
        g.decompose(beta, s, c, d)
        oc, od = oracle.oracle_ldd(G.row_ptr, G.col, s)
        assert np.array_equal(c, oc) and np.array_equal(d, od)
    g.close()


@pytest.mark.parametrize("side", [60, 700])
def test_union_of_row_widths(ldd, cuda, side):
    """Members with rows of 8 and of more, thin (side 60) and thick (side 700) frontiers."""
    Gs = [gen.grid2d(side, side), _graph(300, (32, 8, 1), 1), gen.rgg(3 * side, 2),
          _graph(300, (0,), 1)]
    gs = [ldd.LddGraph(G.row_ptr, G.col) for G in Gs]
    u = ldd.LddUnion(gs)
    for beta in (0.05, 0.9):
        S = [gen.shifts(G.n, beta, i) for i, G in enumerate(Gs)]
        n = sum(G.n for G in Gs)
        c, d = np.empty(n, np.int32), np.empty(n, np.int32)
        u.decompose([beta] * len(Gs), np.concatenate(S), c, d)
        at = 0
        for G, s in zip(Gs, S):
            oc, od = oracle.oracle_ldd(G.row_ptr, G.col, s)
            assert np.array_equal(c[at:at + G.n], oc) and np.array_equal(d[at:at + G.n], od)
            at += G.n
    u.close()
    for g in gs:
        g.close()


@pytest.mark.parametrize("extra", [0, 1 << 14, 1 << 16, 1 << 20])
def test_server_budget_without_room_for_rows(ldd, cuda, extra):
    """A workspace whose budget leaves no room, little and enough for padded rows takes the same
    requests and gives the same results."""
    caps = dict(max_batch=8, slots=1, max_vertices=8192, max_arcs=1 << 18)
    with pytest.raises(ldd.LddError) as e:
        ldd.LddServer(1 << 12, **caps)
    need = int(re.search(r"need (\d+) bytes", str(e.value)).group(1))
    Gs = [gen.grid2d(60, 60), gen.grid2d(32, 32), _graph(300, (32, 8, 1), 1), gen.rgg(900, 3)]
    gs = [ldd.LddGraph(G.row_ptr, G.col) for G in Gs]
    srv = ldd.LddServer(need + extra, **caps)
    jobs = []
    for i in range(16):
        G = Gs[i % 4]
        jobs.append((i % 4, gen.shifts(G.n, 0.1, i), np.empty(G.n, np.int32),
                     np.empty(G.n, np.int32)))
    tickets = [srv.submit(gs[i], 0.1, s, c, d) for i, s, c, d in jobs]
    for t, (i, s, c, d) in zip(tickets, jobs):
        srv.wait(t)
        oc, od = oracle.oracle_ldd(Gs[i].row_ptr, Gs[i].col, s)
        assert np.array_equal(c, oc) and np.array_equal(d, od)
    srv.close()
    for g in gs:
        g.close()
