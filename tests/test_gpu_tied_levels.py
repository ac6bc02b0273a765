"""Direct keys whose codes tie across the steps of a bottom-up round: a vertex that
starts one level later than the center that reaches it, a scan that stops at the
pivot's code before it has seen the pivot's own piece, and a center whose push
comes after a start of the same code was counted.  The ids agree with the
fractions, or not; a third center with a better code hides the pair, or not."""
from __future__ import annotations

import numpy as np
import pytest

import ldd_gen as gen
import oracle

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -41  # below the code's last bit


def _check(G, s, c, d):
    oc, od = oracle.oracle_ldd(G.row_ptr, G.col, s)
    bad = np.flatnonzero(c != oc)
    assert bad.size == 0, (bad[:5], c[bad[:5]], oc[bad[:5]])
    assert np.array_equal(d, od)


def _single(ldd, G, s, beta=0.1):
    g = ldd.LddGraph(G.row_ptr, G.col, validate=False)
    g.set_tuning(pull_alpha=1000, pull_gamma=1000)
    c, d = np.empty(G.n, np.int32), np.empty(G.n, np.int32)
    g.decompose(beta, s, c, d)
    st = g.stats()
    _check(G, s, c, d)
    g.close()
    return st


def _union(ldd, G, S, beta=0.1):
    g = ldd.LddGraph(G.row_ptr, G.col, validate=False)
    for s in S:  # one pair per call: another member's order must not answer for it
        u = ldd.LddUnion([g, g])
        u.set_tuning(pull_alpha=1000, pull_gamma=1000)
        quiet = np.linspace(0.0, 0.9, G.n)
        c, d = np.empty(2 * G.n, np.int32), np.empty(2 * G.n, np.int32)
        u.decompose([beta] * 2, np.concatenate([quiet, s]), c, d)
        _check(G, quiet, c[:G.n], d[:G.n])
        _check(G, s, c[G.n:], d[G.n:])
        u.close()
    g.close()


def _star(n, hub, t, third, hub_first):
    G = gen.from_edges(n, [(hub, v) for v in range(n) if v != hub])
    s = np.full(n, 0.25)
    s[hub] = 5.5 + (EPS if hub_first else 0.0)
    s[t] = 4.5 + (0.0 if hub_first else EPS)
    if third:
        s[t + 4] = 4.75
    return G, s


@pytest.mark.parametrize("hub_first", [False, True])
@pytest.mark.parametrize("third", [False, True])
@pytest.mark.parametrize("before", [False, True])
@pytest.mark.parametrize("n", [5000, 70001])
def test_start_one_level_later(ldd, cuda, n, before, third, hub_first):
    """A leaf that starts at the level at which its hub would reach it, with the hub's code.
    n = 70,001: the round has a second pass."""
    hub, t = (n - 1, 3) if before else (2, n - 700)
    G, s = _star(n, hub, t, third, hub_first)
    assert int(s[hub] % 1 * 2 ** 32) == int(s[t] % 1 * 2 ** 32) and s[hub] % 1 != s[t] % 1
    st = _single(ldd, G, s)
    assert st["pull_rounds"] > 0
    assert st["exact_rank"] == 1 or before != hub_first
    _union(ldd, G, [s])


@pytest.mark.parametrize("third", [False, True])
@pytest.mark.parametrize("wide", [0, 5000])
@pytest.mark.parametrize("larger_wins", [False, True])
def test_scan_that_stops_before_the_pivot(ldd, cuda, larger_wins, wide, third):
    """Two hubs with one code, of which the larger has nearly all arcs (the pivot); w has both
    as neighbours (and `wide` others before them), the one with the smaller id first."""
    n = 86000
    small, large, other, w = 80000, 85000, 85001, 79999
    edges = [(large, v) for v in range(5200, 75000)] + [(small, v) for v in range(75000, 75200)]
    edges += [(other, v) for v in range(75300, 75340)] + [(w, small), (w, large)]
    edges += [(w, v) for v in range(100, 100 + wide)]
    edges += [(other, 75199), (small, 74999)]  # one component
    G = gen.from_edges(n, edges)
    s = np.full(n, 0.25)
    s[small] = 5.5 + (0.0 if larger_wins else EPS)
    s[large] = 5.5 + (EPS if larger_wins else 0.0)
    if third:
        s[other] = 5.75
    st = _single(ldd, G, s)
    assert st["pull_rounds"] > 0
    assert st["exact_rank"] == 1 or not larger_wins
    _union(ldd, G, [s])


@pytest.mark.parametrize("start_wins", [False, True])
def test_push_after_a_counted_start(ldd, cuda, start_wins):
    """The first pass of a round appends vertex t (level L + 1).  Vertex a's long row is put off, so
    that the small hub's push reaches it in the second pass: same code as t, smaller id.  In the
    next round w's scan meets a first and stops."""
    n = 80000
    a, hub, t, w, big = 2, 5000, 6000, 7000, 9000
    edges = [(big, v) for v in range(9001, n)] + [(a, v) for v in range(100, 3100)]
    edges += [(hub, a), (a, w), (t, w)]
    G = gen.from_edges(n, edges)
    s = np.full(n, 0.125)
    s[hub] = 5.5 + (0.0 if start_wins else EPS)
    s[big] = 5.25
    s[t] = 4.5 + (EPS if start_wins else 0.0)
    st = _single(ldd, G, s)
    assert st["pull_rounds"] > 1
    assert st["exact_rank"] == 1 or not start_wins
    _union(ldd, G, [s])


@pytest.mark.parametrize("how", ["single", "batch", "replay", "union", "blocks"])
@pytest.mark.parametrize("name", ["rmat", "grid"])
def test_fractions_that_all_tie(ldd, cuda, name, how):
    """Integer shifts and halves: every meeting ties, the ranked keys answer."""
    G = gen.rmat(14, seed=5) if name == "rmat" else gen.grid2d(150, 131)
    g = ldd.LddGraph(G.row_ptr, G.col)
    S = [np.floor(gen.shifts(G.n, 0.1, 1)), np.floor(gen.shifts(G.n, 0.3, 2) * 2.0) / 2.0]
    out = [np.empty(G.n, np.int32) for _ in range(4)]
    if how == "single" or how == "replay":
        g.set_graph_replay(how == "replay")
        for _ in range(3):
            for s in S:
                g.decompose(0.1, s, out[0], out[1])
                _check(G, s, out[0], out[1])
                assert g.stats()["exact_rank"] == 1 or name == "rmat"
    elif how == "batch":
        g.decompose_batch([0.1, 0.3], S, out[:2], out[2:])
        _check(G, S[0], out[0], out[2])
        _check(G, S[1], out[1], out[3])
    elif how == "union":
        u = ldd.LddUnion([g, g])
        c, d = np.empty(2 * G.n, np.int32), np.empty(2 * G.n, np.int32)
        u.decompose([0.1, 0.3], np.concatenate(S), c, d)
        for i, s in enumerate(S):
            _check(G, s, c[i * G.n:(i + 1) * G.n], d[i * G.n:(i + 1) * G.n])
        u.close()
    else:
        c = [np.empty(G.n, np.int32) for _ in S]
        d = [np.empty(G.n, np.int32) for _ in S]
        g.block_decompose([0.1, 0.3], S, c, d)
        _check(G, S[0], c[0], d[0])
    g.close()
