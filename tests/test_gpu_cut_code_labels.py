"""Piece codes for several labelings at a time, with labelings that shifts can be
chosen to give: one piece, fewer than a code names, more, none shared, and
hubs alone; a graph whose vertices fit the shared-memory table and one whose
cold ones are read from global memory."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import ldd_gen as gen
import oracle

pytestmark = pytest.mark.gpu


def _shifts(G, seed):
    """Shift vectors with the labelings that they give in the first places."""
    rng = np.random.default_rng(seed)
    by_degree = np.argsort(-np.diff(G.row_ptr), kind="stable")
    low = rng.random(G.n) * 0.5

    def centers(ids):
        s = low.copy()
        s[ids] = 30.5 + rng.random(len(ids)) * 0.4
        return s

    hubs_alone = low.copy()
    hubs_alone[rng.choice(by_degree[2000:], 40, replace=False)] = 2.5
    hubs_alone[by_degree[:300]] = 2.9
    return [centers(by_degree[:1]), centers(by_degree[:9]), centers(by_degree[:16]),
            centers(by_degree[:200]), low, hubs_alone,
            centers(rng.choice(by_degree[:G.n // 4], 3000, replace=False))]


@pytest.mark.parametrize("scale", [15, 18])
def test_labelings_of_a_batch(ldd, cuda, scale):
    G = gen.rmat(scale, edge_factor=24, seed=9)
    # the rule for codes: hubs, enough edges, more than one labeling on the device
    assert G.m >= 1 << 19 and int(np.diff(G.row_ptr).max()) > 32
    own = np.diff(G.row_ptr) > 0
    assert (own.sum() > 98304) == (scale == 18)  # cold ends of edges outside the table
    S = _shifts(G, scale)
    g = ldd.LddGraph(G.row_ptr, G.col, validate=False)
    want = []
    for s in S:
        oc, _ = oracle.oracle_ldd(G.row_ptr, G.col, s)
        want.append(oracle.oracle_cut_edges(G.row_ptr, G.col, oc))
    pieces = [len(np.unique(oracle.oracle_ldd(G.row_ptr, G.col, s)[0][own])) for s in S[:5]]
    assert 9 <= pieces[1] <= pieces[2] <= pieces[3] < pieces[4] == int(own.sum())
    t = [torch.from_numpy(s).to(cuda) for s in S]
    c = [torch.empty(G.n, dtype=torch.int32, device=cuda) for _ in S]
    d = [torch.empty(G.n, dtype=torch.int32, device=cuda) for _ in S]
    for pick in ((0, 1), (4, 5), (2, 3, 4), (6, 0, 5), (3, 4, 6, 2), (0, 1, 5, 6),
                 (0, 1, 2, 3, 4, 5, 6)):
        cuts = g.decompose_batch([0.5] * len(pick), [t[i] for i in pick],
                                 [c[i] for i in pick], [d[i] for i in pick])
        assert [int(x) for x in cuts] == [want[i] for i in pick], pick
    g.close()


@pytest.mark.parametrize("scale", [15, 18])
def test_labelings_of_a_union(ldd, cuda, scale):
    G = gen.rmat(scale, edge_factor=24, seed=9)
    H = gen.rmat(9, seed=2)
    S = _shifts(G, scale)
    g, h = ldd.LddGraph(G.row_ptr, G.col, validate=False), ldd.LddGraph(H.row_ptr, H.col)
    u = ldd.LddUnion([h, g, h, g])
    for i in range(len(S)):
        parts = [gen.shifts(H.n, 0.3, i), S[i], gen.shifts(H.n, 5.0, i), S[(i + 3) % len(S)]]
        c, d = np.empty(u.total, np.int32), np.empty(u.total, np.int32)
        cuts = u.decompose([0.3] * 4, np.concatenate(parts), c, d)
        for j, (X, s) in enumerate(zip((H, G, H, G), parts)):
            oc, _ = oracle.oracle_ldd(X.row_ptr, X.col, s)
            assert np.array_equal(c[u.offsets[j]:u.offsets[j + 1]], oc)
            assert cuts[j] == oracle.oracle_cut_edges(X.row_ptr, X.col, oc), (i, j)
    u.close()
    g.close()
    h.close()
