"""Cut counts by piece codes (graphs with hubs and at least 2^19 edges):
labelings with one piece, a few, more than a code names, and none shared with a
hub; one to four at a time; in unions of members on both sides of the rule."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import ldd_gen as gen
import oracle

pytestmark = pytest.mark.gpu


def _labelings(G, seed):
    rng = np.random.default_rng(seed)
    by_degree = np.argsort(-np.diff(G.row_ptr), kind="stable")
    few = by_degree[rng.integers(0, 3, G.n)]
    many = by_degree[rng.integers(0, 40, G.n)]
    hubs_alone = rng.integers(0, G.n, G.n)
    hubs_alone[by_degree[:300]] = by_degree[:300]
    mostly = np.where(rng.random(G.n) < 0.98, by_degree[0], rng.integers(0, G.n, G.n))
    return [x.astype(np.int32) for x in (np.zeros(G.n), few, many, np.arange(G.n), hubs_alone,
                                         mostly)]


@pytest.mark.parametrize("scale", [15, 17])
def test_any_labelling(ldd, cuda, scale):
    """R-MAT 15 fits the shared-memory table whole, R-MAT 17 does not."""
    G = gen.rmat(scale, edge_factor=24, seed=9)
    assert G.m >= 1 << 19
    g = ldd.LddGraph(G.row_ptr, G.col, validate=False)
    for lab in _labelings(G, scale):
        want = oracle.oracle_cut_edges(G.row_ptr, G.col, lab)
        assert g.cut_edges(lab) == want
        assert g.cut_edges(torch.from_numpy(lab).to(cuda)) == want
    g.close()


@pytest.mark.parametrize("k", [1, 2, 3, 4, 6])
def test_batches(ldd, cuda, k):
    G = gen.rmat(15, edge_factor=24, seed=9)
    betas = [0.05, 3.0, 0.5, 9.0, 0.2, 1.0][:k]  # large beta: thousands of pieces
    sh = [torch.from_numpy(gen.shifts(G.n, b, 3 + i)).to(cuda) for i, b in enumerate(betas)]
    c = [torch.empty(G.n, dtype=torch.int32, device=cuda) for _ in betas]
    d = [torch.empty(G.n, dtype=torch.int32, device=cuda) for _ in betas]
    g = ldd.LddGraph(G.row_ptr, G.col, validate=False)
    for _ in range(2):
        cuts = g.decompose_batch(betas, sh, c, d)
        for x, cut in zip(c, cuts):
            assert cut == oracle.oracle_cut_edges(G.row_ptr, G.col, x.cpu().numpy())
    g.close()


def test_unions(ldd, cuda):
    """Members of every size, an empty one, hot tables larger and smaller than the member."""
    Gs = [gen.rmat(17, edge_factor=6, seed=4), gen.rmat(12), gen.grid2d(61, 50), gen.from_edges(5, []),
          gen.rmat(15), gen.grid2d(7, 3), gen.rmat(12), gen.rgg(3001, 2)]
    gs = [ldd.LddGraph(G.row_ptr, G.col, validate=False) for G in Gs]
    order = [0, 1, 2, 3, 4, 5, 6, 7, 4, 1, 0]
    u = ldd.LddUnion([gs[i] for i in order])
    for replay in (False, True):
        u.set_graph_replay(replay)
        for beta in (0.1, 4.0):
            parts = [gen.shifts(Gs[i].n, beta, 20 + j) for j, i in enumerate(order)]
            c, d = np.empty(u.total, np.int32), np.empty(u.total, np.int32)
            cuts = u.decompose([beta] * len(order), np.concatenate(parts), c, d)
            for j, i in enumerate(order):
                own = c[u.offsets[j]:u.offsets[j + 1]]
                assert cuts[j] == oracle.oracle_cut_edges(Gs[i].row_ptr, Gs[i].col, own), (j, beta)
    u.close()
    for g in gs:
        g.close()
