"""Cut count of one labeling in one launch: edge counts around the lane's four, the
block's 1024 and a full grid, hubs, labels of any origin, and the sum left at zero."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import ldd_gen as gen

pytestmark = pytest.mark.gpu


def _cut(G, c):
    src = np.repeat(np.arange(G.n), np.diff(G.row_ptr))
    return int((c[src] != c[G.col]).sum()) // 2


@pytest.mark.parametrize("kind", ["path", "star"])
@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 31, 32, 33, 127, 129, 1023, 1024, 1025, 40001])
def test_edge_counts(ldd, cuda, kind, m):
    G = gen.from_edges(m + 1, [(i if kind == "path" else 0, i + 1) for i in range(m)])
    g = ldd.LddGraph(G.row_ptr, G.col)
    rng = np.random.default_rng(m)
    for labels in (1, 2, m + 1):
        c = rng.integers(0, labels, G.n).astype(np.int32)
        for where in (c, torch.from_numpy(c).cuda()):
            assert g.cut_edges(where) == _cut(G, c)
    g.close()


@pytest.mark.parametrize("make", [lambda: gen.grid2d(1200, 1100), lambda: gen.rmat(17, seed=2),
                                  lambda: gen.grid2d(2100, 2050)])
def test_full_grids(ldd, cuda, make):
    """More edges than one pass of the grid takes, and more than one launch takes at all."""
    G = make()
    g = ldd.LddGraph(G.row_ptr, G.col)
    c = np.random.default_rng(3).integers(0, 3, G.n).astype(np.int32)
    want = _cut(G, c)
    assert [g.cut_edges(c) for _ in range(3)] == [want] * 3
    g.close()


@pytest.mark.parametrize("host", [True, False])
def test_batches(ldd, cuda, host):
    """Every count of a batch with host outputs, and of a batch of one, is its own."""
    G = gen.rgg(3000, 7)
    g = ldd.LddGraph(G.row_ptr, G.col)
    for betas in ((0.3,), (0.05, 0.8, 0.3)):
        S = [gen.shifts(G.n, b, 5) for b in betas]
        new = lambda: torch.empty(G.n, dtype=torch.int32, device="cpu" if host else "cuda")
        c, d = [new() for _ in betas], [new() for _ in betas]
        cut = g.decompose_batch(list(betas), S, c, d)
        assert [int(x) for x in cut] == [_cut(G, x.cpu().numpy()) for x in c]
    g.close()
