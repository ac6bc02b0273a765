"""Floors far beyond the number of vertices: the start-bucket tables, and what the
scan over them keeps per tile, grow past the sizes that the vertices ask for."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import ldd_gen as gen
import oracle

pytestmark = pytest.mark.gpu


def _shifts(n, top, seed):
    rng = np.random.default_rng(seed)
    s = rng.random(n) * 40.0
    s[rng.integers(0, n, 3)] = top * np.array([1.0, 0.5, 0.999]) + rng.random(3)
    s[rng.integers(0, n)] = top + 0.5  # a vertex that the round loop handles has the most
    return s


def _check(G, s, c, d):
    oc, od = oracle.oracle_ldd(G.row_ptr, G.col, s)
    assert np.array_equal(c, oc) and np.array_equal(d, od)


def _out(n):
    return np.empty(n, np.int32), np.empty(n, np.int32)


@pytest.mark.parametrize("top", [2_500_000, 10_000_000])
@pytest.mark.parametrize("n", [33, 100, 4096, 4097])
def test_long_start_tables(ldd, cuda, n, top):
    G = gen.from_edges(n, [(i, i + 1) for i in range(n - 1)])
    S = [_shifts(n, top, i) for i in range(3)]
    for how in ("single", "beta", "batch", "ranked", "replay", "union"):
        g = ldd.LddGraph(G.row_ptr, G.col)  # the first call grows the tables
        if how in ("single", "beta"):
            for s in S:
                c, d = _out(n)
                g.decompose(1e-6 if how == "single" else 0.1, s, c, d)
                _check(G, s, c, d)
        elif how == "batch":
            c, d = zip(*(_out(n) for _ in S))
            g.decompose_batch([1e-6] * 3, S, c, d)
            for x in zip(S, c, d):
                _check(G, *x)
        elif how == "ranked":
            perm = np.random.default_rng(n).permutation(n).astype(np.int32)
            levels = S[0].astype(np.int32)
            c, d = _out(n)
            g.decompose_ranked(levels, perm, c, d)
            _check(G, levels + (1.0 - (perm + 1.0) / (n + 2.0)), c, d)
        elif how == "replay":
            g.set_graph_replay(True)
            t = torch.from_numpy(S[1]).to(cuda)
            c = torch.empty(n, dtype=torch.int32, device=cuda)
            d = torch.empty(n, dtype=torch.int32, device=cuda)
            for _ in range(3):
                g.decompose(1e-6, t, c, d)
                _check(G, S[1], c.cpu().numpy(), d.cpu().numpy())
        else:
            u = ldd.LddUnion([g] * 3)
            c, d = _out(3 * n)
            u.decompose([1e-6] * 3, np.concatenate(S), c, d)
            for i, s in enumerate(S):
                _check(G, s, c[i * n:(i + 1) * n], d[i * n:(i + 1) * n])
            u.close()
        g.close()
