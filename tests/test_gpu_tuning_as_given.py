"""Tuning values are obeyed as they are given, also where they equal the stored
ones, and what a graph reports is what it runs with."""
from __future__ import annotations

import numpy as np
import pytest

import ldd_gen as gen
import oracle

pytestmark = pytest.mark.gpu


def _union_run(u, G, k, beta=0.1):
    parts = [gen.shifts(G.n, beta, 3 + i) for i in range(k)]
    c, d = np.empty(u.total, np.int32), np.empty(u.total, np.int32)
    u.decompose([beta] * k, np.concatenate(parts), c, d)
    for i, s in enumerate(parts):
        oc, od = oracle.oracle_ldd(G.row_ptr, G.col, s)
        assert np.array_equal(c[i * G.n:(i + 1) * G.n], oc)
        assert np.array_equal(d[i * G.n:(i + 1) * G.n], od)
    return u.stats()


def test_levels_per_window_of_a_union(ldd, cuda):
    G = gen.grid2d(90, 80)
    g = ldd.LddGraph(G.row_ptr, G.col)
    u = ldd.LddUnion([g] * 3)
    assert _union_run(u, G, 3)["bfs_windows"] > 0  # untouched: four levels
    u.set_tuning(window_levels=1)  # one, whatever is stored
    assert u.tuning()["window_levels"] == 1 and _union_run(u, G, 3)["bfs_windows"] == 0
    u.set_tuning(window_levels=4)
    assert u.tuning()["window_levels"] == 4 and _union_run(u, G, 3)["bfs_windows"] > 0
    u.set_tuning(window_levels=0)
    assert u.tuning()["window_levels"] == 0 and _union_run(u, G, 3)["bfs_windows"] == 0
    u.close()
    u = ldd.LddUnion([g] * 3)
    u.set_tuning(**u.tuning())  # what it reports, given back
    assert u.tuning()["window_levels"] == 1 and _union_run(u, G, 3)["bfs_windows"] == 0
    t = u.autotune(np.concatenate([gen.shifts(G.n, 0.1, i) for i in range(3)]), reps=1)
    assert u.tuning()["window_levels"] == t["window_levels"]
    assert (_union_run(u, G, 3)["bfs_windows"] > 0) == (t["window_levels"] > 1 and
                                                        t["low_degree_rounds"] == 1)
    u.close()
    g.close()


def test_bottom_up_rounds_of_low_degree_graphs(ldd, cuda):
    """Top-down until a threshold is given: reported as 0; the general one is obeyed."""
    G = gen.rgg(200_000, 3)
    assert int(np.diff(G.row_ptr).max()) <= 32
    g = ldd.LddGraph(G.row_ptr, G.col)
    s = gen.shifts(G.n, 0.5, 4)
    oc, od = oracle.oracle_ldd(G.row_ptr, G.col, s)
    c, d = np.empty(G.n, np.int32), np.empty(G.n, np.int32)

    def pulls(**tuning):
        if tuning:
            g.set_tuning(**tuning)
        for name, value in tuning.items():
            assert g.tuning()[name] == value
        g.decompose(0.5, s, c, d)
        assert np.array_equal(c, oc) and np.array_equal(d, od)
        return g.stats()["pull_rounds"]

    assert g.tuning()["pull_alpha"] == 0 and pulls() == 0
    assert pulls(window_levels=1) == 0
    assert pulls(pull_alpha=14, pull_gamma=64, window_levels=1) > 0
    assert pulls(pull_alpha=0) == 0
    g.close()
    g = ldd.LddGraph(G.row_ptr, G.col)
    u = ldd.LddUnion([g, g])
    assert u.tuning()["pull_alpha"] == 0
    assert _union_run(u, G, 2, 0.5)["pull_rounds"] == 0
    u.set_tuning(pull_alpha=14, pull_gamma=64, window_levels=1)
    assert _union_run(u, G, 2, 0.5)["pull_rounds"] > 0
    u.close()
    g.close()
    H = gen.rmat(12)
    h = ldd.LddGraph(H.row_ptr, H.col)
    assert h.tuning()["pull_alpha"] == 14
    h.close()
