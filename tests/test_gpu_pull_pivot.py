"""Large bottom-up rounds stop their scans at a pivot rank and let the frontier
vertices of smaller rank push (k_bfs.cu): exact where the smallest rank at the
frontier's level belongs to a center that few candidates can reach, where two
large pieces meet, and where rows end on either side of the pass's shares."""
from __future__ import annotations

import numpy as np
import pytest

import ldd_gen as gen
import oracle

pytestmark = pytest.mark.gpu


def _rows():
    """A hub joined to every vertex but the rest of the rows' own leaves: rows of the lengths
    around the scan limits, and leaves that see one of them before the hub."""
    n = 90_000
    u, v = [np.zeros(n - 1000, np.int64)], [np.arange(1000, n)]
    for i, d in enumerate((7, 8, 9, 31, 32, 33, 255, 256, 257, 1023, 1024, 1025, 2055, 2056, 2057,
                           20_000)):
        w = 1 + i
        leaves = (np.arange(d, dtype=np.int64) * 37 + i * 101) % (n - 1000) + 1000
        u.append(np.full(d, w)), v.append(leaves)
        u.append(np.array([w])), v.append(np.array([1 + (i + 1) % 16]))
    rng = np.random.default_rng(3)
    u.append(rng.integers(1000, n, 60_000)), v.append(rng.integers(1000, n, 60_000))
    u, v = np.concatenate(u), np.concatenate(v)
    keep = u != v
    a = np.unique(np.concatenate([u[keep] * n + v[keep], v[keep] * n + u[keep]]))
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(a // n, minlength=n))
    return gen.CSR("rows", rp, (a % n).astype(np.int32))


GRAPHS = {"rmat17": lambda: gen.rmat(17, seed=5), "rows": _rows}


def _shifts(G, kind, seed):
    """Every vertex below one, and centers at one level: the largest hub, and `few` low-degree
    vertices or the next `hubs` with larger fractions (smaller ranks)."""
    rng = np.random.default_rng(seed)
    deg = np.diff(G.row_ptr)
    order = np.argsort(-deg, kind="stable")
    s = rng.random(G.n) * 0.9
    s[order[0]] = 3.25
    low = np.flatnonzero((deg > 0) & (deg < 4))
    if kind == "few":
        s[rng.choice(low, 40, replace=False)] = 3.5 + 0.01 * np.arange(40)
    elif kind == "hubs":
        s[order[1:12]] = 3.3 + 0.05 * np.arange(11)
    elif kind == "many":
        s[rng.choice(low, low.size // 2, replace=False)] += 3.0
    return s


@pytest.mark.parametrize("kind", ["alone", "few", "hubs", "many"])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_pivot_rounds_exact(ldd, cuda, name, kind):
    G = GRAPHS[name]()
    g = ldd.LddGraph(G.row_ptr, G.col)
    assert g.stats()["n_active"] >= 1 << 16
    c, d = np.empty(G.n, np.int32), np.empty(G.n, np.int32)
    base = g.tuning()
    for seed, tune in ((1, {}), (2, dict(pull_alpha=1000, pull_gamma=1000)),
                       (3, dict(bfs_blocks_per_sm=2, pull_alpha=1000, pull_gamma=1000))):
        g.set_tuning(**(base | tune))
        s = _shifts(G, kind, seed)
        g.decompose(0.5, s, c, d)
        oc, od = oracle.oracle_ldd(G.row_ptr, G.col, s)
        assert np.array_equal(c, oc) and np.array_equal(d, od), (seed, tune)
    assert g.stats()["pull_rounds"] > 0
    g.close()


@pytest.mark.parametrize("extra", [3, 2100], ids=["shared_tables", "global_tables"])
def test_pivot_rounds_exact_in_unions(ldd, cuda, extra):
    big = [GRAPHS["rmat17"](), GRAPHS["rows"]()]
    small = gen.rmat(6, seed=2)
    gs = [ldd.LddGraph(G.row_ptr, G.col) for G in (*big, small)]
    members = [(big[0], gs[0], "few"), (big[1], gs[1], "hubs"), (big[0], gs[0], "many"),
               *[(small, gs[2], "alone")] * extra]
    u = ldd.LddUnion([m[1] for m in members])
    parts = [_shifts(m[0], m[2], 10 + i % 7) for i, m in enumerate(members)]
    c, d = np.empty(u.total, np.int32), np.empty(u.total, np.int32)
    for per_sm in (1, 2):
        u.set_tuning(bfs_blocks_per_sm=per_sm, pull_alpha=1000, pull_gamma=1000)
        u.decompose([0.5] * len(members), np.concatenate(parts), c, d)
        assert u.stats()["pull_rounds"] > 0
        at = 0
        for i, (G, _, _) in enumerate(members):
            if i < 12:
                oc, od = oracle.oracle_ldd(G.row_ptr, G.col, parts[i])
                assert np.array_equal(c[at:at + G.n], oc) and np.array_equal(d[at:at + G.n], od), i
            at += G.n
    u.close()
    for g in gs:
        g.close()


@pytest.mark.parametrize("beta", [0.05, 0.6])
def test_scan_steps(ldd, cuda, beta):
    """Bottom-up rows of every length around the scan's steps, the only settled neighbour last."""
    lengths = [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 15, 16, 17, 30, 31, 32, 33, 34, 40] * 3
    pool = 40
    c = pool + len(lengths)  # the center: the largest id, so the last of every row
    edges = [(d, pool + i) for i, n in enumerate(lengths) for d in range(n - 1)]
    edges += [(pool + i, c) for i in range(len(lengths))]
    G = gen.from_edges(c + 1, edges)
    g = ldd.LddGraph(G.row_ptr, G.col)
    u = ldd.LddUnion([g, g])
    for x in (g, u):
        x.set_tuning(pull_alpha=1000, pull_gamma=1000)
    parts = []
    for seed in range(2):
        s = gen.shifts(G.n, beta, seed)
        s[c] = s.max() + 1.25
        oc, od = oracle.oracle_ldd(G.row_ptr, G.col, s)
        cc, dd = np.empty(G.n, np.int32), np.empty(G.n, np.int32)
        g.decompose(beta, s, cc, dd)
        assert np.array_equal(cc, oc) and np.array_equal(dd, od)
        parts.append((s, oc, od))
    cc, dd = np.empty(2 * G.n, np.int32), np.empty(2 * G.n, np.int32)
    u.decompose([beta, beta], np.concatenate([p[0] for p in parts]), cc, dd)
    assert np.array_equal(cc, np.concatenate([p[1] for p in parts]))
    assert np.array_equal(dd, np.concatenate([p[2] for p in parts]))
    u.close()
    g.close()
