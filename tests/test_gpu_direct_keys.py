"""Direct keys (level, leading fraction bits, vertex id in one word) and start
buckets that the round loop fills as it goes: exact where codes tie and the ids
are ordered otherwise than the fractions, where floors exceed what beta
suggests, and where the buckets are filled in several goes."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import ldd_gen as gen
import oracle

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -44  # below the code's last bit


def _check(G, s, c, d):
    oc, od = oracle.oracle_ldd(G.row_ptr, G.col, s)
    assert np.array_equal(c, oc) and np.array_equal(d, od)


def _run(g, G, beta, s):
    c, d = np.empty(G.n, np.int32), np.empty(G.n, np.int32)
    g.decompose(beta, s, c, d)
    _check(G, s, c, d)
    return g.stats()


@pytest.mark.parametrize("later_wins", [False, True])
@pytest.mark.parametrize("n", [9, 30, 41, 2001])
def test_two_tied_centers_on_a_path(ldd, cuda, n, later_wins):
    """Both ends of a path start at one level with equal codes; the middle vertex decides by the
    fractions (paths of up to 32 vertices run in the small-component solver)."""
    G = gen.from_edges(n, [(i, i + 1) for i in range(n - 1)])
    s = np.linspace(0.0, 0.4, n)
    s[0] = s[-1] = n + 0.5
    s[-1 if later_wins else 0] += 2.0 ** -41
    assert int(s[0] * 2 ** 32) == int(s[-1] * 2 ** 32) and s[0] != s[-1]
    g = ldd.LddGraph(G.row_ptr, G.col)
    st = _run(g, G, 0.01, s)
    assert st["exact_rank"] == (1 if later_wins and n % 2 == 1 else 0)
    g.close()


@pytest.mark.parametrize("pull", [0, 1000])
@pytest.mark.parametrize("name", ["rmat", "grid"])
def test_tied_centers(ldd, cuda, name, pull):
    """A few centers at the top level with equal codes and every order of fractions, top-down and
    bottom-up, with windows of levels and without, alone and in a union."""
    G = gen.rmat(14, seed=3) if name == "rmat" else gen.grid2d(120, 97)
    rng = np.random.default_rng(8)
    deg = np.diff(G.row_ptr)
    g = ldd.LddGraph(G.row_ptr, G.col)
    u = ldd.LddUnion([g, g])
    for levels in (1, 8):
        for x in (g, u):
            x.set_tuning(pull_alpha=pull, pull_gamma=1000, window_levels=levels)
        parts = []
        for seed in range(4):
            s = rng.random(G.n) * 0.9
            top = rng.choice(np.flatnonzero(deg > 1), 5, replace=False)
            s[top] = (20 if name == "grid" else 3) + 0.5 + EPS * rng.permutation(5)
            _run(g, G, 0.1, s)
            parts.append(s)
        for i in (0, 2):
            c, d = np.empty(2 * G.n, np.int32), np.empty(2 * G.n, np.int32)
            u.decompose([0.1, 0.1], np.concatenate(parts[i:i + 2]), c, d)
            for j in range(2):
                _check(G, parts[i + j], c[j * G.n:(j + 1) * G.n], d[j * G.n:(j + 1) * G.n])
    u.close()
    g.close()


def test_floors_beyond_what_beta_suggests(ldd, cuda):
    """beta only sizes the level field: larger floors widen it, alone, in a batch, in a union
    (whose lifts come on top) and in a replayed sequence."""
    G = gen.rgg(30000, 4)
    g = ldd.LddGraph(G.row_ptr, G.col)
    items = [gen.shifts(G.n, b, 5 + i) for i, b in enumerate((0.5, 0.001, 0.3, 0.002))]
    items[2][17] = 3.0e6 + 0.25
    for s in items:
        _run(g, G, 50.0, s)
    c = [np.empty(G.n, np.int32) for _ in items]
    d = [np.empty(G.n, np.int32) for _ in items]
    g.decompose_batch([50.0] * 4, items, c, d)
    for s, x, y in zip(items, c, d):
        _check(G, s, x, y)
    u = ldd.LddUnion([g] * 4)
    cc, dd = np.empty(4 * G.n, np.int32), np.empty(4 * G.n, np.int32)
    u.decompose([50.0] * 4, np.concatenate(items), cc, dd)
    for i, s in enumerate(items):
        _check(G, s, cc[i * G.n:(i + 1) * G.n], dd[i * G.n:(i + 1) * G.n])
    g.set_graph_replay(True)
    for beta, s in ((0.5, items[0]), (0.5, items[0]), (0.001, items[1]), (0.5, items[0]),
                    (50.0, items[1])):
        _run(g, G, beta, s)
    u.close()
    g.close()


@pytest.mark.parametrize("low_degree", [0, 1])
@pytest.mark.parametrize("beta", [0.05, 1.0, 8.0])
def test_buckets_filled_in_several_goes(ldd, cuda, beta, low_degree):
    """Components that start long after the others are settled, floors that are nearly all 0
    (large beta), and sizes around the blocks that the fill looks at."""
    rng = np.random.default_rng(2)
    parts, at = [], 0
    for w in (33, 127, 128, 129, 1000, 4097):
        parts += [(at + i, at + i + 1) for i in range(w - 1)]
        parts += [(at + int(i), at + int(j)) for i, j in rng.integers(0, w, (w // 2, 2)) if i != j]
        at += w
    G = gen.from_edges(at + 70, parts)
    s = gen.shifts(G.n, beta, 3)
    s[33:160] += 900.0
    s[161:170] += 40.0
    g = ldd.LddGraph(G.row_ptr, G.col)
    g.set_tuning(low_degree_rounds=low_degree)
    for x in (s, s[::-1].copy(), np.floor(s) + rng.permutation(G.n) / G.n):
        _run(g, G, beta, x)
    t = torch.from_numpy(s).to(cuda)
    c = torch.empty(G.n, dtype=torch.int32, device=cuda)
    d = torch.empty(G.n, dtype=torch.int32, device=cuda)
    g.set_graph_replay(True)
    for _ in range(3):
        g.decompose(beta, t, c, d)
        _check(G, s, c.cpu().numpy(), d.cpu().numpy())
    g.close()
