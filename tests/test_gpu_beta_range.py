"""Shifts larger than beta suggests: the wider range is remembered, so that later
calls, batches and replays need no second key pass; and one call with a tiny
beta or a huge shift does not change what others run."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import ldd_gen as gen
import oracle

pytestmark = pytest.mark.gpu


def _bufs(G, cuda, k=1):
    return ([torch.empty(G.n, dtype=torch.int32, device=cuda) for _ in range(k)],
            [torch.empty(G.n, dtype=torch.int32, device=cuda) for _ in range(k)])


def _check(G, s, c, d):
    oc, od = oracle.oracle_ldd(G.row_ptr, G.col, s)
    assert np.array_equal(c.cpu().numpy(), oc) and np.array_equal(d.cpu().numpy(), od)


@pytest.mark.parametrize("name", ["rmat", "grid"])
def test_wider_range_is_remembered(ldd, cuda, name):
    G = gen.rmat(18, edge_factor=4, seed=2) if name == "rmat" else gen.rgg(200_000, 5)
    g = ldd.LddGraph(G.row_ptr, G.col, validate=False)
    (c,), (d,) = _bufs(G, cuda)
    beta = 5.0  # the shifts: floors beyond 36.8 / beta and what 18 id and 32 code bits leave
    drawn = 0.0002
    S = [gen.shifts(G.n, drawn, i) for i in range(4)]
    assert all(20_000 < s.max() < G.n for s in S)
    T = [torch.from_numpy(s).to(cuda) for s in S]
    plain = []
    for s, t in zip(S, T):
        g.decompose(drawn, t, c, d)
        plain.append(g.stats()["launches"])
    g.decompose(beta, T[0], c, d)
    wide = [g.stats()["launches"]]
    for s, t in zip(S, T):
        g.decompose(beta, t, c, d)
        _check(G, s, c, d)
        wide.append(g.stats()["launches"])
    assert wide[1:] == plain and wide[0] > plain[0]  # one key pass each from the second call on
    k = len(S)
    cc, dd = _bufs(G, cuda, k)
    g.decompose_batch([drawn] * k, T, cc, dd, want_cut=False)
    one = g.stats()["launches"]
    g.decompose(beta, T[0], c, d)
    for _ in range(2):
        g.decompose_batch([beta] * k, T, cc, dd, want_cut=False)
        assert g.stats()["launches"] == one  # no member redone alone
        for s, x, y in zip(S, cc, dd):
            _check(G, s, x, y)
    g.close()


def test_replay_with_shifts_beyond_beta(ldd, cuda):
    G = gen.rgg(200_000, 5)
    g = ldd.LddGraph(G.row_ptr, G.col, validate=False)
    g.set_graph_replay(True)
    (c,), (d,) = _bufs(G, cuda)
    replayed = []
    for i in range(6):
        s = gen.shifts(G.n, 0.0002, i)
        g.decompose(5.0, torch.from_numpy(s).to(cuda), c, d)
        _check(G, s, c, d)
        replayed.append(g.stats()["replayed"])
    assert replayed[2:] == [1] * 4
    u = ldd.LddUnion([g, g])
    u.set_graph_replay(True)
    replayed = []
    for i in range(6):
        parts = [gen.shifts(G.n, 0.0002, 2 * i), gen.shifts(G.n, 0.0004, 2 * i + 1)]
        cc, dd = np.empty(u.total, np.int32), np.empty(u.total, np.int32)
        u.decompose([5.0, 7.0], np.concatenate(parts), cc, dd)
        for j, s in enumerate(parts):
            oc, od = oracle.oracle_ldd(G.row_ptr, G.col, s)
            assert np.array_equal(cc[j * G.n:(j + 1) * G.n], oc)
            assert np.array_equal(dd[j * G.n:(j + 1) * G.n], od)
        replayed.append(u.stats()["replayed"])
    assert replayed[2:] == [1] * 4
    u.close()
    g.close()


@pytest.mark.parametrize("beta", [1e-12, 1e-6, 1e-4])
def test_a_tiny_beta_changes_nothing_for_the_others(ldd, cuda, beta):
    """A replayed graph: after one call whose beta leaves few code bits or none, calls with an
    ordinary beta are replayed with the keys they had."""
    G = gen.rmat(17, edge_factor=4, seed=3)
    g = ldd.LddGraph(G.row_ptr, G.col, validate=False)
    g.set_graph_replay(True)
    (c,), (d,) = _bufs(G, cuda)
    s = gen.shifts(G.n, 0.1, 1)
    t = torch.from_numpy(s).to(cuda)
    for b in (0.1, 0.1, beta, beta, 0.1, 0.05, beta, 0.1):
        g.decompose(b, t, c, d)
        _check(G, s, c, d)
    assert g.stats()["replayed"] == 1 and g.stats()["exact_rank"] == 0
    # one huge shift, for which few code bits are left: the next call is as it was before
    for v, top in ((np.argmax(np.diff(G.row_ptr)), 2.0e6), (np.argmin(np.diff(G.row_ptr)), 5.0e7)):
        h = s.copy()
        h[v] = top + 0.5
        for x in (h, s):
            g.decompose(0.1, torch.from_numpy(x).to(cuda), c, d)
            _check(G, x, c, d)
        assert g.stats()["replayed"] == 1 and g.stats()["exact_rank"] == 0
    g.close()
