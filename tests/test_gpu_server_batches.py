"""How many waiting requests of wide low-degree graphs a worker takes: room for their
padded rows does not make batches much smaller than the caps allow."""
from __future__ import annotations

import re

import numpy as np
import pytest

import ldd_gen as gen
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("entries", [None, 0, 2, 12, 24])
def test_batches_of_wide_rows(ldd, cuda, entries):
    """Rows of 24 entries and a workspace with room for `entries` per vertex (None: for all of
    them): about 65 graphs fit the caps, and with 12 entries half of them keep their rows."""
    caps = dict(max_batch=128, slots=1, max_vertices=1 << 17, max_arcs=1 << 21)
    with pytest.raises(ldd.LddError) as e:
        ldd.LddServer(1 << 12, **caps)
    need = int(re.search(r"need (\d+) bytes", str(e.value)).group(1))
    G = gen.rgg(1990, 3)
    n = 60000  # a long path with a hub: of the other kind, and thousands of levels
    big = gen.from_edges(n, [(i, i + 1) for i in range(n - 1)] + [(0, 2 * i + 5) for i in range(40)])
    assert 16 < int(np.diff(G.row_ptr).max()) <= 24
    g, b = ldd.LddGraph(G.row_ptr, G.col), ldd.LddGraph(big.row_ptr, big.col)
    srv = ldd.LddServer(2 << 30 if entries is None else need + (4 << 17) * entries, **caps)
    most = 0
    for rep in range(3):
        s0 = gen.shifts(big.n, 0.002, rep)
        c0, d0 = np.empty(big.n, np.int32), np.empty(big.n, np.int32)
        jobs = [(gen.shifts(G.n, 0.1, 200 * rep + i), np.empty(G.n, np.int32),
                 np.empty(G.n, np.int32)) for i in range(110)]
        first = srv.submit(b, 0.002, s0, c0, d0)  # the others wait behind this one
        tickets = [srv.submit(g, 0.1, *job) for job in jobs]
        srv.wait(first)
        for t, (s, c, d) in zip(tickets, jobs):
            most = max(most, srv.wait(t)["batch_size"])
            oc, od = oracle.oracle_ldd(G.row_ptr, G.col, s)
            assert np.array_equal(c, oc) and np.array_equal(d, od)
    assert most >= (30 if entries == 12 else 55), most
    assert entries != 12 or most < 55
    srv.close()
    g.close()
    b.close()
