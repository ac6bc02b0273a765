"""Padded neighbour rows and piece codes are for speed only: where device memory is
too short for rows, graphs, unions and block decompositions run without, and
unions without hubs have no buffers for codes."""
from __future__ import annotations

import gc

import numpy as np
import pytest
import torch

import ldd_gen as gen
import oracle

pytestmark = pytest.mark.gpu


class _Hold:
    """Leaves `free` bytes of device memory free, in what torch holds."""

    def __init__(self, free):
        gc.collect()
        torch.cuda.empty_cache()
        torch.cuda.synchronize()
        have = torch.cuda.mem_get_info()[0]
        self.t = torch.empty(have - free, dtype=torch.uint8, device="cuda")

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        del self.t
        torch.cuda.empty_cache()


def _wide_path(n, chords=30):
    """A path with chords at vertex 0, whose row of 31 makes every padded row 32 wide."""
    e = [(i, i + 1) for i in range(n - 1)] + [(0, (i + 1) * (n // 90)) for i in range(chords)]
    a = np.array(e, dtype=np.int64)
    src = np.concatenate([a[:, 0], a[:, 1]])
    dst = np.concatenate([a[:, 1], a[:, 0]])
    order = np.lexsort((dst, src))
    row = np.zeros(n + 1, np.int64)
    np.add.at(row, src + 1, 1)
    return np.cumsum(row).astype(np.int32), dst[order].astype(np.int32)


def _used(make):
    """Device memory that `make` takes, once its kernels are loaded."""
    for _ in range(2):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        x = make()
        torch.cuda.synchronize()
        took = before - torch.cuda.mem_get_info()[0]
        x.close()
    return took


def _run(g, n, s, oc, od, windows):
    c, d = np.empty(n, np.int32), np.empty(n, np.int32)
    g.decompose(0.5, s, c, d)
    assert np.array_equal(c, oc) and np.array_equal(d, od)
    assert (g.stats()["bfs_windows"] > 0) == windows


def test_graph_union_and_blocks_without_rows(ldd, cuda):
    n = 1 << 21
    row, col = _wide_path(n)
    assert int(np.diff(row).max()) == 31
    rows = n * 32 * 4
    s = gen.shifts(n, 0.5, 3)
    oc, od = oracle.oracle_ldd(row, col, s)
    make = lambda: ldd.LddGraph(row, col, validate=False)  # noqa: E731
    took = _used(make)
    assert took > rows
    g = make()
    _run(g, n, s, oc, od, True)
    g.close()
    with _Hold(took - rows // 2):
        g = make()
        assert g.tuning()["pull_alpha"] == 14  # the general rounds' default
        _run(g, n, s, oc, od, False)
        g.close()

    g = make()
    union = lambda: ldd.LddUnion([g, g])  # noqa: E731
    took = _used(union)
    assert took > 2 * rows
    c, d = np.empty(2 * n, np.int32), np.empty(2 * n, np.int32)
    for short in (False, True):
        with _Hold((took - rows) if short else 2 * took + 8 * rows):
            u = union()
            u.decompose([0.5] * 2, np.concatenate([s, s]), c, d)
            assert (u.stats()["bfs_windows"] > 0) == (not short)
            for i in range(2):
                assert np.array_equal(c[i * n:(i + 1) * n], oc)
                assert np.array_equal(d[i * n:(i + 1) * n], od)
            u.close()
    g.close()

    def blocks():
        h = make()
        out = [np.empty(n, np.int32) for _ in range(4)]
        blk = np.empty(len(col), np.int32)
        k, left = h.block_decompose([0.5] * 2, [s, s], out[:2], out[2:], blk)[:2]
        assert np.array_equal(out[0], oc) and np.array_equal(out[2], od)
        h.out = (k, left, blk, *out)
        return h

    both = _used(blocks)
    h = blocks()
    want = h.out
    h.close()
    with _Hold(both - rows // 2):  # rows for the graph, or none: not for the residual graphs
        h = blocks()
        for x, y in zip(want, h.out):
            assert np.array_equal(x, y)
        h.close()


def test_union_without_hubs_has_no_code_buffers(ldd, cuda):
    n = 1 << 21
    took = []
    for chords in (30, 60):
        row, col = _wide_path(n, chords)
        g = ldd.LddGraph(row, col, validate=False)
        took.append(_used(lambda: ldd.LddUnion([g, g])))
        g.close()
    rows = 2 * n * 32 * 4
    codes = 2 * n * (2 + 2 + 6)  # code words of vertices, groups and hot table, and that table
    assert abs(took[1] - (took[0] - rows) - codes) < codes // 4, (took, rows, codes)
