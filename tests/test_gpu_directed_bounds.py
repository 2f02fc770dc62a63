"""Directed graphs whose reached vertices include some without rows, which the
degree order puts last: the vertices that a traversal's sweeps look at must
follow from the rows' targets, not from the symmetry test, which compares two
64-bit sums over the edges and can be passed by a directed graph.  The four
edges below are such a case: the sums of the hash over them and over their
reversals agree."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13577_gb300 as bfs  # noqa: E402

# vertex of the base graph -> vertex without a row
EDGES = [(1396, 65783), (14222, 66382), (17848, 66904), (32174, 67091)]


def _with_edges(off, col, n, edges):
    src = np.concatenate([np.repeat(np.arange(len(off) - 1), np.diff(off)), [a for a, _ in edges]])
    dst = np.concatenate([col, [b for _, b in edges]])
    order = np.argsort(src, kind="stable")
    new = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(src, minlength=n), out=new[1:])
    return new, np.ascontiguousarray(dst[order].astype(np.int32))


@pytest.mark.parametrize("edges", [EDGES, EDGES[:3]], ids=["passes_symmetry_test", "fails_it"])
def test_targets_without_rows_are_found(edges):
    # no hubs, so that a level of 1 M entries runs dense and batches filter
    off, col = graphgen.erdos_renyi(16, 64, seed=61)
    off, col = _with_edges(off, col, 65536 + 2048, edges)
    n = len(off) - 1
    roots = graphgen.pick_roots(off, 64, seed=10)
    ref, _ = oracle.bfs_multi(off, col, roots)
    assert all((ref[:, b] >= 0).all() for _, b in edges)
    ctx = bfs.Context(0)
    g = bfs.Graph(ctx, off, col)
    d = torch.empty(n, dtype=torch.int32, device="cuda")
    for i in range(4):
        g.run(int(roots[i]), d)
        st = g.sync()
        assert np.array_equal(d.cpu().numpy(), ref[i])
        assert st["reached"] == int((ref[i] >= 0).sum())
    for k in (64, 3):
        rows = torch.empty((k, n), dtype=torch.int32, device="cuda")
        for flags in (0, bfs.BFS_HOST_LOOP, bfs.BFS_GRAPH_LOOP):
            rows.fill_(-7)
            g.run_batch(roots[:k], rows, flags=flags)
            g.batch_sync()
            assert np.array_equal(rows.cpu().numpy(), ref[:k])
    g.close()
    ctx.close()
