"""Batched runs on graphs with enough entries for the filter of vertices that
every live lane has reached (from 2^20 on), and just too few, against the
oracle in all three loops: with and without the rows' class counts, in the
caller's order, directed, with lanes that end at once (isolated roots) or many
levels before the others (a path hung on the graph)."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13577_gb300 as bfs  # noqa: E402

MIN = 1 << 20


def _graph(kind):
    off, col = graphgen.kronecker(16, 16, seed=81)
    n = len(off) - 1
    src = np.repeat(np.arange(n), np.diff(off))
    if kind == "path":   # 30 new vertices in a row behind the heaviest one
        chain = np.concatenate([[int(np.argmax(np.diff(off)))], np.arange(n, n + 30)])
        src = np.concatenate([src, chain[:-1], chain[1:]])
        col = np.concatenate([col, chain[1:], chain[:-1]])
        n += 30
        order = np.lexsort((col, src))
        src, col = src[order], col[order]
    if kind == "directed":
        keep = (col > src) | (src % 3 == 0)
        src, col = src[keep], col[keep]
    if kind in ("least", "too_few"):
        m = MIN if kind == "least" else MIN - 1
        src, col = src[:m], col[:m]
    off = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(src, minlength=n), out=off[1:])
    return off, np.ascontiguousarray(col.astype(np.int32))


@pytest.mark.parametrize("kind", ["own", "arena", "caller_order", "directed", "path", "least", "too_few"])
def test_filtered_batches_match_oracle(kind):
    off, col = _graph(kind)
    n, nnz = len(off) - 1, len(col)
    assert (nnz >= MIN) == (kind != "too_few")
    arena = torch.empty(16 * nnz + 1024 * n, dtype=torch.uint8, device="cuda") \
        if kind == "arena" else None
    ctx = bfs.Context(0, arena=arena)
    g = bfs.Graph(ctx, off, col, flags=bfs.BFS_UPLOAD_NO_RELABEL if kind == "caller_order" else 0)
    for k in (64, 33, 2):
        roots = graphgen.pick_roots(off, k, seed=12)
        roots[k // 2] = int(np.flatnonzero(np.diff(off) == 0)[3])
        ref, info = oracle.bfs_multi(off, col, roots)
        rows = torch.empty((k, n), dtype=torch.int32, device="cuda")
        for flags in (0, bfs.BFS_HOST_LOOP, bfs.BFS_GRAPH_LOOP):
            rows.fill_(-7)
            g.run_batch(roots, rows, flags=flags)
            st = g.batch_sync()
            assert np.array_equal(rows.cpu().numpy(), ref)
            assert st["levels"] == int(ref.max()) + 1 and st["reached"] == int((ref >= 0).sum())
            assert st["edges_scanned"] == int(((ref >= 0) * np.diff(off)).sum())
    g.close()
    ctx.close()
