"""Batched rows around the depths at which the level planes and the rows'
output change: last levels of 15, 16, 17 (four planes to eight), 125 (the
deepest int8 row), 254, 255 and 256 (levels kept in planes to levels written
straight into the rows); vertex counts that allow four-vertex stores and ones
that do not; partly filled batches; a lane that ends at once; all three loops.
The graph is a path with leaves, so every level has new vertices in some lane."""
from __future__ import annotations

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13577_gb300 as bfs  # noqa: E402


def _path(length, n):
    """Path 0 .. length, vertex v > length hung on path vertex v % length, the
    last vertex isolated."""
    v = np.arange(length)
    h = np.arange(length + 1, n - 1)
    src, dst = np.concatenate([v, h]), np.concatenate([v + 1, h % length])
    s, d = np.concatenate([src, dst]), np.concatenate([dst, src])
    order = np.lexsort((d, s))
    off = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(s, minlength=n), out=off[1:])
    return off, np.ascontiguousarray(d[order].astype(np.int32))


@pytest.mark.parametrize("extra", [40, 43])
@pytest.mark.parametrize("depth", [15, 16, 17, 125, 254, 255, 256])
def test_rows_of_deep_batches(depth, extra):
    n = ((depth + 4) // 4) * 4 + extra
    off, col = _path(depth, n)
    ctx = bfs.Context(0)
    g = bfs.Graph(ctx, off, col)
    for k in (64, 37, 3):
        # lane 0 from the path's end: its last level is `depth`
        roots = np.concatenate([[0], (np.arange(1, k) * 7) % (n - 1)]).astype(np.int32)
        roots[k // 2] = n - 1
        ref, _ = oracle.bfs_multi(off, col, roots)
        assert ref[0].max() == depth and (ref[k // 2] >= 0).sum() == 1
        for dtype in (torch.int32, torch.int8) if ref.max() <= 125 else (torch.int32,):
            rows = torch.empty((k, n), dtype=dtype, device="cuda")
            for flags in (0, bfs.BFS_HOST_LOOP, bfs.BFS_GRAPH_LOOP):
                rows.fill_(-7)
                g.run_batch(roots, rows, flags=flags)
                st = g.batch_sync()
                assert np.array_equal(rows.cpu().numpy().astype(np.int32), ref)
                assert st["levels"] == int(ref.max()) + 1
    g.close()
    ctx.close()
