"""Renumbering of rows around the sizes at which the partition by degree class
changes its path: 32-entry chunks, the 128 entries read together, and a row
much longer than both.  A batched run that skips the visited classes of every
row and a direction-optimizing one (which reads rows front to back) must equal
the oracle, whatever the class counts of the rows are."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13577_gb300 as bfs  # noqa: E402

ROWS = [1, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129, 160, 255, 256, 257, 385, 70001]


@pytest.mark.parametrize("flags", [0, bfs.BFS_UPLOAD_NO_RELABEL], ids=["ordered", "caller_order"])
def test_row_lengths_around_the_chunks(flags):
    # a random graph of 131,072 vertices whose first vertices get rows of these
    # lengths besides: targets of every degree class, both directions stored
    off, col = graphgen.erdos_renyi(17, 20, seed=71)
    n = len(off) - 1
    rng = np.random.default_rng(72)
    src = np.repeat(np.arange(n), np.diff(off))
    keep = (src >= len(ROWS)) & (col >= len(ROWS))
    extra = [rng.choice(np.arange(len(ROWS), n), d, replace=False) for d in ROWS]
    a = np.repeat(np.arange(len(ROWS)), ROWS)
    b = np.concatenate(extra)
    s = np.concatenate([src[keep], a, b])
    t = np.concatenate([col[keep], b, a])
    order = np.lexsort((t, s))
    off = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(s, minlength=n), out=off[1:])
    col = np.ascontiguousarray(t[order].astype(np.int32))
    assert list(np.diff(off)[:len(ROWS)]) == ROWS
    ctx = bfs.Context(0)
    g = bfs.Graph(ctx, off, col, flags=flags)
    roots = np.concatenate([np.arange(len(ROWS)), graphgen.pick_roots(off, 21, seed=11)]).astype(np.int32)
    ref, _ = oracle.bfs_multi(off, col, roots)
    rows = torch.empty((len(roots), n), dtype=torch.int32, device="cuda")
    d = torch.empty(n, dtype=torch.int32, device="cuda")
    for direction in (0, 1):
        g.set_option(bfs.BFS_OPT_DIRECTION, direction)
        rows.fill_(-7)
        g.run_batch(roots, rows)
        g.batch_sync()
        assert np.array_equal(rows.cpu().numpy(), ref)
        for i in range(len(ROWS)):
            g.run(int(roots[i]), d)
            st = g.sync()
            assert np.array_equal(d.cpu().numpy(), ref[i])
            assert st["edges_scanned"] == int(np.diff(off)[ref[i] >= 0].sum())
    g.close()
    ctx.close()
