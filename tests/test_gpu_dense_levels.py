"""Levels large enough for the mark-and-sweep expansion of the default
single-source traversal, against the oracle: skewed graphs with and without
the rows' class counts (library allocation, caller's arena, caller's vertex
order), a graph without hubs, vertex counts off every tile size, and a
directed graph whose reached vertices include ones without out-edges.
Distances are whole numbers and must be equal; parents must be one level
closer along an edge."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13577_gb300 as bfs  # noqa: E402


def _induced(off, col, n):
    """Subgraph on the vertices below n."""
    src = np.repeat(np.arange(len(off) - 1), np.diff(off))
    keep = (src < n) & (col < n)
    new = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(src[keep], minlength=n), out=new[1:])
    return new, np.ascontiguousarray(col[keep])


def _directed(off, col):
    """The entries (v, u) with u > v of the vertices v not divisible by 3:
    directed, and a third of the vertices have no out-edges."""
    src = np.repeat(np.arange(len(off) - 1), np.diff(off))
    keep = (col > src) & (src % 3 != 0)
    new = np.zeros(len(off), dtype=np.int64)
    np.cumsum(np.bincount(src[keep], minlength=len(off) - 1), out=new[1:])
    return new, np.ascontiguousarray(col[keep])


@pytest.mark.parametrize("kind", ["skewed", "skewed_odd", "skewed_arena", "skewed_caller_order",
                                  "uniform_odd", "directed"])
def test_dense_levels_match_oracle(kind):
    if kind.startswith("uniform"):
        off, col = graphgen.erdos_renyi(18, 32, seed=41)
    else:
        off, col = graphgen.kronecker(20 if kind != "skewed_odd" else 19, 16, seed=42)
    if kind.endswith("odd"):
        off, col = _induced(off, col, len(off) - 1 - 1237)
    if kind == "directed":
        off, col = _directed(off, col)
    n, nnz = len(off) - 1, len(col)
    arena = torch.empty(16 * nnz + 256 * n, dtype=torch.uint8, device="cuda") \
        if kind == "skewed_arena" else None
    ctx = bfs.Context(0, arena=arena)
    g = bfs.Graph(ctx, off, col,
                  flags=bfs.BFS_UPLOAD_NO_RELABEL if kind == "skewed_caller_order" else 0)
    d = torch.empty(n, dtype=torch.int32, device="cuda")
    p = torch.empty(n, dtype=torch.int32, device="cuda")
    for r in graphgen.pick_roots(off, 3, seed=7):
        ref, _, info = oracle.bfs(off, col, int(r))
        for parent in (None, p):
            g.run(int(r), d, parent)
            st = g.sync()
            got = d.cpu().numpy()
            assert np.array_equal(got, ref)
            assert (st["levels"], st["edges_scanned"]) == (info["levels"], info["edges_scanned"])
            assert st["reached"] == int((ref >= 0).sum())
        assert oracle.check_bfs(off, col, int(r), got, p.cpu().numpy())["ok"]
    g.close()
    ctx.close()


@pytest.mark.parametrize("kind", ["skewed", "arena", "caller_order", "directed"])
@pytest.mark.parametrize("k", [64, 5])
def test_batched_filters_match_oracle(kind, k):
    """Entries to vertices every live lane has reached are filtered out; a
    lane that ends at once (an isolated root) must not keep the filter off
    nor be affected by it."""
    off, col = graphgen.kronecker(16, 8, seed=43)
    if kind == "directed":
        off, col = _directed(off, col)
    n, nnz = len(off) - 1, len(col)
    roots = graphgen.pick_roots(off, k, seed=8)
    roots[k // 2] = int(np.flatnonzero(np.diff(off) == 0)[3])
    arena = torch.empty(16 * nnz + 1024 * n, dtype=torch.uint8, device="cuda") \
        if kind == "arena" else None
    ctx = bfs.Context(0, arena=arena)
    g = bfs.Graph(ctx, off, col, flags=bfs.BFS_UPLOAD_NO_RELABEL if kind == "caller_order" else 0)
    ref, _ = oracle.bfs_multi(off, col, roots)
    for dtype in (torch.int32, torch.int8):
        d = torch.empty((k, n), dtype=dtype, device="cuda")
        g.run_batch(roots, d)
        g.batch_sync()
        assert np.array_equal(d.cpu().numpy().astype(np.int32), ref)
    g.close()
    ctx.close()
