"""Mark-and-sweep levels on small graphs (the threshold lowered by the test
hook): vertex counts around a bitmap word, a sweep's tile and a prefix step,
hubs, long paths, directed graphs, sparse and dense levels in turn.  From the
oracle's levels it follows which levels ran dense, and that some did.
Distances must be equal; parents one level closer along an edge."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen
import oracle
from tests import graphs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13577_gb300 as bfs  # noqa: E402

GRAPHS = {
    "pair": lambda: graphs.path(2),
    "path_31": lambda: graphs.path(31),
    "path_33": lambda: graphs.path(33),
    "path_700": lambda: graphs.path(700),
    "star_3000": lambda: graphs.star(3000),
    "complete_64": lambda: graphs.complete(64),
    "grid": lambda: graphs.grid(40, 53),
    "tree_2047": lambda: graphs.binary_tree(2047),
    "random_2049": lambda: graphs.random_graph(2049, 9000, seed=1),
    "random_33000": lambda: graphs.random_graph(33000, 200000, seed=2),
    "two_parts": lambda: graphs.disjoint_union(graphs.random_graph(1000, 4000, seed=3),
                                               graphs.random_graph(999, 3000, seed=4)),
    "directed": lambda: graphs.random_graph(5000, 20000, seed=5, undirected=False),
    "directed_path": lambda: graphs.directed_path(300),
    "kron": lambda: graphgen.kronecker(13, 16, seed=91),
}


@pytest.mark.parametrize("dense_min", [1, 600, 20000])
@pytest.mark.parametrize("how", ["own", "arena", "caller_order"])
def test_dense_levels_of_small_graphs(dense_min, how):
    ran = 0
    for name, make in GRAPHS.items():
        off, col = make()
        n, nnz = len(off) - 1, len(col)
        arena = torch.empty(16 * nnz + 256 * n + (1 << 20), dtype=torch.uint8, device="cuda") \
            if how == "arena" else None
        ctx = bfs.Context(0, arena=arena)
        g = bfs.Graph(ctx, off, col, flags=bfs.BFS_UPLOAD_NO_RELABEL if how == "caller_order" else 0)
        assert bfs.load().bfs_debug_set_dense_min(g.handle, dense_min) == 0
        d = torch.empty(n, dtype=torch.int32, device="cuda")
        p = torch.empty(n, dtype=torch.int32, device="cuda")
        for r in (0, n // 2, n - 1):
            ref, _, info = oracle.bfs(off, col, r)
            entries = np.bincount(ref[ref >= 0], weights=np.diff(off)[ref >= 0])
            ran += int((entries[1:] >= dense_min).sum())
            for parent in (None, p):
                d.fill_(-7)
                g.run(r, d, parent)
                st = g.sync()
                assert np.array_equal(d.cpu().numpy(), ref), (name, r)
                assert (st["levels"], st["edges_scanned"]) == (info["levels"], info["edges_scanned"])
                assert st["reached"] == int((ref >= 0).sum())
            assert oracle.check_bfs(off, col, r, ref, p.cpu().numpy())["ok"], (name, r)
        assert bfs.load().bfs_debug_set_dense_min(g.handle, 0) == 0
        assert bfs.load().bfs_debug_set_dense_min(g.handle, -1) == bfs.BFS_ERR_INVALID_ARG
        g.close()
        ctx.close()
    assert ran >= 10
