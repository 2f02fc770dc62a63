"""bfs_run_static up to its limits, against the oracle: levels of more than
8 M entries (skewed and uniform graphs, an odd vertex count near the largest
accepted), entry counts on both sides of the 2^22 where the launch takes more
CTAs, each traversal twice in a row on the shared scratch, with and without
parents.  Distances are whole numbers and must be equal; parents must be one
level closer along an edge."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_13577_gb300 as bfs  # noqa: E402


def _graph(kind):
    if kind == "uniform":
        return graphgen.erdos_renyi(18, 64, seed=51)
    off, col = graphgen.kronecker(19, 16, seed=52)
    if kind == "skewed_odd":   # the subgraph on the first 524,287 - 100 vertices
        n = (1 << 19) - 101
        src = np.repeat(np.arange(len(off) - 1), np.diff(off))
        keep = (src < n) & (col < n)
        off = np.zeros(n + 1, dtype=np.int64)
        np.cumsum(np.bincount(src[keep], minlength=n), out=off[1:])
        col = np.ascontiguousarray(col[keep])
    if kind.startswith("cut"):  # the first entries only (directed)
        cut = (1 << 22) + int(kind[3:])
        off, col = np.minimum(off, cut), np.ascontiguousarray(col[:cut])
    return off, col


@pytest.mark.parametrize("kind", ["skewed", "skewed_odd", "uniform", "cut0", "cut1"])
def test_static_large_graphs_match_oracle(kind):
    off, col = _graph(kind)
    n = len(off) - 1
    d_off, d_col = torch.from_numpy(off).cuda(), torch.from_numpy(col).cuda()
    dist = torch.empty(n, dtype=torch.int32, device="cuda")
    parent = torch.empty(n, dtype=torch.int32, device="cuda")
    deepest = 0
    for r in graphgen.pick_roots(off, 2, seed=9):
        ref, _, info = oracle.bfs(off, col, int(r))
        levels = np.bincount(ref[ref >= 0], weights=np.diff(off)[ref >= 0])
        deepest = max(deepest, int(levels.max()))
        for par in (None, parent):
            dist.fill_(-7)
            st = bfs.bfs_run_static(d_off, d_col, int(r), dist, par)
            assert np.array_equal(dist.cpu().numpy(), ref)
            assert (st["levels"], st["edges_scanned"]) == (info["levels"], info["edges_scanned"])
            assert st["reached"] == int((ref >= 0).sum())
        assert oracle.check_bfs(off, col, int(r), ref, parent.cpu().numpy())["ok"]
    if not kind.startswith("cut"):
        assert deepest >= 1 << 23   # a level of at least 8 M entries ran
