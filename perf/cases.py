"""The traversals this library is used for, as cases that can be timed.

A case is a dict of plain values: what runs (``call``), on which graph
(``graph``, ``n`` vertices, ``ef`` generated edges per vertex or the mesh's
``width``), with which options, and in which row type.  ``prepare`` builds
the graph from the seed on the GPU and hands it to the library (an uploaded
graph handle, a server, or the caller's own device CSR, as the call wants);
``run`` makes one pass through the public entry points.

Where a call can return parents they are asked for (``parents``), but only
the distances come back from ``run``: any neighbour one level closer is a
valid parent and which one is written is unspecified, so two runs of the
same build already differ there.
"""
from __future__ import annotations

import torch

import paper_2103_13577_gb300 as bfs

DEV = "cuda"


def listed():
    return [
        # the smallest call: one root of a 4096-vertex graph (a service asking
        # about one neighbourhood), where launch and grid barriers are the cost
        {"name": "root_4k", "call": "root", "graph": "kron", "n": 4096, "ef": 8, "parents": True},
        # a caller with a fixed device-memory plan: CSR checked and traversed
        # with the library's own scratch
        {"name": "static_64k", "call": "static", "graph": "kron", "n": 65536, "ef": 8,
         "parents": True},
        # ordinary graph with an odd vertex count, compact int8 rows
        {"name": "root_200k_int8", "call": "root", "graph": "kron", "n": 200003, "ef": 16,
         "int8": True},
        # the benchmark's headline: scale 22, edge factor 16, distances and parents
        {"name": "root_4m", "call": "root", "graph": "kron", "n": 4194304, "ef": 16,
         "parents": True},
        # the same traversal with direction-optimizing levels allowed
        {"name": "root_4m_direction", "call": "root", "graph": "kron", "n": 4194304, "ef": 16,
         "parents": True, "direction": 1},
        # no hubs: uniform random graph of mean degree 32
        {"name": "root_uniform_1m", "call": "root", "graph": "uniform", "n": 1000003, "ef": 16,
         "parents": True},
        # high diameter, degree 4 (road- and mesh-like): hundreds of small levels
        {"name": "root_mesh", "call": "root", "graph": "mesh", "n": 250500, "width": 500},
        # 64 roots in one launch (all-pairs samples, landmark distances): the
        # benchmark's batched workload
        {"name": "batch64_4m", "call": "batch", "graph": "kron", "n": 4194304, "ef": 16, "k": 64},
        # a partly filled batch on an odd vertex count, int8 rows
        {"name": "batch17_200k_int8", "call": "batch", "graph": "kron", "n": 200003, "ef": 16,
         "k": 17, "int8": True},
        # batched with direction-optimizing levels allowed
        {"name": "batch64_1m_direction", "call": "batch", "graph": "kron", "n": 1048576,
         "ef": 16, "k": 64, "int8": True, "direction": 1},
        # shortest-path counts over the edges of some weights (betweenness,
        # filtered reach), scratch from the context's arena
        {"name": "paths_1m_weights", "call": "paths", "graph": "kron", "n": 1048576, "ef": 16,
         "weights": True},
        # a burst of queries on two resident graphs through the server, int8
        # rows into pinned host memory
        {"name": "serve_burst", "call": "serve", "graph": "kron", "n": 262144, "ef": 16,
         "k": 96, "int8": True},
    ]


def _log_int(rng, lo, hi):
    """Log-uniform in [lo, hi], about one in four a power of two."""
    x = int(round(lo * (hi / lo) ** rng.random()))
    if rng.random() < 0.25:
        x = 1 << max(x.bit_length() - 1, lo.bit_length() - 1)
    return max(lo, min(hi, x))


def draw(rng):
    call = rng.choice(["root", "root", "root", "batch", "batch", "static", "paths", "serve"])
    graph = rng.choice(["kron", "kron", "kron", "uniform", "mesh"])
    if call in ("paths", "serve") or (call == "batch" and graph == "mesh"):
        graph = "kron"
    ef = rng.choice([8, 16])
    case = {"call": call, "graph": graph}
    if graph == "mesh":
        case["width"] = rng.randint(40, 500)
        case["n"] = case["width"] * rng.randint(40, 500)
    else:
        top = {"root": 4 << 20, "batch": 2 << 20, "static": 1 << 19, "paths": 2 << 20,
               "serve": 400000}[call]
        case["n"] = _log_int(rng, 4096, top)
        case["ef"] = ef
    if call in ("root", "static"):
        case["parents"] = rng.random() < 0.5
    if call == "root" and graph != "mesh":
        case["int8"] = not case["parents"] and rng.random() < 0.5
        case["direction"] = rng.choice([0, 0, 1])
    if call in ("batch", "serve"):
        case["k"] = rng.choice([64, rng.randint(2, 64)])
        case["int8"] = rng.random() < 0.5
    if call == "batch":
        case["direction"] = rng.choice([0, 0, 1])
    if call == "paths":
        case["weights"] = rng.random() < 0.5
    return case


# ------------------------------------------------------------------ inputs

def _csr(src, dst, n):
    """Undirected CSR (int64 offsets, int32 columns) of the pairs: both
    directions, no self-loops, no duplicates, rows sorted."""
    keep = src != dst
    src, dst = src[keep], dst[keep]
    keys = torch.cat([src * n + dst, dst * n + src])
    del src, dst, keep
    keys = torch.sort(keys).values
    first = torch.ones(keys.numel(), dtype=torch.bool, device=DEV)
    torch.ne(keys[1:], keys[:-1], out=first[1:])
    keys = keys[first]
    rows = torch.div(keys, n, rounding_mode="floor")
    col = (keys - rows * n).to(torch.int32)
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(rows, minlength=n), 0, out=off[1:])
    return off, col


def _kron(n, ef, gen):
    """R-MAT with initiator 0.57/0.19/0.19/0.05 and a random vertex
    permutation; for n below a power of two, the induced subgraph of as many
    more edges as leaves about ef * n inside."""
    scale = (n - 1).bit_length()
    m = int(ef * n * ((1 << scale) / n) ** 2)
    src = torch.zeros(m, dtype=torch.int64, device=DEV)
    dst = torch.zeros(m, dtype=torch.int64, device=DEV)
    for _ in range(scale):
        down = torch.rand(m, generator=gen, device=DEV) > 0.76
        right = torch.rand(m, generator=gen, device=DEV) > torch.where(down, 0.19 / 0.24,
                                                                       0.57 / 0.76)
        src = src * 2 + down
        dst = dst * 2 + right
    perm = torch.randperm(1 << scale, generator=gen, device=DEV)
    src, dst = perm[src], perm[dst]
    if n != 1 << scale:
        inside = (src < n) & (dst < n)
        src, dst = src[inside], dst[inside]
    return _csr(src, dst, n)


def _uniform(n, ef, gen):
    src = torch.randint(0, n, (ef * n,), generator=gen, device=DEV)
    dst = torch.randint(0, n, (ef * n,), generator=gen, device=DEV)
    return _csr(src, dst, n)


def _mesh(n, width):
    """Grid of n / width rows, each vertex joined to its four neighbours."""
    v = torch.arange(n, dtype=torch.int64, device=DEV)
    right = v[v % width != width - 1]
    down = v[:n - width]
    return _csr(torch.cat([right, down]), torch.cat([right + 1, down + width]), n)


def _graph(case, gen):
    if case["graph"] == "kron":
        return _kron(case["n"], case["ef"], gen)
    if case["graph"] == "uniform":
        return _uniform(case["n"], case["ef"], gen)
    return _mesh(case["n"], case["width"])


def _roots(off, k, gen):
    """k roots, uniform among the vertices that have a neighbour."""
    some = torch.nonzero(off[1:] > off[:-1]).flatten()
    pick = torch.randint(0, some.numel(), (k,), generator=gen, device=DEV)
    return some[pick].to(torch.int32).cpu().numpy()


class _State:
    """What a program holds between calls; gives the library's handles back
    when it goes."""

    def __init__(self, **kw):
        self.ctx = self.server = None
        self.graphs = []
        self.__dict__.update(kw)

    def __del__(self):
        try:
            if self.server is not None:
                self.server.close()
            for g in self.graphs:
                g.close()
            if self.ctx is not None:
                self.ctx.close()
        except Exception:  # interpreter shutdown
            pass


def _weights(nnz, gen):
    return torch.randint(0, 8, (nnz,), generator=gen, device=DEV, dtype=torch.int32)


def _inputs(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    off, col = _graph(case, gen)
    return off, col, gen


def prepare(case, seed):
    off, col, gen = _inputs(case, seed)
    n, call = case["n"], case["call"]
    k = case.get("k", 1)
    roots = _roots(off, k, gen)
    rows = torch.int8 if case.get("int8") else torch.int32
    if call == "static":
        return _State(call=call, off=off, col=col, root=int(roots[0]),
                      dist=torch.empty(n, dtype=torch.int32, device=DEV),
                      parent=torch.empty(n, dtype=torch.int32, device=DEV)
                      if case.get("parents") else None)
    if call == "paths":
        # scratch is about 40 bytes per vertex plus the tile tables
        arena = torch.empty(64 * n + col.numel() // 16 + (16 << 20), dtype=torch.uint8,
                            device=DEV)
        return _State(call=call, arena=arena, ctx=bfs.Context(0, arena=arena), off=off, col=col,
                      root=int(roots[0]), hops=torch.empty(n, dtype=torch.int32, device=DEV),
                      sigma=torch.empty(n, dtype=torch.float64, device=DEV),
                      weights=_weights(col.numel(), gen) if case.get("weights") else None)
    ctx = bfs.Context(0)
    if call == "serve":
        small = _inputs(dict(case, n=n // 4), seed + 1)
        graphs = [bfs.Graph(ctx, off, col), bfs.Graph(ctx, small[0], small[1])]
        server = bfs.Server(ctx, 4 << 30, num_streams=4)
        ids = [server.add_graph(g) for g in graphs]
        # every third query goes to the smaller graph
        more = _roots(small[0], k, small[2])
        queries = [(ids[1], int(more[i])) if i % 3 == 2 else (ids[0], int(roots[i]))
                   for i in range(k)]
        sizes = [n // 4 if i % 3 == 2 else n for i in range(k)]
        host = torch.empty(sum(sizes), dtype=rows, pin_memory=True)
        return _State(call=call, ctx=ctx, graphs=graphs, server=server, queries=queries,
                      host=host, rows=[r.numpy() for r in torch.split(host, sizes)])
    graph = bfs.Graph(ctx, off, col)
    if case.get("direction"):
        graph.set_option(bfs.BFS_OPT_DIRECTION, case["direction"])
    state = _State(call=call, ctx=ctx, graphs=[graph], parent=None)
    if call == "batch":
        state.roots = roots
        state.dist = torch.empty((k, n), dtype=rows, device=DEV)
    else:
        state.root = int(roots[0])
        state.dist = torch.empty(n, dtype=rows, device=DEV)
        if case.get("parents"):
            state.parent = torch.empty(n, dtype=torch.int32, device=DEV)
    return state


def run(state):
    if state.call == "root":
        state.graphs[0].run(state.root, state.dist, state.parent)
        return state.dist
    if state.call == "batch":
        state.graphs[0].run_batch(state.roots, state.dist)
        return state.dist
    if state.call == "static":
        bfs.bfs_run_static(state.off, state.col, state.root, state.dist, state.parent, wait=False)
        return state.dist
    if state.call == "paths":
        state.ctx.run_paths(state.off, state.col, state.root, state.hops, state.sigma,
                            weight=state.weights, lo=0, hi=3)
        return {"hops": state.hops, "sigma": state.sigma}
    tickets = [state.server.submit(g, r, row) for (g, r), row in zip(state.queries, state.rows)]
    for t in tickets:
        state.server.wait(t)
        state.server.release(t)
    return state.host


def work(case):
    """Bytes of one pass: the CSR read once and the rows written once (a
    burst on the server: each of its two graphs read once)."""
    n, k = case["n"], case.get("k", 1)
    nnz = 4 * n if case["graph"] == "mesh" else 2 * case["ef"] * n * 0.95
    graph = 8 * (n + 1) + 4 * nnz
    if case["call"] == "paths":
        return {"bytes": graph + (4 * nnz if case.get("weights") else 0) + 12 * n, "flops": 0}
    if case["call"] == "serve":
        row = (1 if case.get("int8") else 4) * n
        return {"bytes": 1.25 * graph + row * (k - k // 3 + k // 3 / 4), "flops": 0}
    row = (1 if case.get("int8") else 4) * n + (4 * n if case.get("parents") else 0)
    return {"bytes": graph + k * row, "flops": 0}


def exact(case, seed):
    """Shortest-path counts in 64 bits, level by level over the edge list;
    the other calls return whole numbers only."""
    if case["call"] != "paths":
        return None
    off, col, gen = _inputs(case, seed)
    root = int(_roots(off, 1, gen)[0])
    n = case["n"]
    src = torch.repeat_interleave(torch.arange(n, device=DEV), off[1:] - off[:-1])
    dst = col.long()
    if case.get("weights"):
        keep = _weights(col.numel(), gen) <= 3
        src, dst = src[keep], dst[keep]
    hops = torch.full((n,), -1, dtype=torch.int32, device=DEV)
    sigma = torch.zeros(n, dtype=torch.float64, device=DEV)
    hops[root], sigma[root] = 0, 1.0
    level = 0
    while True:
        step = (hops[src] == level) & (hops[dst] < 0)
        if not bool(step.any()):
            return {"hops": hops, "sigma": sigma}
        u, v = src[step], dst[step]
        sigma.index_add_(0, v, sigma[u])
        level += 1
        hops[v] = level
