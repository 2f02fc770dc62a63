"""Benchmark: plain single-source BFS GTEPS on a Kronecker graph.

Workload: undirected Kronecker graph, scale 22, edge factor 16 (initiator
0.57/0.19/0.19/0.05, seeded permutation, no self-loops or duplicates,
int64 offsets + int32 columns), 64 seeded roots of degree >= 1 run one
after another.  One step = the 64 single-source traversals (init, level
loop with degree-binned expansion, visited test-and-set, dist/parent
writes and frontier compaction -- the whole per-GPU level step).

Metric: GTEPS per root = m_c / t (m_c = adjacency entries scanned from
that root, t = that root's traversal time on the device), aggregated by
the harmonic mean over the 64 roots.  Under torchrun each rank traverses
its own 64 roots on its own copy of the graph (weak scaling, no
collective); root i's job throughput is the sum over ranks of m_c divided
by the slowest rank's time for root i.

Also reported: e2e (the same metric through bfs_run with host output
buffers, result copies inside the timed region), the roofline of the
traversal kernel against the measured HBM bandwidth, the CPU oracle on a
bounded sample of roots, a 64-root batched launch on the same graph, and
SM clocks sampled during the timed region.

--impl reference times the CPU oracle (serial FIFO BFS) on the host cores
for the same metric: each step traverses a bounded sample of the roots.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

SCALE, EDGE_FACTOR, GRAPH_SEED, ROOT_SEED, NROOTS = 22, 16, 22, 3, 64
METRIC = "BFS GTEPS (hmean over 64 roots) plain vs 64-root batched; query p50/p99 latency"
WORKLOAD = "kronecker_s22_ef16_plain_64roots"
CSRC = os.path.join(ROOT, "paper_2103_13577_gb300", "csrc")
KERNEL_SRC = os.path.join(CSRC, "bfs_single.cu")
# the single-source and the batched kernel and what both are built from: a
# traffic record of either holds while none of them changes
TRAVERSAL_SRCS = [KERNEL_SRC] + [os.path.join(CSRC, f) for f in
                                 ("bfs_kernels.cu", "bfs_device.cuh", "bfs_internal.h")]
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "bfs_single_persistent_kron_s22_traffic.json")
BATCH_TRAFFIC_FILE = os.path.join(ROOT, "profiles", "bfs_batch_persistent_kron_s22_traffic.json")
PATHS_SRC = os.path.join(CSRC, "bfs_paths.cu")
PATHS_TRAFFIC_FILE = os.path.join(ROOT, "profiles", "paths_persistent_kron_s22_traffic.json")


NOMINAL = ("nominal work: every column entry of the expanded rows once, also those the kernel "
           "skips because they lead to visited vertices; traffic is what it moves (ncu)")


def env_int(name, default):
    try:
        return int(os.environ.get(name, default))
    except ValueError:
        return default


def trimmed_mean(x, cut):
    x = np.sort(np.asarray(x, dtype=np.float64))
    k = int(len(x) * cut)
    return float(x[k:len(x) - k].mean()) if len(x) > 2 * k else float(x.mean())


def hmean(x):
    x = np.asarray(x, dtype=np.float64)
    return float(len(x) / np.sum(1.0 / x))


def measured_hbm_peak():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            return float(json.load(f)["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def kernel_hash(src=KERNEL_SRC):
    h = hashlib.sha256()
    for path in TRAVERSAL_SRCS if src in TRAVERSAL_SRCS else [src]:
        with open(path, "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def recorded_traffic(path=TRAFFIC_FILE, src=KERNEL_SRC):
    """DRAM bytes per launch from the committed ncu capture, or None when the
    kernel source changed since the capture."""
    try:
        with open(path) as f:
            rec = json.load(f)
        if rec.get("kernel_sha256_16") != kernel_hash(src):
            return None
        return float(rec["dram_bytes_per_launch"])
    except Exception:
        return None


class ClockSampler:
    """nvidia-smi samples (200 ms) of SM clocks and throttle reasons."""
    FIELDS = ("clocks.sm,clocks.max.sm,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if not self.proc:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in self.lines:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 7:
                continue
            try:
                sm.append(float(parts[0]))
                smax.append(float(parts[1]))
            except ValueError:
                continue
            for nm, val in zip(names, parts[3:7]):
                if val.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def workload_config(n, m, world):
    """The `config` of the JSON line: the workload only, identical for both
    arms."""
    return {"workload": WORKLOAD,
            "graph": f"kronecker scale {SCALE} edge factor {EDGE_FACTOR} "
                     "A/B/C=0.57/0.19/0.19, permuted, symmetric, deduplicated",
            "vertices": int(n), "directed_entries": int(m), "roots": NROOTS,
            "root_seed": ROOT_SEED, "graph_seed": GRAPH_SEED,
            "l2": "inputs larger than L2 (column array %.0f MB > 129 MB)" % (m * 4 / 1e6),
            "parallelism": f"replicas x{world}"}


def make_workload(rank):
    import graphgen
    off, col, _ = workload_graph("kronecker", SCALE, EDGE_FACTOR, GRAPH_SEED)
    roots = graphgen.pick_roots(off, NROOTS, seed=ROOT_SEED + 7919 * rank)
    return off, col, roots


# ------------------------------------------- batched roofline numerator
def batch_frontier_sums(rows, deg):
    """Frontiers of a top-down 64-root batched traversal, recovered from its
    distance rows: for every level L, |A_L| = the vertices some lane reaches
    at level L (one queue entry each, carrying its lane set) and D_L = the
    sum of their degrees (the column entries level L expands); plus R = the
    vertices any lane reaches.  rows: [k][N] distances (-1 unreached, int32
    or int8), deg: [N] out-degrees; torch tensors on one device."""
    sizes, degs = [], []
    top = int(rows.max().item())
    for level in range(top + 1):
        a = (rows == level).any(0)
        sizes.append(int(a.sum().item()))
        degs.append(int(deg[a].sum().item()))
    reached = int((rows >= 0).any(0).sum().item())
    return sizes, degs, reached


def batch_algorithmic_bytes(sizes, degs, reached: int, n: int, k: int, elem: int) -> float:
    """Nominal bytes of one top-down batched launch (bfs_batch_persistent),
    each item once:
      init      16 N                 visited/next lane-set pairs cleared
      level L   4 D_L                column entries of the frontier's rows
                + 28 |A_L|           two row offsets, queue entry (vertex + lane set)
                + 16 N               sweep reads every vertex's lane-set pair
                + 92 |A_L|           producing A_L: pair write-back, 64-byte
                                     level row, queue entry
      emit      12 N + 64 R          visited set and renumbering of every vertex,
                                     level rows of the reached ones
                + k N elem           the k distance rows
    Lane-set updates of the neighbours (atomicOr on next) and the level-row
    re-reads of vertices reached before are cache traffic, not counted.  A
    measure of the work, the same for every kernel, and not of what this one
    moves: rows skip the entries that lead to vertices every lane has, and
    levels below 16 touch 32 of a level row's 64 bytes."""
    per_level = sum(4 * d + 120 * a + 16 * n for a, d in zip(sizes, degs))
    return float(per_level + 16 * n + 12 * n + 64 * reached + k * n * elem)


# ---------------------------------------------------------------- oracle
def paths_measure(bfs, torch, dev_, stream, off, col, roots, n):
    """bfs_run_paths (shortest-path counts) on the caller's CSR resident on
    the device, every entry kept and with a weight filter keeping weights
    0-3 of uniform 0-7 (about half the entries); device time per root from
    CUDA events on the stream, scratch carved from an arena context.
    Algorithmic bytes per traversal: 4 m_c columns (+ 4 m_c weights when
    filtered) + 60 n_c (row offsets 16, frontier queue entry written and
    read 24, sigma read as a frontier vertex 8 and written once 8, hops 4)
    + 12 N (hops and sigma initialised); the visited-bitmap probes, the
    next-frontier marks, the sigma additions and the per-level bitmap scans
    (N / 8 bytes) are cache traffic, not counted."""
    peak, _ = measured_hbm_peak()
    arena = torch.empty(int(64 * n + (64 << 20)), dtype=torch.uint8, device=dev_)
    pctx = bfs.Context(dev_.index, arena=arena)
    d_off = torch.from_numpy(np.ascontiguousarray(off, dtype=np.int64)).to(dev_)
    d_col = torch.from_numpy(np.ascontiguousarray(col, dtype=np.int32)).to(dev_)
    wts = np.random.default_rng(5).integers(0, 8, len(col)).astype(np.int32)
    d_w = torch.from_numpy(wts).to(dev_)
    hops = torch.empty(n, dtype=torch.int32, device=dev_)
    sigma = torch.empty(n, dtype=torch.float64, device=dev_)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    out = {"roots": len(roots), "note": "hops + shortest-path counts (Brandes forward phase), "
           "top-down only; GTEPS = entries of the reached rows / time"}
    for name, w, lo, hi in (("all_entries", None, 0, 0), ("weights_0_3_of_0_7", d_w, 0, 3)):
        pctx.run_paths(d_off, d_col, int(roots[0]), hops, sigma, w, lo, hi, stream=stream)
        ms, edges, nbytes = [], [], []
        for r in roots:
            ev[0].record(stream)
            st = pctx.run_paths(d_off, d_col, int(r), hops, sigma, w, lo, hi, stream=stream)
            ev[1].record(stream)
            torch.cuda.synchronize(dev_)
            ms.append(ev[0].elapsed_time(ev[1]))
            edges.append(st["edges_scanned"])
            nbytes.append((8 if w is not None else 4) * st["edges_scanned"] + 60 * st["reached"]
                          + 12 * n)
        ms, edges, nbytes = np.array(ms), np.array(edges, dtype=np.float64), np.array(nbytes, dtype=np.float64)
        gbs = float(np.mean(nbytes / (ms * 1e-3)) / 1e9)
        out[name] = {"gteps": hmean(edges / (ms * 1e-3) / 1e9), "root_ms_median": float(np.median(ms)),
                     "levels_last_root": int(st["levels"]),
                     "roofline": {"bound": "hbm", "achieved": gbs, "peak": peak, "unit": "GB/s",
                                  "frac": gbs / peak,
                                  "traffic": recorded_traffic(PATHS_TRAFFIC_FILE, PATHS_SRC)
                                  if name == "all_entries" else None,
                                  "kernel": "paths_persistent",
                                  "algorithmic_bytes_per_traversal": float(nbytes.mean())}}
    pctx.close()
    del arena, d_off, d_col, d_w, hops, sigma
    return out


def run_oracle_sample(off, col, roots, budget_s):
    """Serial oracle over as many roots as fit in budget_s (at least one)."""
    import oracle
    gteps, used = [], []
    t_start = time.perf_counter()
    for r in roots:
        t0 = time.perf_counter()
        _, _, info = oracle.bfs(off, col, int(r))
        dt = time.perf_counter() - t0
        gteps.append(info["edges_scanned"] / dt / 1e9)
        used.append(int(r))
        if time.perf_counter() - t_start > budget_s:
            break
    return gteps, used


def run_oracle_parallel(off, col, roots, budget_s):
    """The serial oracle on distinct roots, one per host core at a time (the
    oracle is C called through ctypes, which releases the GIL): whole-run
    throughput in GTEPS, the roots used and the thread count."""
    from concurrent.futures import ThreadPoolExecutor

    import oracle
    cores = max(1, os.cpu_count() or 1)
    done_m, used = 0, []
    t0 = time.perf_counter()
    with ThreadPoolExecutor(max_workers=cores) as ex:
        i = 0
        while i < len(roots):
            batch = [int(r) for r in roots[i:i + cores]]
            for _, _, info in ex.map(lambda r: oracle.bfs(off, col, r), batch):
                done_m += info["edges_scanned"]
            used += batch
            i += cores
            if time.perf_counter() - t0 > budget_s:
                break
    dt = time.perf_counter() - t0
    return done_m / dt / 1e9, used, cores


def reference_arm(args, rank, world):
    if rank != 0:
        return
    off, col, roots = make_workload(0)
    per_step = max(1, env_int("BFS_REF_ROOTS_PER_STEP", 2))
    i = 0
    for _ in range(args.warmup):
        run_oracle_sample(off, col, roots[i:i + 1], 0)
        i = (i + 1) % len(roots)
    gteps, step_ms = [], []
    for _ in range(args.steps):
        sel = [roots[(i + j) % len(roots)] for j in range(per_step)]
        i = (i + per_step) % len(roots)
        t0 = time.perf_counter()
        g, _ = run_oracle_sample(off, col, sel, 1e9)
        step_ms.append((time.perf_counter() - t0) * 1e3)
        gteps.extend(g)
    value = hmean(gteps)
    sample = f"{per_step} of the 64 roots per step, serial FIFO BFS on one host core"
    line = {
        "metric": METRIC, "value": value, "unit": "GTEPS", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": float(np.mean(step_ms)), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "int32", "data": "synthetic",
        "impl": "reference",
        "config": workload_config(len(off) - 1, len(col), world),
        "cpu_baseline": {"value": value, "unit": "GTEPS", "cores": 1, "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": value, "unit": "GTEPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


# ------------------------------------------------------------------ GPU arm
def aggregate_ranks(t_root, m_c, step_ms, world, device):
    """Whole-job numbers over ranks: root slot i takes the slowest rank's
    time and the sum of the ranks' m_c; the step time is the slowest rank's.
    Returns (per-root times, per-root edges, ms per step, hmean GTEPS)."""
    import torch
    import torch.distributed as dist_mod
    if world > 1:
        t_all = torch.tensor(t_root, dtype=torch.float64, device=device)
        dist_mod.all_reduce(t_all, op=dist_mod.ReduceOp.MAX)
        m_all = torch.tensor(np.asarray(m_c, dtype=np.float64), dtype=torch.float64, device=device)
        dist_mod.all_reduce(m_all, op=dist_mod.ReduceOp.SUM)
        s_all = torch.tensor([float(np.mean(step_ms))], dtype=torch.float64, device=device)
        dist_mod.all_reduce(s_all, op=dist_mod.ReduceOp.MAX)
        t_job, m_job, ms_step = t_all.cpu().numpy(), m_all.cpu().numpy(), float(s_all.item())
    else:
        t_job = np.asarray(t_root, dtype=np.float64)
        m_job = np.asarray(m_c, dtype=np.float64)
        ms_step = float(np.mean(step_ms))
    return t_job, m_job, ms_step, hmean(m_job / (t_job * 1e-3) / 1e9)


def gpu_arm(args, rank, world, local_rank):
    import torch
    import torch.distributed as dist_mod

    import paper_2103_13577_gb300 as bfs

    torch.cuda.set_device(local_rank)
    dev_ = torch.device("cuda", local_rank)
    off, col, roots = make_workload(rank)
    n = len(off) - 1
    ctx = bfs.Context(local_rank)
    g = bfs.Graph(ctx, off, col)
    if args.bins:
        g.set_bins(*[int(x) for x in args.bins.split(",")])
    if args.ctas_per_sm:
        g.set_option(bfs.BFS_OPT_CTAS_PER_SM, args.ctas_per_sm)
    stream = torch.cuda.current_stream(dev_)
    dist = torch.empty(n, dtype=torch.int32, device=dev_)
    parent = torch.empty(n, dtype=torch.int32, device=dev_)

    def barrier():
        if world > 1:
            dist_mod.barrier()

    # per-root m_c and n_c from the device's own counters (untimed pass)
    m_c = np.zeros(NROOTS, dtype=np.int64)
    n_c = np.zeros(NROOTS, dtype=np.int64)
    for i, r in enumerate(roots):
        g.run(int(r), dist, parent, stream=stream)
        st = g.sync(stream)
        m_c[i], n_c[i] = st["edges_scanned"], st["reached"]

    ev = [[torch.cuda.Event(enable_timing=True) for _ in range(NROOTS + 1)] for _ in range(args.steps)]
    for _ in range(args.warmup):
        for r in roots:
            g.run(int(r), dist, parent, stream=stream)
    torch.cuda.synchronize(dev_)
    barrier()
    torch.cuda.synchronize(dev_)
    clocks = ClockSampler(local_rank)
    clocks.start()
    time.sleep(0.25)
    for s in range(args.steps):
        ev[s][0].record(stream)
        for i, r in enumerate(roots):
            g.run(int(r), dist, parent, stream=stream)
            ev[s][i + 1].record(stream)
    torch.cuda.synchronize(dev_)
    barrier()
    torch.cuda.synchronize(dev_)
    clk = clocks.stop()
    root_ms = np.array([[ev[s][i].elapsed_time(ev[s][i + 1]) for i in range(NROOTS)]
                        for s in range(args.steps)])
    step_ms = np.array([ev[s][0].elapsed_time(ev[s][NROOTS]) for s in range(args.steps)])
    st = g.sync(stream)
    assert st["status"] == 0

    t_root = root_ms.mean(axis=0)
    t_job, m_job, ms_step, value = aggregate_ranks(t_root, m_c, step_ms, world, dev_)

    # e2e: the public call with host outputs (copies inside the timed region)
    h_dist = torch.empty(n, dtype=torch.int32, pin_memory=True).numpy()
    h_par = torch.empty(n, dtype=torch.int32, pin_memory=True).numpy()
    for r in roots[:3]:
        g.run(int(r), h_dist, h_par)
    barrier()
    e2e_ms = np.zeros(NROOTS)
    e2e_steps = args.steps
    for _ in range(e2e_steps):
        for i, r in enumerate(roots):
            t0 = time.perf_counter()
            g.run(int(r), h_dist, h_par)
            e2e_ms[i] += (time.perf_counter() - t0) * 1e3
    e2e_ms /= e2e_steps
    if world > 1:
        t_e = torch.tensor(e2e_ms, dtype=torch.float64, device=dev_)
        dist_mod.all_reduce(t_e, op=dist_mod.ReduceOp.MAX)
        e2e_ms = t_e.cpu().numpy()
    e2e_value = hmean(m_job / (e2e_ms * 1e-3) / 1e9)

    # direction-optimizing mode on the same roots (bottom-up levels touch fewer
    # edges; GTEPS still counts m_c, the top-down work, and is flagged so)
    g.set_option(bfs.BFS_OPT_DIRECTION, 1)
    for r in roots[:3]:
        g.run(int(r), dist, parent, stream=stream)
    do_ev = [torch.cuda.Event(enable_timing=True) for _ in range(NROOTS + 1)]
    do_reps = max(1, min(args.steps, 3))
    do_ms = np.zeros(NROOTS)
    for _ in range(do_reps):
        do_ev[0].record(stream)
        for i, r in enumerate(roots):
            g.run(int(r), dist, parent, stream=stream)
            do_ev[i + 1].record(stream)
        torch.cuda.synchronize(dev_)
        do_ms += np.array([do_ev[i].elapsed_time(do_ev[i + 1]) for i in range(NROOTS)])
    do_ms /= do_reps
    do_st = g.sync(stream)
    g.set_option(bfs.BFS_OPT_DIRECTION, 0)
    if world > 1:
        t_d = torch.tensor(do_ms, dtype=torch.float64, device=dev_)
        dist_mod.all_reduce(t_d, op=dist_mod.ReduceOp.MAX)
        do_ms = t_d.cpu().numpy()
    do_value = hmean(m_job / (do_ms * 1e-3) / 1e9)

    # the paper's own scheme (per-level LRB binning, one kernel per bin on its
    # own stream, host-driven levels) on the same roots, for comparison
    lrb_ms = np.zeros(NROOTS)
    for r in roots[:2]:
        g.run_lrb(int(r), dist, stream=stream)
    lev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    for i, r in enumerate(roots):
        lev[0].record(stream)
        g.run_lrb(int(r), dist, stream=stream)
        lev[1].record(stream)
        torch.cuda.synchronize(dev_)
        lrb_ms[i] = lev[0].elapsed_time(lev[1])
    lrb_value = hmean(m_c / (lrb_ms * 1e-3) / 1e9)

    # shortest-path counts and weight-filtered traversal (bfs_run_paths)
    paths = paths_measure(bfs, torch, dev_, stream, off, col, roots[:8], n)

    # 64-root batched launch on the same graph (one persistent launch)
    bd = torch.empty((NROOTS, n), dtype=torch.int32, device=dev_)
    for _ in range(2):
        g.run_batch(roots, bd, stream=stream)
    bst = g.batch_sync(stream)
    bev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    reps = 3
    bev[0].record(stream)
    for _ in range(reps):
        g.run_batch(roots, bd, stream=stream)
    bev[1].record(stream)
    bst = g.batch_sync(stream)
    batch_ms = bev[0].elapsed_time(bev[1]) / reps
    batch_gteps = bst["edges_scanned"] / (batch_ms * 1e-3) / 1e9
    # algorithmic bytes of the batched launch from its frontiers (the rows)
    deg_dev = torch.from_numpy(np.diff(off)).to(dev_)
    b_sizes, b_degs, b_reached = batch_frontier_sums(bd, deg_dev)
    b_bytes = batch_algorithmic_bytes(b_sizes, b_degs, b_reached, n, NROOTS, 4)
    del deg_dev
    g.set_option(bfs.BFS_OPT_DIRECTION, 1)
    g.run_batch(roots, bd, stream=stream)
    g.batch_sync(stream)
    bev[0].record(stream)
    for _ in range(reps):
        g.run_batch(roots, bd, stream=stream)
    bev[1].record(stream)
    bdo = g.batch_sync(stream)
    g.set_option(bfs.BFS_OPT_DIRECTION, 0)
    batch_do_ms = bev[0].elapsed_time(bev[1]) / reps

    # roofline of the traversal kernel (one launch per root), on nominal work
    peak, peak_kind = measured_hbm_peak()
    b_achieved = b_bytes / (batch_ms * 1e-3) / 1e9
    alg_bytes = 4.0 * m_c + 32.0 * n_c + 8.125 * n
    achieved = float(np.mean(alg_bytes / (t_root * 1e-3)) / 1e9)
    traffic = recorded_traffic()

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        gts, used = run_oracle_sample(off, col, roots, args.cpu_budget)
        cpu = {"value": hmean(gts), "unit": "GTEPS", "cores": 1, "kind": "oracle",
               "sample": f"{len(used)} of the 64 roots, serial FIFO BFS on one host core"}
        par, pused, pcores = run_oracle_parallel(off, col, roots, args.cpu_budget)
        cpu["all_cores"] = {"value": par, "unit": "GTEPS", "cores": pcores,
                            "sample": f"{len(pused)} of the 64 roots, one serial BFS per core "
                                      "at a time; sum of m_c over wall time"}

    if rank == 0:
        info = g.info()
        line = {
            "metric": METRIC, "value": value, "unit": "GTEPS", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_step,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int32",
            "data": "synthetic",
            "config": workload_config(n, len(col), world),
            "graph_setup": {"bins": [info["t_small"], info["t_large"], info["chunk_warp"],
                                     info["chunk_cta"]],
                            "relabelled": bool(info["relabelled"])},
            "aggregate_gteps": float(m_job.sum() / (t_job.sum() * 1e-3) / 1e9),
            "conventions": {
                "trimmed_mean_gteps": trimmed_mean(m_job / (t_job * 1e-3) / 1e9, 0.1),
                "paper_m_over_t_hmean": hmean(world * len(col) / (t_job * 1e-3) / 1e9),
                "graph500_half_m_c_hmean": value / 2.0,
                "note": "trimmed mean drops the fastest and slowest 10 % of roots; paper "
                        "convention divides the graph's directed entries M by t; Graph500 "
                        "counts undirected edges, m_c / 2"},
            "root_ms_median": float(np.median(t_job)),
            "e2e": {"value": e2e_value, "unit": "GTEPS", "h2d_bytes_per_step": 4 * NROOTS,
                    "d2h_bytes_per_step": 2 * 4 * n * NROOTS},
            "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                         "frac": achieved / peak, "traffic": traffic,
                         "kernel": "bfs_single_persistent", "bytes": NOMINAL,
                         "peak_source": f"{peak_kind} (MEASURED_PEAKS.json hbm_gbs)"
                         if peak_kind == "measured" else "fallback 6.8 TB/s",
                         "algorithmic_bytes_per_launch": float(alg_bytes.mean())},
            "cpu_baseline": cpu,
            "direction_optimizing": {
                "value": do_value, "unit": "GTEPS", "root_ms_median": float(np.median(do_ms)),
                "bottom_up_levels_last_root": int(do_st["bottom_up_levels"]),
                "note": "BFS_OPT_DIRECTION=1; GTEPS counts m_c (the top-down edge work), "
                        "bottom-up levels examine fewer edges"},
            "paper_lrb_scheme": {
                "value": lrb_value, "unit": "GTEPS", "root_ms_median": float(np.median(lrb_ms)),
                "note": "per-level log2-degree binning, one kernel per bin on its own stream, "
                        "host-driven level loop (bfs_run_lrb), same roots, this rank"},
            "shortest_path_counts": paths,
            "batched": {"roots": NROOTS, "ms": batch_ms, "gteps": batch_gteps,
                        "edges": int(bst["edges_scanned"]), "levels": int(bst["levels"]),
                        "speedup_vs_plain_step": ms_step / batch_ms,
                        "roofline": {"bound": "hbm", "achieved": b_achieved, "peak": peak,
                                     "unit": "GB/s", "frac": b_achieved / peak,
                                     "traffic": recorded_traffic(BATCH_TRAFFIC_FILE),
                                     "kernel": "bfs_batch_persistent", "bytes": NOMINAL,
                                     "algorithmic_bytes_per_launch": b_bytes,
                                     "frontier_entries": int(sum(b_sizes)),
                                     "frontier_edges": int(sum(b_degs))},
                        "direction_optimizing": {
                            "ms": batch_do_ms,
                            "gteps": bdo["edges_scanned"] / (batch_do_ms * 1e-3) / 1e9,
                            "bottom_up_levels": int(bdo["bottom_up_levels"])}},
            "clocks": clk,
            "gpu_launches": int(args.steps * NROOTS),
        }
    g.close()
    ctx.close()
    if rank == 0:
        if world == 1 and not args.no_extras:
            # the other workloads, measured after the headline's timed region:
            # 64-root batched at scale 24 and served queries at 1k / 10k q/s
            del dist, parent
            torch.cuda.empty_cache()
            line["batched_s24"] = batched_measure(24)
            line["serving"] = serve_measure([18, 20, 22, 24], [1000, 10000], 0.5, 10000, 32,
                                            int8_rates=(10000,))
        print(json.dumps(line), flush=True)


# ------------------------------------------------- batched configuration
_GRAPHS = {}


def workload_graph(kind, scale, k, seed):
    """A seeded workload graph, generated once per process (the headline,
    batched and serving workloads share graphs)."""
    import graphgen
    key = (kind, scale, k, seed)
    if key not in _GRAPHS:
        t0 = time.time()
        gen = graphgen.kronecker if kind == "kronecker" else graphgen.erdos_renyi
        off, col = gen(scale, k, seed=seed)
        _GRAPHS[key] = (off, col, time.time() - t0)
    return _GRAPHS[key]


def batched_measure(scale):
    """64 roots in one launch vs 64 single-source runs, on a Kronecker graph
    (edge factor 16) and an Erdos-Renyi graph (average degree 32) of 2^scale
    vertices, each autotuned first (single-source on 4 roots, batched on all
    64).  GTEPS = sum of the 64 roots' m_c / time."""
    import torch

    import graphgen
    import paper_2103_13577_gb300 as bfs

    out = {"workload": f"batched_64roots_s{scale}", "unit": "GTEPS", "graphs": []}
    ctx = bfs.Context(0)
    stream = torch.cuda.current_stream()
    for name, spec in (("kronecker", ("kronecker", scale, 16, 24)),
                       ("erdos_renyi", ("erdos_renyi", scale, 32, 25))):
        off, col, gen_s = workload_graph(*spec)
        n = len(off) - 1
        roots = graphgen.pick_roots(off, NROOTS, seed=ROOT_SEED)
        g = bfs.Graph(ctx, off, col)
        dist = torch.empty(n, dtype=torch.int32, device="cuda")
        parent = torch.empty(n, dtype=torch.int32, device="cuda")
        rec = {"graph": name, "vertices": n, "directed_entries": int(len(col)), "gen_s": gen_s,
               "seed": spec[3]}
        tune_plain = g.autotune(roots[:4])
        rec["tuned_plain"] = {k: tune_plain[k] for k in ("t_small", "t_large", "chunk_warp", "chunk_cta", "ctas_per_sm")}

        def time_plain(direction):
            g.set_option(bfs.BFS_OPT_DIRECTION, direction)
            for r in roots[:3]:
                g.run(int(r), dist, parent, stream=stream)
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            ev[0].record(stream)
            for r in roots:
                g.run(int(r), dist, parent, stream=stream)
            ev[1].record(stream)
            torch.cuda.synchronize()
            g.set_option(bfs.BFS_OPT_DIRECTION, 0)
            return ev[0].elapsed_time(ev[1])

        m_c = 0
        for r in roots:
            g.run(int(r), dist, None, stream=stream)
            m_c += g.sync(stream)["edges_scanned"]
        plain_ms = time_plain(0)
        do_ms = time_plain(1)
        tune_b = g.autotune(roots, batched=True)
        rec["tuned_batched"] = {k: tune_b[k] for k in ("t_small", "t_large", "chunk_warp", "chunk_cta", "ctas_per_sm")}
        res = {}
        for dt_name, dt, direction in (("int32", torch.int32, 0), ("int8", torch.int8, 0),
                                       ("int32_direction_optimizing", torch.int32, 1),
                                       ("int8_direction_optimizing", torch.int8, 1)):
            g.set_option(bfs.BFS_OPT_DIRECTION, direction)
            bd = torch.empty((NROOTS, n), dtype=dt, device="cuda")
            g.run_batch(roots, bd, stream=stream)
            bst = g.batch_sync(stream)
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            reps = 3
            ev[0].record(stream)
            for _ in range(reps):
                g.run_batch(roots, bd, stream=stream)
            ev[1].record(stream)
            bst = g.batch_sync(stream)
            ms = ev[0].elapsed_time(ev[1]) / reps
            res[dt_name] = {"ms": ms, "gteps": bst["edges_scanned"] / (ms * 1e-3) / 1e9,
                            "levels": int(bst["levels"]),
                            "bottom_up_levels": int(bst["bottom_up_levels"])}
            g.set_option(bfs.BFS_OPT_DIRECTION, 0)
            del bd
        rec.update({"sum_m_c": int(m_c), "plain_64_runs_ms": plain_ms,
                    "plain_gteps_aggregate": m_c / (plain_ms * 1e-3) / 1e9,
                    "direction_optimizing_64_runs_ms": do_ms,
                    "direction_optimizing_gteps_aggregate": m_c / (do_ms * 1e-3) / 1e9,
                    "batched": res,
                    "batched_speedup_vs_plain": plain_ms / res["int32"]["ms"],
                    "batched_speedup_vs_direction_optimizing": do_ms / res["int32"]["ms"],
                    "batched_direction_optimizing_speedup_vs_plain":
                        plain_ms / res["int32_direction_optimizing"]["ms"]})
        out["graphs"].append(rec)
        g.close()
        del dist, parent
        torch.cuda.empty_cache()
    ctx.close()
    return out


def batched_arm(args):
    out = {"metric": METRIC, "higher_is_better": True, "data": "synthetic", "dtype": "int32"}
    out.update(batched_measure(args.batch_scale))
    print(json.dumps(out), flush=True)


# --------------------------------------------------- serving configuration
def serve_measure(scales, rates, window_s, max_queries, budget_gib, buf_gib=8.0, int8_rates=()):
    """Served single-root queries on resident Kronecker graphs (edge factor
    16, graph seed = scale; the scale-22 and scale-24 graphs are the headline
    and batched workloads' graphs): seeded Poisson arrivals at each offered
    rate, graph uniform, root uniform over a seeded pool of 256 degree >= 1
    vertices per graph; the server packs same-graph queries into batched
    launches on 4 streams within a fixed memory budget.  The trace is
    replayed by bfs_server_replay (one native submitter thread per graph, a
    native collector).  Latency = completion on the server's monotonic clock
    minus the scheduled arrival; the copy of the result row into the
    caller's pinned host buffer is inside it.  Baseline: the same trace run
    one query at a time by bfs_replay_single (bfs_run with a host row, in
    arrival order, from a native thread), measured, not modelled.  Rates in
    int8_rates run again with int8 result rows (a quarter of the bytes to
    copy to the host), the baseline with int8 rows too."""
    import torch

    import graphgen
    import paper_2103_13577_gb300 as bfs

    ctx = bfs.Context(0)
    graphs = []
    for sc in scales:
        off, col, _ = workload_graph("kronecker", sc, 16, sc)
        g = bfs.Graph(ctx, off, col)
        g.set_option(bfs.BFS_OPT_DIRECTION, 1)
        pool_roots = graphgen.pick_roots(off, 256, seed=200 + sc)
        graphs.append({"scale": sc, "n": len(off) - 1, "g": g, "roots": pool_roots})
    srv = bfs.Server(ctx, int(budget_gib) << 30, num_streams=4)
    for gr in graphs:
        gr["gid"] = srv.add_graph(gr["g"])
        nbuf = int(max(8, min(256, int(buf_gib * (1 << 30)) // (gr["n"] * 4))))
        gr["bufs"] = torch.empty((nbuf, gr["n"]), dtype=torch.int32, pin_memory=True).numpy()
        gr["base_bufs"] = gr["bufs"][:2]
        if int8_rates:
            nb8 = int(max(8, min(256, int(buf_gib * (1 << 30)) // gr["n"])))
            gr["bufs8"] = torch.empty((nb8, gr["n"]), dtype=torch.int8, pin_memory=True).numpy()
            gr["base_bufs8"] = gr["bufs8"][:2]
    handles = [gr["g"].handle for gr in graphs]
    results = []
    for rate, rows in [(r, "int32") for r in rates] + [(r, "int8") for r in int8_rates]:
        bkey, basekey = ("bufs8", "base_bufs8") if rows == "int8" else ("bufs", "base_bufs")
        nq = int(min(max_queries, rate * window_s))
        rng = np.random.default_rng(rate)
        gaps = rng.exponential(1.0 / rate, nq)
        which = rng.integers(0, len(graphs), nq)
        ridx = rng.integers(0, 256, nq)
        gid = np.array([graphs[w]["gid"] for w in which], dtype=np.int32)
        rts = np.array([graphs[w]["roots"][j] for w, j in zip(which, ridx)], dtype=np.int32)
        st0 = srv.stats()
        t0 = time.monotonic_ns() + 20_000_000
        arrival = t0 + (np.cumsum(gaps) * 1e9).astype(np.int64)
        done, status, _ = srv.replay(gid, rts, arrival, [gr[bkey] for gr in graphs],
                                     timeout_us=120_000_000)
        st1 = srv.stats()
        errors = int(np.count_nonzero(status != bfs.BFS_OK))
        lat_ms = (done - arrival) / 1e6
        span_s = (done.max() - arrival[0]) / 1e9
        # the same trace, one query at a time
        t0 = time.monotonic_ns() + 20_000_000
        arrival_b = t0 + (np.cumsum(gaps) * 1e9).astype(np.int64)
        done_b, status_b = bfs.bfs_replay_single(handles, which.astype(np.int32), rts, arrival_b,
                                                 [gr[basekey] for gr in graphs])
        lat_b = (done_b - arrival_b) / 1e6
        launches = st1["launches"] - st0["launches"]
        results.append({
            "offered_qps": rate, "rows": rows, "queries": nq, "errors": errors,
            "p50_ms": float(np.percentile(lat_ms, 50)), "p99_ms": float(np.percentile(lat_ms, 99)),
            "sustained_qps": nq / span_s,
            "launches": int(launches),
            "mean_queries_per_launch": (st1["lanes"] - st0["lanes"]) / max(1, launches),
            "one_at_a_time": {
                "p50_ms": float(np.percentile(lat_b, 50)),
                "p99_ms": float(np.percentile(lat_b, 99)),
                "sustained_qps": nq / ((done_b.max() - arrival_b[0]) / 1e9),
                "errors": int(np.count_nonzero(status_b != bfs.BFS_OK))},
        })
    srv.close()
    out = {"workload": "served_queries_kronecker_s" + "_".join(map(str, scales)), "unit": "ms",
           "memory_budget_gib": budget_gib, "streams": 4, "window_s": window_s,
           "host_buffers_per_graph": {f"s{gr['scale']}": int(gr["bufs"].shape[0]) for gr in graphs},
           "rates": results, "server": srv_stats_of(st1),
           "baseline": "the same arrival trace through bfs_replay_single: bfs_run with a pinned "
                       "host row per query, in arrival order (measured)"}
    for gr in graphs:
        gr["g"].close()
    ctx.close()
    return out


def srv_stats_of(st):
    return {k: int(v) for k, v in st.items()}


def serve_arm(args):
    out = {"metric": METRIC, "data": "synthetic"}
    out.update(serve_measure([int(x) for x in args.serve_scales.split(",")],
                             [int(x) for x in args.serve_rates.split(",")], args.serve_window,
                             args.serve_max_queries, args.serve_budget,
                             int8_rates=[int(x) for x in args.serve_rates.split(",")][1:]))
    print(json.dumps(out), flush=True)


# ---------------------------------------------------- largest configuration
def large_arm(args):
    """Kronecker graph of the paper's headline size on one GPU (default
    scale 29, edge factor 8): 64 roots as single-source runs (top-down and
    direction-optimizing) and as one 64-root batched launch with int8
    distances; one root checked against the CPU oracle, and batched lane 0
    against its single-source run."""
    import torch

    import graphgen
    import oracle
    import paper_2103_13577_gb300 as bfs

    rec = {"metric": METRIC, "unit": "GTEPS", "data": "synthetic",
           "workload": f"kronecker_s{args.large_scale}_ef{args.large_ef}_64roots"}
    t0 = time.time()
    off, col = graphgen.kronecker(args.large_scale, args.large_ef, seed=29)
    rec["gen_s"] = time.time() - t0
    n = len(off) - 1
    rec.update({"vertices": n, "directed_entries": int(len(col))})
    roots = graphgen.pick_roots(off, NROOTS, seed=ROOT_SEED)
    ctx = bfs.Context(0)
    t0 = time.time()
    g = bfs.Graph(ctx, off, col)
    torch.cuda.synchronize()
    rec["upload_s"] = time.time() - t0
    info = g.info()
    rec["device_gb"] = info["device_bytes"] / 1e9
    stream = torch.cuda.current_stream()
    dist = torch.empty(n, dtype=torch.int32, device="cuda")
    parent = torch.empty(n, dtype=torch.int32, device="cuda")
    tune = g.autotune(roots[:2])
    rec["tuned"] = {k: tune[k] for k in ("t_small", "t_large", "chunk_warp", "chunk_cta", "ctas_per_sm")}
    m_c = np.zeros(NROOTS)
    n_c = np.zeros(NROOTS)
    for i, r in enumerate(roots):
        g.run(int(r), dist, None, stream=stream)
        st = g.sync(stream)
        m_c[i], n_c[i] = st["edges_scanned"], st["reached"]
    for direction, key in ((0, "plain"), (1, "direction_optimizing")):
        g.set_option(bfs.BFS_OPT_DIRECTION, direction)
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(NROOTS + 1)]
        ev[0].record(stream)
        for i, r in enumerate(roots):
            g.run(int(r), dist, parent, stream=stream)
            ev[i + 1].record(stream)
        torch.cuda.synchronize()
        ms = np.array([ev[i].elapsed_time(ev[i + 1]) for i in range(NROOTS)])
        rec[key] = {"gteps_hmean": hmean(m_c / (ms * 1e-3) / 1e9), "root_ms_median": float(np.median(ms)),
                    "total_ms": float(ms.sum())}
        if direction == 0:
            peak, _ = measured_hbm_peak()
            alg = 4.0 * m_c + 32.0 * n_c + 8.125 * n
            ach = float(np.mean(alg / (ms * 1e-3)) / 1e9)
            rec[key]["roofline"] = {"bound": "hbm", "achieved": ach, "peak": peak, "unit": "GB/s",
                                    "frac": ach / peak}
    g.set_option(bfs.BFS_OPT_DIRECTION, 0)
    # oracle on one root (serial, host) -- distances bit-exact
    g.run(int(roots[0]), dist, parent, stream=stream)
    g.sync(stream)
    t0 = time.time()
    d_ref, _, _ = oracle.bfs(off, col, int(roots[0]))
    rec["oracle_s_one_root"] = time.time() - t0
    d0 = dist.cpu().numpy()
    rec["oracle_equal_root0"] = bool(np.array_equal(d0, d_ref))
    del d_ref
    bd = torch.empty((NROOTS, n), dtype=torch.int8, device="cuda")
    g.run_batch(roots, bd, stream=stream)
    bst = g.batch_sync(stream)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    ev[0].record(stream)
    g.run_batch(roots, bd, stream=stream)
    ev[1].record(stream)
    bst = g.batch_sync(stream)
    bms = ev[0].elapsed_time(ev[1])
    rec["batched_int8"] = {"ms": bms, "gteps": bst["edges_scanned"] / (bms * 1e-3) / 1e9,
                           "levels": int(bst["levels"]),
                           "lane0_equals_single_source": bool(
                               np.array_equal(bd[0].cpu().numpy().astype(np.int32), d0))}
    g.close()
    ctx.close()
    print(json.dumps(rec), flush=True)


# ------------------------------------------------- profiling workloads
def levels_arm(args):
    """Small fixed workloads for ncu captures (no JSON line): a seeded
    Kronecker graph of --levels-scale (edge factor 16, seed 22), roots as in
    the headline workload.  --levels-mode:
      hostloop    two single-source traversals with BFS_HOST_LOOP, so each
                  level is its own kernel launch (one ncu result per level);
      do          the same with the direction-optimizing mode;
      persistent  two single-source traversals, device-side level loop;
      timeline    persistent launches with the level timeline: the median
                  time of init, seed and every level over 8 roots, top-down
                  and direction-optimizing;
      batch       four 64-root batched launches (int32 rows, top-down): the
                  mean device time of the last two, the frontier sums and the
                  algorithmic bytes of one launch;
      paths       two shortest-path-count traversals (bfs_run_paths, every
                  entry kept) on the caller's CSR copied to the device."""
    import torch

    import graphgen
    import paper_2103_13577_gb300 as bfs

    mode = args.levels_mode
    off, col = graphgen.kronecker(args.levels_scale, 16, seed=GRAPH_SEED)
    n = len(off) - 1
    roots = graphgen.pick_roots(off, 4, seed=ROOT_SEED)
    ctx = bfs.Context(0)
    if mode == "paths":
        d_off = torch.from_numpy(off).cuda()
        d_col = torch.from_numpy(np.ascontiguousarray(col, dtype=np.int32)).cuda()
        hops = torch.empty(n, dtype=torch.int32, device="cuda")
        sigma = torch.empty(n, dtype=torch.float64, device="cuda")
        for r in roots[:2]:
            print(ctx.run_paths(d_off, d_col, int(r), hops, sigma), flush=True)
        ctx.close()
        return
    g = bfs.Graph(ctx, off, col)
    if mode == "batch":
        rows = torch.empty((NROOTS, n), dtype=torch.int32, device="cuda")
        broots = graphgen.pick_roots(off, NROOTS, seed=ROOT_SEED)
        stream = torch.cuda.current_stream()
        for _ in range(2):
            g.run_batch(broots, rows, stream=stream)
        g.batch_sync(stream)
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        ev[0].record(stream)
        for _ in range(2):
            g.run_batch(broots, rows, stream=stream)
        ev[1].record(stream)
        st = g.batch_sync(stream)
        ms = ev[0].elapsed_time(ev[1]) / 2
        deg = torch.from_numpy(np.diff(off)).cuda()
        sizes, degs, reached = batch_frontier_sums(rows, deg)
        b = batch_algorithmic_bytes(sizes, degs, reached, n, NROOTS, 4)
        print(json.dumps({"ms": ms, "levels": int(st["levels"]),
                          "edges_scanned": int(st["edges_scanned"]), "frontier_entries": sizes,
                          "frontier_edges": degs, "reached": reached, "algorithmic_bytes": b,
                          "gbs": b / (ms * 1e-3) / 1e9}), flush=True)
    else:
        dist = torch.empty(n, dtype=torch.int32, device="cuda")
        par = torch.empty(n, dtype=torch.int32, device="cuda")
        if mode == "timeline":
            level_timeline(bfs, g, graphgen.pick_roots(off, 8, seed=ROOT_SEED), dist, par)
        else:
            flags = bfs.BFS_HOST_LOOP if mode in ("hostloop", "do") else 0
            if mode == "do":
                g.set_option(bfs.BFS_OPT_DIRECTION, 1)
            for r in roots[:2]:
                g.run(int(r), dist, par, flags=flags)
                print(g.sync(), flush=True)
    g.close()
    ctx.close()


def level_timeline(bfs, g, roots, dist, par):
    """Median %globaltimer gaps between init, seed and each level (persistent
    launches, bfs_debug_set_timeline), top-down and direction-optimizing."""
    import torch

    stamps = torch.zeros(64, dtype=torch.int64, device="cuda")
    bfs.bfs_debug_set_timeline(g.handle, stamps)
    for direction in (0, 1):
        g.set_option(bfs.BFS_OPT_DIRECTION, direction)
        rows = []
        for rep in range(2):
            for r in roots:
                stamps.zero_()
                g.run(int(r), dist, par)
                st = g.sync()
                t = stamps.cpu().numpy()
                k = 3 + st["levels"]
                if rep == 1:
                    rows.append(np.diff(t[:k]) / 1e3)
        width = max(len(x) for x in rows)
        a = np.full((len(rows), width), np.nan)
        for i, x in enumerate(rows):
            a[i, :len(x)] = x
        med = np.nanmedian(a, axis=0)
        tot = np.median([x.sum() for x in rows])
        names = ["init", "seed"] + [f"L{i}" for i in range(width - 2)]
        print(f"direction {direction} total_us {tot:.1f} " +
              " ".join(f"{nm}={v:.1f}" for nm, v in zip(names, med)), flush=True)
    g.set_option(bfs.BFS_OPT_DIRECTION, 0)
    bfs.bfs_debug_set_timeline(g.handle, None)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--bins", default="", help="t_small,t_large,chunk_warp,chunk_cta")
    ap.add_argument("--ctas-per-sm", type=int, default=0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extras", action="store_true",
                    help="headline line only: skip the scale-24 batched and serving sections")
    ap.add_argument("--cpu-budget", type=float, default=15.0)
    ap.add_argument("--serve-scales", default="18,20,22,24")
    ap.add_argument("--serve-rates", default="1000,10000,50000")
    ap.add_argument("--serve-window", type=float, default=1.0)
    ap.add_argument("--serve-max-queries", type=int, default=20000)
    ap.add_argument("--serve-budget", type=int, default=32, help="GiB")
    ap.add_argument("--large-scale", type=int, default=29)
    ap.add_argument("--large-ef", type=int, default=8)
    ap.add_argument("--workload", default="plain",
                    choices=["plain", "batched", "serve", "large", "levels"],
                    help="plain: the headline line (default); batched: the 64-root batched "
                         "configuration on Kronecker and Erdos-Renyi graphs; serve: the query "
                         "server; large: scale 29; levels: small fixed runs for ncu captures")
    ap.add_argument("--levels-mode", default="hostloop",
                    choices=["hostloop", "do", "persistent", "timeline", "batch", "paths"])
    ap.add_argument("--levels-scale", type=int, default=22)
    ap.add_argument("--batch-scale", type=int, default=24)
    args = ap.parse_args()
    args.warmup = max(3, args.warmup)
    rank = env_int("RANK", 0)
    world = env_int("WORLD_SIZE", 1)
    local_rank = env_int("LOCAL_RANK", 0)
    if args.impl == "reference":
        reference_arm(args, rank, world)
        return
    if args.workload == "batched":
        if rank == 0:
            batched_arm(args)
        return
    if args.workload == "serve":
        if rank == 0:
            serve_arm(args)
        return
    if args.workload == "large":
        if rank == 0:
            large_arm(args)
        return
    if args.workload == "levels":
        if rank == 0:
            levels_arm(args)
        return
    if world > 1:
        import torch
        import torch.distributed as dist_mod
        torch.cuda.set_device(local_rank)
        dist_mod.init_process_group("nccl")
    gpu_arm(args, rank, world, local_rank)
    if world > 1:
        import torch.distributed as dist_mod
        dist_mod.destroy_process_group()


if __name__ == "__main__":
    main()
