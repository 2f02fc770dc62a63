// bfs_kernels.cu -- the top-down level step on sm_103a: the single-source
// traversal with every optional path (the default one is bfs_single.cu), the
// batched traversal, and the host- and graph-driven level loops.
//
// Algorithm 2 Phase 1 with one compute node (= Algorithm 1 with an atomic
// enqueue): every vertex v of the current frontier scans adj(v); each
// neighbour u whose distance is still infinity is claimed by exactly one
// thread (the claim is an atomicOr on the visited bitmap; Algorithm 2 gates
// the distance write on the success of the atomic enqueue), which writes
// d[u] = level + 1 and appends u to the next frontier.  When the frontier is
// empty the traversal ends (the While loop of Algorithm 1).
//
// GB300 design:
//  * The whole level loop runs inside one cooperative persistent launch
//    (grid = resident CTAs of all 152 SMs) separated by a grid barrier
//    whose wait is bounded by %globaltimer, so no per-level host round trip;
//    the same level kernels also run as the body of a CUDA-graph while loop
//    (phases 5-9 of the step kernels) or one launch per level from the host.
//  * Load balancing replaces the paper's Logarithmic Radix Binning (one
//    kernel per log2-degree bin, Section "Load Balanced Traversals Per
//    compute-node") with three degree bins written while the next frontier
//    is built: deg < t_small (edges of 32 vertices spread over the warp by a
//    scan), t_small <= deg < t_large (warp chunks of 16-byte column units
//    over several rows, 128-bit loads) and deg >= t_large (CTA chunks;
//    heavy vertices span many CTAs).  Each bin counter packs (entries << 34 |
//    edge prefix) so that one 64-bit atomicAdd per bin reserves queue slots
//    and edge ranges at once; warp and CTA work items are fixed-size edge
//    chunks, located through a chunk-start table filled at enqueue time.
//  * Probes read the visited bitmap with plain loads, 8 per lane in flight;
//    the atomicOr claims are batched -- per probe round when it has many
//    candidates, otherwise per 64-entry stage at flush time.
//  * The batched traversal carries a 64-bit source-lane set per vertex:
//    phase A ORs the frontier lanes into next[u] (or, bottom-up, ORs the
//    neighbours' frontier lanes into each vertex that lacks some), phase B
//    (a sweep) turns the lanes that are new into distances and the next
//    frontier.
#include "bfs_device.cuh"

namespace bfs {
inline namespace device_optional {

// ------------------------------------------------------------ expansion
// A heavy vertex's column run read through shared memory (BFS_OPT_TMA_STAGE):
// the warp's 256-entry blocks of the run (block j at wbase + 2048 j
// entries from a4, as in the CTA-interleaved schedule below) stream through
// its two 1 KB buffers, each filled by one TMA bulk copy that lane 0 issues
// two blocks ahead, so the next block is in flight while the current one is
// probed.  valid entries: [lo, hi) relative to a4 (16-byte aligned).
__device__ void expand_segment_staged(const TraversalParams& P, Stage<false>& S, long long a4,
                                      int lo, int hi, int32_t v, int level, int nxt, int nslot,
                                      int wbase) {
    const unsigned lane = lane_id();
    const int nblk = wbase < hi ? (hi - wbase + 2047) / 2048 : 0;
    if (nblk == 0 || !S.tma_ok) return;
    uint4* const buf = S.tma_buf;
    unsigned long long* const bar = S.tma_bar;
    unsigned ph = S.tma_ph;
    const int32_t* const colp = P.col + a4;
    auto issue = [&](int j) {  // lane 0
        const int rw = wbase + j * 2048;
        const int cnt = min(256, hi - rw);
        const unsigned bytes = (unsigned)((cnt * 4 + 15) & ~15);
        const int b = j & 1;
        // the buffer's previous contents were read by the generic proxy
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(bar + b, bytes);
        tma_load_1d(buf + b * 64, colp + rw, bytes, bar + b);
    };
    if (lane == 0) {
        issue(0);
        if (nblk > 1) issue(1);
    }
    int j = 0;
    bool ok = true;
    for (; j < nblk; ++j) {
        const int b = j & 1;
        ok = __all_sync(FULL_MASK, mbar_wait_bounded(P, bar + b, (ph >> b) & 1u));
        if (!ok) break;
        ph ^= 1u << b;
        const uint4 x0 = buf[b * 64 + lane], x1 = buf[b * 64 + 32 + lane];
        __syncwarp();
        if (lane == 0 && j + 2 < nblk) issue(j + 2);
        const int r0 = wbase + j * 2048 + 4 * (int)lane, r1 = r0 + 128;
        unsigned okm = 0u;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (r0 + c >= lo && r0 + c < hi) okm |= 1u << c;
            if (r1 + c >= lo && r1 + c < hi) okm |= 1u << (4 + c);
        }
        const int32_t u[8] = {(int32_t)x0.x, (int32_t)x0.y, (int32_t)x0.z, (int32_t)x0.w,
                              (int32_t)x1.x, (int32_t)x1.y, (int32_t)x1.z, (int32_t)x1.w};
        const int32_t vv[8] = {v, v, v, v, v, v, v, v};
        visit_plain_k<8>(P, S, okm, u, [&](int j) { return vv[j]; }, level, nxt, nslot);
    }
    if (!ok) {
        // a copy did not land in time: stop the launch, then let the copies
        // still in flight (blocks j and j + 1) complete before leaving
        if (lane == 0) {
            raise_status(P, kDevTimeout);
            give_up(P);
            for (int k = j; k < min(j + 2, nblk); ++k) {
                const int b = k & 1;
                const unsigned long long t0 = global_timer_ns();
                while (!mbar_try_wait(bar + b, (ph >> b) & 1u) &&
                       global_timer_ns() - t0 < (unsigned long long)P.timeout_ns) {
                }
                ph ^= 1u << b;
            }
            S.tma_ok = 0;
        }
    }
    if (lane == 0) S.tma_ph = ph;
    __syncwarp();
}

// One level's expansion.  CTA chunks (bin 2) are pulled from a counter so
// heavy vertices spread over whichever CTAs are free; warp items (bin 1
// chunks, then bin 0 groups) are equal-sized by construction and dealt out
// round robin over all warps of the grid, with no atomics or CTA barriers.
// Each warp flushes its staged discoveries at the end; the CTA adds its
// discovered-vertex count with one atomic.
// Bottom-up level (Section "Top Down Vs. Bottom Up"; the paper notes its
// exchange works with either direction): every vertex not yet visited looks
// for a neighbour in the current frontier bitmap and stops at the first.
// A warp owns one 32-vertex visited word at a time, so claims need no
// atomics.  Found vertices go through the same stage as top-down winners
// (distance level + 1, parent = the frontier neighbour, next frontier).
__device__ void bottom_up_level(const TraversalParams& P, Stage<false>& S, int level, int nxt,
                                int nslot) {
    const uint32_t* F = P.fb[level % 3];
    const unsigned lane = lane_id();
    const long long words = (P.bu_limit + 31) / 32;
    const long long nwarps = (long long)gridDim.x * kWarps;
    for (long long w = (long long)blockIdx.x * kWarps + (threadIdx.x >> 5); w < words; w += nwarps) {
        const uint32_t vis = __ldcg(P.visited + w);
        const long long v = w * 32 + lane;
        const bool unv = v < P.bu_limit && !((vis >> lane) & 1u);
        if (__ballot_sync(FULL_MASK, unv) == 0u) continue;
        bool found = false;
        int32_t par = 0;
        if (unv) {
            long long k = __ldg(P.off + v);
            const long long e = __ldg(P.off + v + 1);
            for (; k + 4 <= e && !found; k += 4) {
                const int32_t u0 = __ldg(P.col + k), u1 = __ldg(P.col + k + 1);
                const int32_t u2 = __ldg(P.col + k + 2), u3 = __ldg(P.col + k + 3);
                const uint32_t f0 = F[u0 >> 5], f1 = F[u1 >> 5], f2 = F[u2 >> 5], f3 = F[u3 >> 5];
                if ((f0 >> (u0 & 31)) & 1u) { found = true; par = u0; }
                else if ((f1 >> (u1 & 31)) & 1u) { found = true; par = u1; }
                else if ((f2 >> (u2 & 31)) & 1u) { found = true; par = u2; }
                else if ((f3 >> (u3 & 31)) & 1u) { found = true; par = u3; }
            }
            for (; k < e && !found; ++k) {
                const int32_t u0 = __ldg(P.col + k);
                if ((F[u0 >> 5] >> (u0 & 31)) & 1u) { found = true; par = u0; }
            }
        }
        // the warp is the only one looking at word w, so the flush's claim of
        // a found vertex always wins
        stage_push<false>(P, S, found, (int32_t)v, par, 0ull, level, nxt, nslot);
    }
}

// Batched bottom-up level (a multi-source BFS over lane sets): every vertex
// that lacks some lane whose frontier is non-empty ORs the frontier lane
// sets of its neighbours and stops once it has every such lane.  Rows are
// scanned two ways: a warp scans one row 32 entries per step, OR-reducing
// the lane sets across the warp (the heavy vertices -- below `heavy_end`
// in the degree order, one vertex per warp spread over the grid -- and any
// heavy row met among the light ones), and a lane scans a light row four
// entries at a time.  The lanes found go to next[v] (each vertex has one
// owner, so no atomics) and the sweep turns them into distances and the
// next frontier, as after a top-down level.  Frontier sets are read past
// L1 (the previous level's sweep wrote them).
__device__ __forceinline__ uint64_t warp_scan_row(const unsigned long long* F, const int32_t* col,
                                                  long long k, long long e, uint64_t need) {
    const unsigned lane = lane_id();
    uint64_t found = 0ull;
    for (long long kk = k; kk < e; kk += 32) {
        uint64_t f = 0ull;
        if (kk + lane < e) f = __ldcg(F + __ldg(col + kk + lane));
        const unsigned lo = __reduce_or_sync(FULL_MASK, (unsigned)f);
        const unsigned hi = __reduce_or_sync(FULL_MASK, (unsigned)(f >> 32));
        found |= ((uint64_t)hi << 32) | lo;
        if ((found & need) == need) break;
    }
    return found;
}

__device__ void bottom_up_batch_level(const TraversalParams& P, int level) {
    const unsigned lane = lane_id();
    // only lanes whose frontier is non-empty can be found at this level; a
    // lane whose traversal has ended would otherwise keep every vertex it
    // never reaches scanning its whole row
    const uint64_t live = ld_cg_u64(&P.ctl[level % 3].front_lanes);
    const unsigned long long* F = reinterpret_cast<const unsigned long long*>(P.lane_front);
    unsigned long long* const vn = reinterpret_cast<unsigned long long*>(P.lane_vn);
    const long long nwarps = (long long)gridDim.x * kWarps;
    const long long gw = (long long)blockIdx.x * kWarps + (threadIdx.x >> 5);
    const long long heavy_end = min(P.bitmap_from, P.bu_limit);
    for (long long v = gw; v < heavy_end; v += nwarps) {
        const uint64_t need = live & ~__ldcg(vn + 2 * v);
        if (need == 0ull) continue;
        const uint64_t found =
            warp_scan_row(F, P.col, __ldg(P.off + v), __ldg(P.off + v + 1), need);
        if (lane == 0 && (found & need) != 0ull) vn[2 * v + 1] = found & need;
    }
    const long long groups = (P.bu_limit - heavy_end + 31) / 32;
    for (long long w = gw; w < groups; w += nwarps) {
        const long long v = heavy_end + w * 32 + lane;
        uint64_t need = 0ull;
        long long k = 0, e = 0;
        if (v < P.bu_limit) {
            need = live & ~__ldcg(vn + 2 * v);
            if (need != 0ull) {
                k = __ldg(P.off + v);
                e = __ldg(P.off + v + 1);
            }
        }
        const bool heavy = e - k > 32;
        if (__ballot_sync(FULL_MASK, need != 0ull) == 0u) continue;
        uint64_t found = 0ull;
        if (need != 0ull && !heavy) {
            for (; k + 4 <= e; k += 4) {
                const int32_t u0 = __ldg(P.col + k), u1 = __ldg(P.col + k + 1);
                const int32_t u2 = __ldg(P.col + k + 2), u3 = __ldg(P.col + k + 3);
                found |= __ldcg(F + u0) | __ldcg(F + u1) | __ldcg(F + u2) | __ldcg(F + u3);
                if ((found & need) == need) break;
            }
            if ((found & need) != need)
                for (; k < e; ++k) {
                    found |= __ldcg(F + __ldg(P.col + k));
                    if ((found & need) == need) break;
                }
        }
        for (unsigned hm = __ballot_sync(FULL_MASK, need != 0ull && heavy); hm != 0u; hm &= hm - 1u) {
            const int src = __ffs(hm) - 1;
            const uint64_t hf = warp_scan_row(F, P.col, __shfl_sync(FULL_MASK, k, src),
                                              __shfl_sync(FULL_MASK, e, src),
                                              __shfl_sync(FULL_MASK, need, src));
            if ((int)lane == src) found = hf;
        }
        const uint64_t nx = found & need;
        if (nx != 0ull) vn[2 * v + 1] = nx;
    }
}

// Position of the set bit of rank n (0-based) in x, which has more than n
// set bits: the largest p with fewer than n + 1 set bits below p.
__device__ __forceinline__ int nth_set_bit(uint32_t x, int n) {
    int pos = 0;
#pragma unroll
    for (int st = 16; st > 0; st >>= 1)
        if (__popc(x & ((1u << (pos + st)) - 1u)) <= n) pos += st;
    return pos;
}

// Top-down over the frontier bitmap (dense levels, "queue -> bitmap"): the
// light bin (deg < t_small, most of the vertices) is read from the frontier
// bitmap instead of its queue.  A warp takes a tile of 32 bitmap words
// (1024 consecutive vertices); its light frontier vertices, in vertex order,
// are gathered 32 at a time and their rows cut into 16-byte units as in the
// warp bin.  After the degree-ordered renumbering the light vertices are
// one id range with adjacent rows, so a tile's column reads are close to
// one stream.  The heavier bins keep their (balanced) queues.
__device__ void expand_bitmap_tile(const TraversalParams& P, Stage<false>& S, long long tile,
                                   int level, int nxt, int nslot) {
    const uint32_t* F = P.fb[level % 3];
    const unsigned lane = lane_id();
    const long long words = (P.n + 31) / 32;
    const long long w = tile * 32 + lane;
    const uint32_t word = w < words ? __ldcg(F + w) : 0u;
    const int pc = __popc(word);
    const int pincl = warp_incl_scan(pc);
    const int pexcl = pincl - pc;
    const int nfront = __shfl_sync(FULL_MASK, pincl, 31);
    for (int k0 = 0; k0 < nfront; k0 += 32) {
        const int k = k0 + (int)lane;
        int o = 0;
#pragma unroll
        for (int st = 16; st > 0; st >>= 1) {
            const int c = o + st;
            if (__shfl_sync(FULL_MASK, pexcl, c & 31) <= k) o = c;
        }
        const uint32_t ow = __shfl_sync(FULL_MASK, word, o);
        const int oex = __shfl_sync(FULL_MASK, pexcl, o);
        bool ok = k < nfront;
        int32_t v = 0;
        long long a = 0, b = 0;
        if (ok) {
            const int bit = nth_set_bit(ow, k - oex);
            v = (int32_t)((tile * 32 + o) * 32 + bit);
            a = __ldg(P.off + v);
            b = __ldg(P.off + v + 1);
            if (b - a >= P.t_small || b == a) ok = false;
        }
        // unit gather over the (up to 32) rows
        const long long a4 = a & ~3ll;
        const int rlo = (int)(a - a4), rhi = (int)(b - a4);
        const int units = ok ? (rhi + 3) >> 2 : 0;
        const int incl = warp_incl_scan(units);
        const int excl = incl - units;
        const int total = __shfl_sync(FULL_MASK, incl, 31);
        for (int q0 = 0; q0 < total; q0 += 64) {
            unsigned okm = 0u;
            int32_t u[8], vv[8];
            uint64_t mm[8];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int q = q0 + 32 * h + (int)lane;
                int oo = 0;
#pragma unroll
                for (int st = 16; st > 0; st >>= 1) {
                    const int c = oo + st;
                    if (__shfl_sync(FULL_MASK, excl, c & 31) <= q) oo = c;
                }
                const long long a4o = __shfl_sync(FULL_MASK, a4, oo);
                const int lo_o = __shfl_sync(FULL_MASK, rlo, oo);
                const int hi_o = __shfl_sync(FULL_MASK, rhi, oo);
                const int xo = __shfl_sync(FULL_MASK, excl, oo);
                const int32_t vo = __shfl_sync(FULL_MASK, v, oo);
                const int r = 4 * (q - xo);
                int4 x = make_int4(0, 0, 0, 0);
                if (q < total) {
                    x = __ldcs(reinterpret_cast<const int4*>(P.col + a4o + r));
                    okm |= unit_mask(r, lo_o, hi_o) << (4 * h);
                }
                u[4 * h + 0] = x.x;
                u[4 * h + 1] = x.y;
                u[4 * h + 2] = x.z;
                u[4 * h + 3] = x.w;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    vv[4 * h + c] = vo;
                    mm[4 * h + c] = 0ull;
                }
            }
            visit_k<false, 8>(P, S, okm, u, vv, mm, level, nxt, nslot);
        }
    }
}

}  // inline namespace

// Batched top-down levels: what the previous sweep found out about vertices
// that every live lane has reached.  Their bitmap is used once it holds a
// 64th of the vertices; when it holds a whole prefix of the degree order, the
// rows skip the entries that lead there (see kCutDegree).
__device__ __forceinline__ void batch_filters(const TraversalParams& P, Stage<true>& S,
                                              const LevelShape& L, int level) {
    if (lane_id() != 0) return;
    const uint32_t* full = nullptr;
    const uint16_t* cut = nullptr;
    // (a level of few entries does not wait for the counters)
    if (P.full != nullptr && level > 0 && 16 * (L.edges[0] + L.edges[1] + L.edges[2]) >= P.nnz) {
        const LevelCtl& C = P.ctl[level % 3];
        if (64ll * __ldcg(&C.full_count) >= P.sweep_limit) {
            full = P.full;
            const unsigned clear = __ldcg(&C.clear_word);
            const long long prefix = clear == 0u ? P.sweep_limit : 32ll * (0xffffffffu - clear);
            if (P.cut != nullptr)
                for (int c = 0; c < kCutClasses; ++c)
                    if (P.cut_bound[c] > 0 && P.cut_bound[c] <= prefix) cut = P.cut + c * P.n;
        }
    }
    S.hot = full;
    S.cut = cut;
}
template <bool kBatch>
__device__ __forceinline__ void batch_filters(const TraversalParams&, Stage<kBatch>&,
                                              const LevelShape&, int) {}

template <bool kBatch, bool kStaged = false>
__device__ void expand_level(const TraversalParams& P, Stage<kBatch>& S, const LevelShape& L,
                             int level, uint32_t* s_hot, int dir = 0) {
    __shared__ int s_disc;
    const int nslot = (level + 1) % 3;
    const int nxt = (level & 1) ^ 1;
    if (threadIdx.x == 0) s_disc = 0;
    if (lane_id() == 0) S.disc = 0;
    if (!kBatch) {
        // large levels: copy the hot prefix of the visited bitmap (after the
        // degree-ordered renumbering, the highest-degree vertices) into
        // shared memory; most probes of a dense level end there
        const long long ledges = L.edges[0] + L.edges[1] + L.edges[2];
        const int words = (P.hot_words > 0 && ledges >= P.hot_min_edges)
                              ? (int)min((long long)P.hot_words, (long long)((P.n + 31) / 32)) : 0;
        if (words > 0) {
            const int w4 = words / 4;
            const uint4* src = reinterpret_cast<const uint4*>(P.visited);
            uint4* dst = reinterpret_cast<uint4*>(s_hot);
            for (int i = threadIdx.x; i < w4; i += kBlock) dst[i] = __ldcg(src + i);
            for (int i = w4 * 4 + threadIdx.x; i < words; i += kBlock) s_hot[i] = __ldcg(P.visited + i);
        }
        if (lane_id() == 0) {
            S.hot = s_hot;
            S.hot_bits = words * 32;
        }
    } else {
        batch_filters(P, S, L, level);
    }
    __syncthreads();
    bool bottom_up = false;
    if (dir == 2) {
        if constexpr (kBatch) bottom_up_batch_level(P, level);
        else bottom_up_level(P, S, level, nxt, nslot);
        bottom_up = true;
    }
    if (!bottom_up) expand_top_down<kBatch, kStaged>(P, S, L, level, dir == 1);
    stage_flush<kBatch>(P, S, level, nxt, nslot);
    if (!kBatch) {
        if (lane_id() == 0 && S.disc > 0) atomicAdd(&s_disc, S.disc);
        __syncthreads();
        if (threadIdx.x == 0 && s_disc > 0) atomicAdd(&P.ctl[nslot].discovered, (unsigned)s_disc);
    }
}

// ------------------------------------------------------------- init/seed
__device__ void fill_u64(uint64_t* p, long long n, long long tid, long long nthreads) {
    for (long long i = tid; i < n; i += nthreads) p[i] = 0ull;
}

__device__ void init_plain(const TraversalParams& P, long long tid, long long nthreads) {
    if (blockIdx.x == 0 && threadIdx.x < 3 * (int)(sizeof(LevelCtl) / 8))
        reinterpret_cast<unsigned long long*>(P.ctl)[threadIdx.x] = 0ull;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        P.stats->levels = 0;
        P.stats->reached = 0;
        P.stats->edges = 0;
        P.stats->status = 0;
        P.stats->max_level = 0;
        P.stats->bu_levels = 0;
        P.stats->graph_seen = 0;
        P.stats->graph_level = 0;
        P.stats->graph_prev_bu = 0;
        P.stats->graph_dir = 0;
    }
    const long long words = (P.n + 31) / 32;
    fill_bytes(P.visited, words * 4, 0, tid, nthreads);
    if (P.fb[0])
        for (int f = 0; f < 3; ++f) fill_bytes(P.fb[f], words * 4, 0, tid, nthreads);
    fill_bytes(P.dist, P.n * 4, 0xff, tid, nthreads);
    if (P.parent) fill_bytes(P.parent, P.n * 4, 0xff, tid, nthreads);
}

__device__ void seed_plain(const TraversalParams& P, Stage<false>& S) {
    if (blockIdx.x != 0 || threadIdx.x >= 32) return;
    const bool l0 = threadIdx.x == 0;
    const int32_t root = P.old2new ? __ldg(P.old2new + P.root_caller) : P.root_caller;
    if (l0) P.ctl[0].discovered = 1u;
    // staged with level -1 and itself as parent: the flush writes dist 0 and
    // parent = root, and queues the root in the bin of its degree
    stage_push<false>(P, S, l0, root, root, 0ull, -1, 0, 0);
    stage_flush<false>(P, S, -1, 0, 0);
}

// Per-level housekeeping of the frontier bitmaps: the bitmap the level after
// next will fill is cleared now (it held the previous level's frontier);
// bottom-up levels are counted.
__device__ void prepare_level(const TraversalParams& P, int level, int dir, long long tid,
                              long long nthreads) {
    if (!P.fb[0]) return;
    fill_bytes(P.fb[(level + 2) % 3], ((P.n + 31) / 32) * 4, 0, tid, nthreads);
    if (dir == 2 && blockIdx.x == 0 && threadIdx.x == 0) P.stats->bu_levels += 1;
}

// Books the level that is about to be expanded; block 0, thread 0 only.
__device__ void book_level(const TraversalParams& P, const LevelShape& S, int level) {
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    // clear the slot that the level after next will fill
    unsigned long long* z = reinterpret_cast<unsigned long long*>(P.ctl + (level + 2) % 3);
    for (int i = 0; i < (int)(sizeof(LevelCtl) / 8); ++i) z[i] = 0ull;
    if (S.discovered > 0) {
        P.stats->levels = level + 1;
        P.stats->reached += S.discovered;
    }
    P.stats->edges += S.edges[0] + S.edges[1] + S.edges[2];
}

// Direction of a batched level: bottom-up when the frontier's degree sum
// exceeds the degree sum of the vertices some lane has not reached yet plus
// 4 entries per vertex (a bottom-up level reads every vertex's lane sets),
// decided afresh each level.  Unlike the single-source rule (Beamer et al.,
// alpha 15 / beta 18) a bottom-up vertex stops only once it has every lane
// it lacks, not at its first frontier neighbour, so bottom-up pays off only
// on the levels whose frontiers cover most of the graph.
__device__ __forceinline__ int batch_direction(const TraversalParams& P, const LevelShape& L,
                                               bool prev_bu) {
    (void)prev_bu;
    if (P.dir_mode == 0) return 0;
    if (P.dir_mode == 2) return 2;
    const long long mf = L.edges[0] + L.edges[1] + L.edges[2];
    const long long full = (long long)ld_cg_u64(
        reinterpret_cast<const unsigned long long*>(&P.stats->full_edges));
    return mf > P.nnz - full + 4 * P.n ? 2 : 0;
}

// ------------------------------------------- graph-captured level loop
// End of one loop-body launch (one CTA, thread 0): carry the direction
// state to the next level and set the while node's condition -- 0 when the
// next frontier is empty (its discoveries of degree-0 vertices are booked
// first, as the device-side loop does) or the launch failed.
__device__ void graph_advance_plain(const TraversalParams& P) {
    if (threadIdx.x != 0) return;
    DevStats* st = P.stats;
    const int level = st->graph_level;
    const int slot = level % 3, nslot = (level + 1) % 3;
    long long mf = 0, nf_next = 0;
#pragma unroll
    for (int b = 0; b < kBins; ++b) {
        mf += (long long)(ld_cg_u64(&P.ctl[slot].packed[b]) & kEdgeMask);
        nf_next += (long long)(ld_cg_u64(&P.ctl[nslot].packed[b]) >> kCountShift);
    }
    st->graph_seen += mf;
    st->graph_prev_bu = st->graph_dir == 2 ? 1 : 0;
    st->graph_level = level + 1;
    unsigned go = 1u;
    if (nf_next == 0 || ld_volatile_i32(&st->status) != 0) {
        if (nf_next == 0) book_level(P, read_level(P, level + 1), level + 1);
        go = 0u;
    }
    cudaGraphSetConditional(P.graph_cond, go);
}

// Batched body end: records the level count, applies the int8 depth limit
// and sets the while node's condition for the next level.
__device__ void graph_advance_batch(const TraversalParams& P) {
    if (threadIdx.x != 0) return;
    DevStats* st = P.stats;
    const int level = st->graph_level;
    const int nslot = (level + 1) % 3;
    if (ld_cg_u64(reinterpret_cast<const unsigned long long*>(&P.ctl[nslot].new_lanes)) > 0ull)
        st->levels = level + 2;
    long long nf_next = 0;
#pragma unroll
    for (int b = 0; b < kBins; ++b)
        nf_next += (long long)(ld_cg_u64(&P.ctl[nslot].packed[b]) >> kCountShift);
    st->graph_level = level + 1;
    st->graph_prev_bu = st->graph_dir == 2 ? 1 : 0;
    unsigned go = (nf_next > 0 && ld_volatile_i32(&st->status) == 0) ? 1u : 0u;
    if (go && P.dist_int8 && level + 2 > 126) {
        raise_status(P, kDevDepth);
        go = 0u;
    }
    cudaGraphSetConditional(P.graph_cond, go);
}

// --------------------------------------------------------- plain kernels
// kStaged: heavy runs go through the TMA staging buffers (BFS_OPT_TMA_STAGE);
// a separate instantiation, so the default kernel carries none of that code.
template <int MB, bool kStaged>
__global__ void __launch_bounds__(kBlock, MB)
bfs_plain_persistent(const __grid_constant__ TraversalParams P) {
    extern __shared__ uint4 s_dyn[];
    uint32_t* s_hot = reinterpret_cast<uint32_t*>(s_dyn);
    __shared__ Stage<false> s_stage[kWarps];
    Stage<false>& S = s_stage[threadIdx.x >> 5];
    stage_init(S);
    if (kStaged) tma_setup(P, S, s_dyn);
    const long long nthreads = (long long)gridDim.x * kBlock;
    const long long tid = (long long)blockIdx.x * kBlock + threadIdx.x;
    stamp(P, 0);
    init_plain(P, tid, nthreads);
    __shared__ unsigned long long epoch;
    if (threadIdx.x == 0) epoch = 0ull;
    if (grid_barrier(P, epoch)) {
        stamp(P, 1);
        seed_plain(P, S);
        if (grid_barrier(P, epoch)) {
            stamp(P, 2);
            long long seen_edges = 0;  // edges of all frontiers so far (same in every CTA)
            bool prev_bu = false;
            for (int level = 0;; ++level) {
                const LevelShape L = read_level(P, level);
                book_level(P, L, level);
                const long long nf = L.cnt[0] + L.cnt[1] + L.cnt[2];
                if (nf == 0) break;
                const long long mf = L.edges[0] + L.edges[1] + L.edges[2];
                seen_edges += mf;
                const int dir = (P.fb[0]) ? choose_direction(P.dir_mode, prev_bu, mf, P.nnz - seen_edges,
                                                           nf, P.n, P.do_alpha, P.do_beta,
                                                           P.bitmap_div)
                                        : 0;
                prepare_level(P, level, dir, tid, nthreads);
                expand_level<false, kStaged>(P, S, L, level, s_hot, dir);
                prev_bu = dir == 2;
                if (!grid_barrier(P, epoch)) break;
                stamp(P, 3 + level);
            }
        }
    }
    kernel_exit(P);
}

// Host-loop variant: one launch per phase / level, no grid barrier.
template <int MB, bool kStaged>
__global__ void __launch_bounds__(kBlock, MB)
bfs_plain_step(const __grid_constant__ TraversalParams P) {
    extern __shared__ uint4 s_dyn[];
    uint32_t* s_hot = reinterpret_cast<uint32_t*>(s_dyn);
    __shared__ Stage<false> s_stage[kWarps];
    Stage<false>& S = s_stage[threadIdx.x >> 5];
    stage_init(S);
    if (kStaged) tma_setup(P, S, s_dyn);
    const long long nthreads = (long long)gridDim.x * kBlock;
    const long long tid = (long long)blockIdx.x * kBlock + threadIdx.x;
    if (P.phase == 0) {
        init_plain(P, tid, nthreads);
    } else if (P.phase == 1) {
        seed_plain(P, S);
    } else if (P.phase == 2) {
        const LevelShape L = read_level(P, P.level);
        book_level(P, L, P.level);
        if (L.cnt[0] + L.cnt[1] + L.cnt[2] == 0) return;
        const int dir = (P.fb[0] && P.dir_override > 0) ? P.dir_override : 0;
        prepare_level(P, P.level, dir, tid, nthreads);
        expand_level<false, kStaged>(P, S, L, P.level, s_hot, dir);
    } else if (P.phase == 5) {
        // graph-captured loop body: the level and the direction state come
        // from the device (written by the previous body launch)
        const int level = ld_volatile_i32(&P.stats->graph_level);
        const LevelShape L = read_level(P, level);
        book_level(P, L, level);
        const long long nf = L.cnt[0] + L.cnt[1] + L.cnt[2];
        if (nf == 0) return;
        const long long mf = L.edges[0] + L.edges[1] + L.edges[2];
        const long long seen = *(volatile long long*)&P.stats->graph_seen + mf;
        const int dir = P.fb[0] ? choose_direction(P.dir_mode,
                                                   ld_volatile_i32(&P.stats->graph_prev_bu) != 0,
                                                   mf, P.nnz - seen, nf, P.n, P.do_alpha,
                                                   P.do_beta, P.bitmap_div)
                                : 0;
        if (blockIdx.x == 0 && threadIdx.x == 0) P.stats->graph_dir = dir;
        prepare_level(P, level, dir, tid, nthreads);
        expand_level<false, kStaged>(P, S, L, level, s_hot, dir);
    } else if (P.phase == 6) {
        graph_advance_plain(P);
    }
}

// ------------------------------------------------------- batched kernels
__device__ void init_batch(const TraversalParams& P, long long tid, long long nthreads) {
    if (blockIdx.x == 0 && threadIdx.x < 3 * (int)(sizeof(LevelCtl) / 8))
        reinterpret_cast<unsigned long long*>(P.ctl)[threadIdx.x] = 0ull;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        P.stats->levels = 0;
        P.stats->reached = 0;
        P.stats->edges = 0;
        P.stats->status = 0;
        P.stats->max_level = 0;
        P.stats->bu_levels = 0;
        P.stats->graph_level = 0;
        P.stats->graph_seen = 0;
        P.stats->graph_prev_bu = 0;
        P.stats->graph_dir = 0;
        P.stats->full_edges = 0;
    }
    fill_u64(P.lane_vn, 2 * P.n, tid, nthreads);
    if (P.dir_mode != 0) fill_u64(P.lane_front, P.n, tid, nthreads);
    // distances are not filled here: emit_batch writes every (lane, vertex)
}

// Levels per vertex and lane, bit-sliced: plane j of vertex v (a 64-bit word,
// 8 planes or 64 bytes per vertex) holds bit j of every lane's level, so a
// sweep gives all of a vertex's new lanes their level with one or two 16-byte
// updates of one 32-byte sector.  Planes 4 to 7 exist from level 16 on: that
// level's sweep clears them for the vertices reached before.  The value 255
// means "level >= 255, written straight into dist".
__device__ __forceinline__ ulonglong2* level_planes(const TraversalParams& P, long long v) {
    return reinterpret_cast<ulonglong2*>(P.lane_level + v * 64);
}
__device__ __forceinline__ ulonglong2 plane_bits(int lvl, int pair, uint64_t lanes) {
    return make_ulonglong2((lvl >> (2 * pair)) & 1 ? lanes : 0ull,
                           (lvl >> (2 * pair + 1)) & 1 ? lanes : 0ull);
}

// Bits 4q .. 4q + 3 of x, one per byte (a 4-bit number times 2^0 + 2^7 + 2^14
// + 2^21 puts bit i at bit 8 i, among others that the mask removes).
template <typename T>
__device__ __forceinline__ uint32_t spread4(T x, int q) {
    return (((uint32_t)(x >> (4 * q)) & 0xfu) * 0x00204081u) & 0x01010101u;
}
// Byte b of x, sign-extended.
template <int B>
__device__ __forceinline__ int signed_byte(uint32_t x) {
    int r;
    constexpr int kSel = B | ((8 | B) << 4) | ((8 | B) << 8) | ((8 | B) << 12);
    asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(x), "n"(kSel));
    return r;
}

// Bytes of four vertices (byte i: lane i) to rows of four vertices: row[i]
// byte j is b[j] byte i.
__device__ __forceinline__ void transpose4(const uint32_t (&b)[4], uint32_t (&row)[4]) {
    const uint32_t t0 = __byte_perm(b[0], b[1], 0x5140), t1 = __byte_perm(b[2], b[3], 0x5140);
    const uint32_t t2 = __byte_perm(b[0], b[1], 0x7362), t3 = __byte_perm(b[2], b[3], 0x7362);
    row[0] = __byte_perm(t0, t1, 0x5410);
    row[1] = __byte_perm(t0, t1, 0x7632);
    row[2] = __byte_perm(t2, t3, 0x5410);
    row[3] = __byte_perm(t2, t3, 0x7632);
}

// Low byte of x as a level, 255 as -1.
__device__ __forceinline__ int level_or_none(uint32_t x) { return (int)((x + 1u) & 0xffu) - 1; }

// emit_batch for levels 16 to 254 and rows that allow wide stores: all 8
// planes, 16 lanes at a time (those of four vertices and 64 lanes would take
// 64 registers; a vertex's 64 bytes come from L1 after the first 16 lanes).
// Where there are fewer groups of four vertices than threads, each 16 lanes of
// a group are a thread of their own.  A million vertices, 64 lanes, 22 levels:
// 790 us with one store per value, 765 so (int8 rows 789 and 743).
__device__ void emit_deep_rows(const TraversalParams& P, long long tid, long long nthreads) {
    const unsigned long long* const vn = reinterpret_cast<const unsigned long long*>(P.lane_vn);
    const unsigned groups = (unsigned)(P.n >> 2), parts = (unsigned)(P.nlanes + 15) / 16;
    const bool spread = groups < nthreads;
    const unsigned items = spread ? groups * parts : groups;   // fewer than 2^30
    for (unsigned it = (unsigned)tid; it < items; it += (unsigned)nthreads) {
        const unsigned p0 = spread ? it / groups : 0u, p1 = spread ? p0 + 1u : parts;
        const long long c0 = 4ll * (it - (spread ? p0 * groups : 0u));
#pragma unroll 1
        for (unsigned part = p0; part < p1; ++part) {
            uint32_t vis[4], pl[4][4];   // pl: planes 2k (low half) and 2k + 1
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const long long v = P.old2new ? __ldg(P.old2new + c0 + j) : c0 + j;
                vis[j] = reinterpret_cast<const uint16_t*>(vn + 2 * v)[part];
                const uint16_t* const row = reinterpret_cast<const uint16_t*>(level_planes(P, v)) + part;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    pl[j][k] = vis[j] != 0u ? (uint32_t)row[8 * k] | (uint32_t)row[8 * k + 4] << 16 : 0u;
            }
#pragma unroll 1
            for (int q = 0; q < 4 && 16 * (int)part + 4 * q < P.nlanes; ++q) {
                uint32_t b[4], row[4];   // levels, 0xff (no level here) where unreached
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    b[j] = ~(spread4(vis[j], q) * 0xffu);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        b[j] |= spread4(pl[j][k], q) << (2 * k) | spread4(pl[j][k], q + 4) << (2 * k + 1);
                }
                transpose4(b, row);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int lane_idx = 16 * (int)part + 4 * q + i;
                    if (lane_idx >= P.nlanes) break;
                    const long long idx = (long long)lane_idx * P.n + c0;
                    if (P.dist_int8)
                        *reinterpret_cast<uint32_t*>(reinterpret_cast<int8_t*>(P.dist) + idx) = row[i];
                    else
                        *reinterpret_cast<int4*>(P.dist + idx) =
                            make_int4(level_or_none(row[i]), level_or_none(row[i] >> 8),
                                      level_or_none(row[i] >> 16), level_or_none(row[i] >> 24));
                }
            }
        }
    }
}

// After the last level: dist rows in the caller's numbering, unreached lanes
// -1, from the level planes.  `top`: no level is above it.  Four consecutive
// caller vertices per thread: their levels of four lanes are spread to bytes,
// transposed, and each lane row gets one 16-byte (int32) or 4-byte (int8)
// store covering all four vertices, when the row starts keep that alignment
// (n a multiple of 4, dist 16-byte aligned) and no level is above 254;
// otherwise one vertex per thread and one store per value.
__device__ void emit_batch(const TraversalParams& P, int top, long long tid, long long nthreads) {
    const unsigned long long* const vn = reinterpret_cast<const unsigned long long*>(P.lane_vn);
    const bool wide = (P.n & 3) == 0 && ((uintptr_t)P.dist & 15) == 0;
    if (wide && top >= 16 && top < 255) {
        emit_deep_rows(P, tid, nthreads);
        return;
    }
    if (wide && top < 16) {
        const long long groups = P.n >> 2;
        for (long long g = tid; g < groups; g += nthreads) {
            const long long c0 = g << 2;
            uint64_t vis[4];
            ulonglong2 lo[4], hi[4];   // planes 0, 1 and 2, 3
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const long long v = P.old2new ? __ldg(P.old2new + c0 + j) : c0 + j;
                vis[j] = __ldcg(vn + 2 * v);
                lo[j] = hi[j] = make_ulonglong2(0ull, 0ull);
                if (vis[j] != 0ull) {
                    lo[j] = __ldcg(level_planes(P, v));
                    hi[j] = __ldcg(level_planes(P, v) + 1);
                }
            }
#pragma unroll 1
            for (int q = 0; 4 * q < P.nlanes; ++q) {
                uint32_t b[4];   // of vertex j: the four lanes' levels, 0xff unreached
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    b[j] = (spread4(lo[j].x, q) | spread4(lo[j].y, q) << 1 | spread4(hi[j].x, q) << 2 |
                            spread4(hi[j].y, q) << 3) |
                           ~(spread4(vis[j], q) * 0xffu);
                uint32_t row[4];
                transpose4(b, row);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (4 * q + i >= P.nlanes) break;
                    const long long idx = (long long)(4 * q + i) * P.n + c0;
                    if (P.dist_int8)
                        *reinterpret_cast<uint32_t*>(reinterpret_cast<int8_t*>(P.dist) + idx) = row[i];
                    else
                        *reinterpret_cast<int4*>(P.dist + idx) =
                            make_int4(signed_byte<0>(row[i]), signed_byte<1>(row[i]),
                                      signed_byte<2>(row[i]), signed_byte<3>(row[i]));
                }
            }
        }
        return;
    }
    if (top < 16) {
        for (long long c = tid; c < P.n; c += nthreads) {
            const long long v = P.old2new ? __ldg(P.old2new + c) : c;
            const uint64_t vis = __ldcg(vn + 2 * v);
            ulonglong2 lo = make_ulonglong2(0ull, 0ull), hi = lo;
            if (vis != 0ull) {
                lo = __ldcg(level_planes(P, v));
                hi = __ldcg(level_planes(P, v) + 1);
            }
#pragma unroll 1
            for (int q = 0; 4 * q < P.nlanes; ++q) {
                uint32_t b = (spread4(lo.x, q) | spread4(lo.y, q) << 1 | spread4(hi.x, q) << 2 |
                              spread4(hi.y, q) << 3) |
                             ~(spread4(vis, q) * 0xffu);
#pragma unroll
                for (int i = 0; i < 4; ++i, b >>= 8) {
                    if (4 * q + i >= P.nlanes) break;
                    const long long idx = (long long)(4 * q + i) * P.n + c;
                    if (P.dist_int8) reinterpret_cast<int8_t*>(P.dist)[idx] = (int8_t)b;
                    else P.dist[idx] = signed_byte<0>(b);
                }
            }
        }
        return;
    }
    for (long long c = tid; c < P.n; c += nthreads) {
        const long long v = P.old2new ? __ldg(P.old2new + c) : c;
        const uint64_t vis = __ldcg(vn + 2 * v);
        ulonglong2 p[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            p[k] = vis != 0ull ? __ldcg(level_planes(P, v) + k) : make_ulonglong2(0ull, 0ull);
#pragma unroll 1
        for (int q = 0; 4 * q < P.nlanes; ++q) {
            uint32_t b = 0u, hit = spread4(vis, q);   // four lanes' levels, and which are reached
#pragma unroll
            for (int k = 0; k < 4; ++k)
                b |= spread4(p[k].x, q) << (2 * k) | spread4(p[k].y, q) << (2 * k + 1);
#pragma unroll
            for (int i = 0; i < 4; ++i, b >>= 8, hit >>= 8) {
                if (4 * q + i >= P.nlanes) break;
                const int lvl = (int)(b & 0xffu);
                if ((hit & 1u) && lvl == 255) continue;  // deep level, already written
                const int val = hit & 1u ? lvl : -1;
                const long long idx = (long long)(4 * q + i) * P.n + c;
                if (P.dist_int8) reinterpret_cast<int8_t*>(P.dist)[idx] = (int8_t)val;
                else P.dist[idx] = val;
            }
        }
    }
}

// One warp seeds all roots: duplicates share one queue entry whose mask
// holds every lane with that root.
__device__ void seed_batch(const TraversalParams& P, Stage<true>& S) {
    if (blockIdx.x != 0 || threadIdx.x >= 32) return;
    const unsigned lane = lane_id();
    for (int base = 0; base < P.nlanes; base += 32) {
        const int i = base + (int)lane;
        bool first = false;
        int32_t r = 0;
        uint64_t mask = 0ull;
        if (i < P.nlanes) {
            const int32_t cr = P.roots[i];
            first = true;
            for (int j = 0; j < P.nlanes; ++j) {
                if (P.roots[j] == cr) {
                    mask |= 1ull << j;
                    if (j < i) first = false;
                }
            }
            r = P.old2new ? __ldg(P.old2new + cr) : cr;
            if (first) {
#pragma unroll
                for (int p = 0; p < 4; ++p) level_planes(P, r)[p] = make_ulonglong2(0ull, 0ull);
                P.lane_vn[2 * (long long)r] = mask;
                if (P.dir_mode != 0) P.lane_front[r] = mask;
            }
        }
        stage_push<true>(P, S, first, r, 0, mask, -1, 0, 0);
    }
    stage_flush<true>(P, S, -1, 0, 0);
    if (lane == 0) {
        P.ctl[0].front_lanes = P.nlanes >= 64 ? ~0ull : ((1ull << P.nlanes) - 1ull);
        P.stats->reached = P.nlanes;
        P.stats->edges = (long long)S.edges;
        P.stats->levels = 1;
        S.edges = 0ull;
    }
    __syncwarp();
}

// Entries from which a batched level counts as large for its sweep.
constexpr long long kManyEntries = 1ll << 20;

// What a sweep needs to know of the level and adds up over the CTA.
struct SweepShared {
    int track, many;          // see open_sweep; the level expands many entries
    int publish;              // the next level needs to know which lanes have a frontier
    int plain;                // none of these
    uint64_t live;
    unsigned long long full, front, pairs, edges;
    unsigned count, clear;
};

__device__ __forceinline__ uint64_t lanes_of(const TraversalParams& P) {
    return P.nlanes >= 64 ? ~0ull : ((1ull << P.nlanes) - 1ull);
}

// Thread 0, while the level's frontier is being expanded (its counters are
// final).  Vertices that every live lane has reached are looked for (see
// batch_filters) once the frontier holds a 64th of all (vertex, lane) pairs:
// hardly any can be complete before, and the sweeps of small frontiers are
// spared the ballots.  A lane without a frontier now has none later: only the
// others count.  Which lanes those are is asked for (two warp reductions and
// one atomic per warp that found something) when the entries per frontier
// vertex would bring the next frontier to that size; where it was not, every
// lane counts as live.
__device__ __forceinline__ void open_sweep(const TraversalParams& P, SweepShared& X,
                                           unsigned long long front_lanes,
                                           unsigned long long pairs, long long vertices,
                                           long long entries, bool many) {
    X.track = 0;
    X.publish = P.dir_mode != 0;
    X.live = front_lanes != 0ull ? front_lanes : lanes_of(P);
    if (P.full != nullptr) {
        const float all = (float)P.sweep_limit * (float)P.nlanes;
        const float now = 64.f * (float)max(pairs, (unsigned long long)P.nlanes);
        X.track = now >= all;
        X.publish = now * (float)entries >= all * (float)vertices;
    }
    X.many = many;
    X.plain = !X.track && !many && (P.dir_mode != 0 || !X.publish);
    X.full = X.front = X.pairs = X.edges = 0ull;
    X.count = X.clear = 0u;
}
// The same in a launch of its own (host- and graph-driven loops).
__device__ __forceinline__ void open_sweep(const TraversalParams& P, SweepShared& X, int level) {
    if (threadIdx.x == 0) {
        const LevelCtl& C = P.ctl[level % 3];
        long long vertices = 0, entries = 0;
#pragma unroll
        for (int b = 0; b < kBins; ++b) {
            const unsigned long long p = ld_cg_u64(&C.packed[b]);
            vertices += (long long)(p >> kCountShift);
            entries += (long long)(p & kEdgeMask);
        }
        open_sweep(P, X, ld_cg_u64(&C.front_lanes), ld_cg_u64(&C.new_lanes), vertices, entries,
                   entries >= kManyEntries);
    }
    __syncthreads();
}

// Phase B of a batched level: lanes that reached v for the first time get
// distance level + 1 and make v part of the next frontier with those lanes.
// Two forms: kPlain for levels that need none of tracking, publishing in a
// top-down run, counters per CTA and the clearing at level 16.  A small level's
// sweep is a few microseconds of mostly idle warps, and the code of those it
// would run through costs it 0.5 us (116 sweeps of a 60 x 60 mesh, 64 lanes:
// 718 us in one form, 645 in its own).
template <bool kPlain>
__device__ void sweep_batch_form(const TraversalParams& P, Stage<true>& S, SweepShared& X, int level,
                                 long long tid, long long nthreads) {
    const uint64_t live = kPlain ? 0ull : X.live;
    const bool track = !kPlain && X.track != 0;
    const bool publish = kPlain ? P.dir_mode != 0 : X.publish != 0;
    const bool clear_high = !kPlain && level + 1 == 16;
    const int nslot = (level + 1) % 3, nxt = (level + 1) & 1;
    const unsigned lane = lane_id();
    long long my_pairs = 0, my_full = 0;
    unsigned long long my_front = 0ull;  // lanes with a vertex in the next frontier
    // (level 16's sweep also clears planes of vertices that got nothing new)
    const bool skip_idle = !track && !clear_high;
    unsigned full_count = 0u, clear = 0u;
    const uint64_t all_lanes = lanes_of(P);
    // kSweepUnroll vertices per thread and pass, their lane-set pairs loaded
    // together; the trip count is the same for every thread (the stage push
    // is warp-collective).  Two in the plain form: half the code of four, and
    // enough for the few vertices that its graphs have per thread (64 lanes, 65 k
    // vertices with a path of 300: 3373 -> 3274 us; one: 5 lanes on a 300 x 300
    // mesh 7107 -> 7457).
    constexpr int kSweepUnroll = kPlain ? 2 : 4;
    const long long stride = nthreads * kSweepUnroll;
    const long long nround = (P.n + stride - 1) / stride * stride;
    ulonglong2* const pairs = reinterpret_cast<ulonglong2*>(P.lane_vn);
    for (long long v0 = tid; v0 < nround; v0 += stride) {
        ulonglong2 vnu[kSweepUnroll];
#pragma unroll
        for (int x = 0; x < kSweepUnroll; ++x) {
            const long long v = v0 + x * nthreads;
            vnu[x] = v < P.n ? __ldcg(pairs + v) : make_ulonglong2(0ull, 0ull);
        }
        // most warps of a small level's sweep have nothing new: the sweep is
        // issue-bound there, so they leave before the per-vertex work
        uint64_t any = 0ull;
#pragma unroll
        for (int x = 0; x < kSweepUnroll; ++x) any |= vnu[x].y;
        if (skip_idle && __ballot_sync(FULL_MASK, any != 0ull) == 0u) {
            if (P.dir_mode != 0) {
#pragma unroll
                for (int x = 0; x < kSweepUnroll; ++x)
                    if (v0 + x * nthreads < P.n) P.lane_front[v0 + x * nthreads] = 0ull;
            }
            continue;
        }
#pragma unroll
        for (int x = 0; x < kSweepUnroll; ++x) {
            const long long v = v0 + x * nthreads;
            uint64_t fresh = 0ull;
            bool reached_before = false;  // some lane had reached v at an earlier level
            bool full = v >= P.sweep_limit;
            if (v < P.n) {
                const ulonglong2 vn = vnu[x];
                full = full || (live & ~(vn.x | vn.y)) == 0ull;
                if (vn.y != 0ull) {
                    fresh = vn.y & ~vn.x;
                    reached_before = vn.x != 0ull;
                    pairs[v] = make_ulonglong2(vn.x | fresh, 0ull);
                    my_pairs += __popcll(fresh);
                    // bottom-up bookkeeping: edges of vertices every lane has now reached
                    if (P.dir_mode != 0 && fresh != 0ull && (vn.x | fresh) == all_lanes)
                        my_full += __ldg(P.off + v + 1) - __ldg(P.off + v);
                }
                if (P.dir_mode != 0) P.lane_front[v] = fresh;
                my_front |= fresh;
            }
            if (track) {
                const unsigned w = __ballot_sync(FULL_MASK, full);
                if (lane == 0 && v < P.sweep_limit) {
                    P.full[v >> 5] = w;
                    full_count += __popc(w);
                    if (w != FULL_MASK) clear = max(clear, 0xffffffffu - (unsigned)(v >> 5));
                }
            }
            if (clear_high && v < P.n && vnu[x].x != 0ull) {
                level_planes(P, v)[2] = make_ulonglong2(0ull, 0ull);
                level_planes(P, v)[3] = make_ulonglong2(0ull, 0ull);
            }
            // the new lanes' level: a first visit writes the planes, a later one
            // adds to those that the level's bits name
            if (fresh != 0ull) {
                const int lvl = level + 1 < 255 ? level + 1 : 255;
                ulonglong2* const planes = level_planes(P, v);
                ulonglong2 z[4];   // all reads before the first write: one round trip
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    z[p] = make_ulonglong2(0ull, 0ull);
                    if (reached_before && ((lvl >> (2 * p)) & 3) != 0) z[p] = __ldcg(planes + p);
                }
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const ulonglong2 y = plane_bits(lvl, p, fresh);
                    const bool write = reached_before ? ((lvl >> (2 * p)) & 3) != 0
                                                      : p < 2 || lvl >= 16;
                    if (write) planes[p] = make_ulonglong2(y.x | z[p].x, y.y | z[p].y);
                }
                if (level + 1 >= 255) {
                    // deep levels: the distance goes straight to the output
                    const int32_t cv = P.new2old ? __ldg(P.new2old + v) : (int32_t)v;
                    for (unsigned long long f = fresh; f != 0ull; f &= f - 1ull) {
                        const long long idx = (long long)(__ffsll((long long)f) - 1) * P.n + cv;
                        if (P.dist_int8) reinterpret_cast<int8_t*>(P.dist)[idx] = (int8_t)(level + 1);
                        else P.dist[idx] = level + 1;
                    }
                }
            }
            stage_push<true>(P, S, fresh != 0ull, (int32_t)(v < P.n ? v : 0), 0, fresh, level, nxt,
                             nslot);
        }
    }
    stage_flush<true>(P, S, level, nxt, nslot);
    my_pairs = warp_incl_scan(my_pairs);
    if (P.dir_mode != 0) my_full = warp_incl_scan(my_full);
    unsigned long long front = 0ull;
    if (publish) {
        const unsigned flo = __reduce_or_sync(FULL_MASK, (unsigned)my_front);
        const unsigned fhi = __reduce_or_sync(FULL_MASK, (unsigned)(my_front >> 32));
        front = ((unsigned long long)fhi << 32) | flo;
    }
    LevelCtl& N = P.ctl[nslot];
    unsigned long long* const reached = reinterpret_cast<unsigned long long*>(&P.stats->reached);
    unsigned long long* const edges = reinterpret_cast<unsigned long long*>(&P.stats->edges);
    unsigned long long* const full_edges = reinterpret_cast<unsigned long long*>(&P.stats->full_edges);
    if (kPlain || !X.many) {
        if (lane == 31) {
            if (my_pairs > 0) {
                atomicAdd(&N.new_lanes, (unsigned long long)my_pairs);
                atomicAdd(reached, (unsigned long long)my_pairs);
            }
            if (my_full > 0) atomicAdd(full_edges, (unsigned long long)my_full);
        }
        if (lane == 0) {
            if (front != 0ull) atomicOr(&N.front_lanes, front);
            if (full_count > 0u) atomicAdd(&N.full_count, full_count);
            if (clear > 0u) atomicMax(&N.clear_word, clear);
            if (S.edges != 0ull) atomicAdd(edges, S.edges);
            S.edges = 0ull;
        }
        __syncwarp();
        return;
    }
    // The counters all lie in two lines, and a line takes one reduction every
    // 2.3 ns.  After a large level every warp has some, which would cost 10 us
    // and more: they are added up per CTA first.  On smaller levels the extra
    // step's round trip costs more than it saves.
    if (lane == 31) {
        if (my_pairs > 0) atomicAdd(&X.pairs, (unsigned long long)my_pairs);
        if (my_full > 0) atomicAdd(&X.full, (unsigned long long)my_full);
    }
    if (lane == 0) {
        if (front != 0ull) atomicOr(&X.front, front);
        if (full_count > 0u) atomicAdd(&X.count, full_count);
        if (clear > 0u) atomicMax(&X.clear, clear);
        if (S.edges != 0ull) atomicAdd(&X.edges, S.edges);
        S.edges = 0ull;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (X.pairs > 0ull) {
            atomicAdd(&N.new_lanes, X.pairs);
            atomicAdd(reached, X.pairs);
        }
        if (X.edges > 0ull) atomicAdd(edges, X.edges);
        if (X.full > 0ull) atomicAdd(full_edges, X.full);
        if (X.front != 0ull) atomicOr(&N.front_lanes, X.front);
        if (X.count > 0u) atomicAdd(&N.full_count, X.count);
        if (X.clear > 0u) atomicMax(&N.clear_word, X.clear);
    }
}

__device__ __forceinline__ void sweep_batch(const TraversalParams& P, Stage<true>& S, SweepShared& X,
                                            int level, long long tid, long long nthreads) {
    if (X.plain && level + 1 != 16) sweep_batch_form<true>(P, S, X, level, tid, nthreads);
    else sweep_batch_form<false>(P, S, X, level, tid, nthreads);
}

__device__ void book_batch_level(const TraversalParams& P, int level) {
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    unsigned long long* z = reinterpret_cast<unsigned long long*>(P.ctl + (level + 2) % 3);
    for (int i = 0; i < (int)(sizeof(LevelCtl) / 8); ++i) z[i] = 0ull;
}

template <int MB>
__global__ void __launch_bounds__(kBlock, MB)
bfs_batch_persistent(const __grid_constant__ TraversalParams P) {
    __shared__ Stage<true> s_stage[kWarps];
    __shared__ SweepShared s_sweep;
    Stage<true>& S = s_stage[threadIdx.x >> 5];
    stage_init(S);
    const long long nthreads = (long long)gridDim.x * kBlock;
    const long long tid = (long long)blockIdx.x * kBlock + threadIdx.x;
    stamp(P, 0);
    init_batch(P, tid, nthreads);
    __shared__ unsigned long long epoch;
    if (threadIdx.x == 0) epoch = 0ull;
    if (grid_barrier(P, epoch)) {
        stamp(P, 1);
        seed_batch(P, S);
        if (grid_barrier(P, epoch)) {
            stamp(P, 2);
            bool prev_bu = false;
            int level = 0;
            for (;; ++level) {
                unsigned long long front_lanes = 0ull, pairs = 0ull;
                if (threadIdx.x == 0 && P.full != nullptr) {   // in flight with the counters of the shape
                    front_lanes = ld_cg_u64(&P.ctl[level % 3].front_lanes);
                    pairs = ld_cg_u64(&P.ctl[level % 3].new_lanes);
                }
                const LevelShape L = read_level(P, level);
                if (L.cnt[0] + L.cnt[1] + L.cnt[2] == 0) break;
                if (P.dist_int8 && level + 1 > 126) {
                    if (blockIdx.x == 0 && threadIdx.x == 0) raise_status(P, kDevDepth);
                    break;
                }
                book_batch_level(P, level);
                const int dir = batch_direction(P, L, prev_bu);
                if (dir == 2 && blockIdx.x == 0 && threadIdx.x == 0) P.stats->bu_levels += 1;
                if (threadIdx.x == 0)
                    open_sweep(P, s_sweep, front_lanes, pairs, L.cnt[0] + L.cnt[1] + L.cnt[2],
                               L.edges[0] + L.edges[1] + L.edges[2],
                               L.edges[0] + L.edges[1] + L.edges[2] >= kManyEntries);
                expand_level<true>(P, S, L, level, nullptr, dir);
                prev_bu = dir == 2;
                if (!grid_barrier(P, epoch)) break;
                stamp(P, 3 + 2 * level);
                sweep_batch(P, S, s_sweep, level, tid, nthreads);
                if (!grid_barrier(P, epoch)) break;
                stamp(P, 4 + 2 * level);
                if (blockIdx.x == 0 && threadIdx.x == 0) {
                    if (__ldcg(reinterpret_cast<const unsigned long long*>(
                            &P.ctl[(level + 1) % 3].new_lanes)) > 0ull)
                        P.stats->levels = level + 2;
                }
            }
            // every sweep is complete here (the loop exits right after a barrier
            // or before any expansion of an empty level)
            if (ld_volatile_i32(&P.stats->abort) == 0) emit_batch(P, level, tid, nthreads);
        }
    }
    kernel_exit(P);
}

template <int MB>
__global__ void __launch_bounds__(kBlock, MB)
bfs_batch_step(const __grid_constant__ TraversalParams P) {
    __shared__ Stage<true> s_stage[kWarps];
    __shared__ SweepShared s_sweep;
    Stage<true>& S = s_stage[threadIdx.x >> 5];
    stage_init(S);
    const long long nthreads = (long long)gridDim.x * kBlock;
    const long long tid = (long long)blockIdx.x * kBlock + threadIdx.x;
    if (P.phase == 0) {
        init_batch(P, tid, nthreads);
    } else if (P.phase == 1) {
        seed_batch(P, S);
    } else if (P.phase == 2) {
        const LevelShape L = read_level(P, P.level);
        if (L.cnt[0] + L.cnt[1] + L.cnt[2] == 0) return;
        book_batch_level(P, P.level);
        expand_level<true>(P, S, L, P.level, nullptr);
    } else if (P.phase == 3) {
        open_sweep(P, s_sweep, P.level);
        sweep_batch(P, S, s_sweep, P.level, tid, nthreads);
    } else if (P.phase == 4) {
        // the first level with an empty frontier: the host's, or the graph loop's
        emit_batch(P, P.graph_cond ? ld_volatile_i32(&P.stats->graph_level) : P.level, tid, nthreads);
    } else if (P.phase == 7) {
        // graph-captured loop body: expansion of the device's current level
        const int level = ld_volatile_i32(&P.stats->graph_level);
        const LevelShape L = read_level(P, level);
        if (L.cnt[0] + L.cnt[1] + L.cnt[2] == 0) return;
        book_batch_level(P, level);
        const int dir = batch_direction(P, L, ld_volatile_i32(&P.stats->graph_prev_bu) != 0);
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            P.stats->graph_dir = dir;
            if (dir == 2) P.stats->bu_levels += 1;
        }
        expand_level<true>(P, S, L, level, nullptr, dir);
    } else if (P.phase == 8) {
        const int level = ld_volatile_i32(&P.stats->graph_level);
        open_sweep(P, s_sweep, level);
        sweep_batch(P, S, s_sweep, level, tid, nthreads);
    } else if (P.phase == 9) {
        graph_advance_batch(P);
    }
}

// ------------------------------------------------------ upload helpers
// CSR validation: flags[0] |= 1 for a column out of range, |= 2 for a
// decreasing offset.
__global__ void csr_check_kernel(const int64_t* off, const int32_t* col, long long n, long long nnz,
                                 int* flags) {
    const long long nthreads = (long long)gridDim.x * blockDim.x;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    int bad = 0;
    for (long long e = tid; e < nnz; e += nthreads) {
        const int32_t c = col[e];
        if (c < 0 || (long long)c >= n) bad |= 1;
    }
    for (long long v = tid; v < n; v += nthreads)
        if (off[v + 1] < off[v]) bad |= 2;
    if (bad) atomicOr(flags, bad);
}

// Symmetry test for the bottom-up step: the multiset of edges (v, u) equals
// the multiset of reversed edges (u, v) exactly when every edge is stored in
// both directions.  Both multisets are summed through a 64-bit mixing hash
// (order independent, wrapping); unequal sums prove asymmetry, equal sums
// mean symmetric up to a 2^-64-scale collision chance.
__device__ __forceinline__ unsigned long long edge_hash(unsigned long long a, unsigned long long b) {
    unsigned long long z = (a << 32 | b) + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void symmetry_hash_kernel(const int64_t* off, const int32_t* col, long long n,
                                     unsigned long long* sums) {
    const long long nwarps = (long long)gridDim.x * (blockDim.x / 32);
    const int lane = threadIdx.x & 31;
    unsigned long long fwd = 0, rev = 0;
    for (long long v = (long long)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); v < n;
         v += nwarps) {
        const long long b = off[v], e = off[v + 1];
        for (long long k = b + lane; k < e; k += 32) {
            const unsigned long long u = (unsigned)col[k];
            fwd += edge_hash((unsigned long long)v, u);
            rev += edge_hash(u, (unsigned long long)v);
        }
    }
    atomicAdd(&sums[0], fwd);
    atomicAdd(&sums[1], rev);
}

// Degree histogram by bin: counts[b] vertices and edges[b] entries.
__global__ void degree_bins_kernel(const int64_t* off, long long n, int t_small, int t_large,
                                   unsigned long long* counts, unsigned long long* edges,
                                   unsigned long long* maxdeg) {
    __shared__ unsigned long long s_c[kBins], s_e[kBins], s_m;
    if (threadIdx.x < kBins) { s_c[threadIdx.x] = 0; s_e[threadIdx.x] = 0; }
    if (threadIdx.x == 0) s_m = 0;
    __syncthreads();
    const long long nthreads = (long long)gridDim.x * blockDim.x;
    unsigned long long c[kBins] = {0, 0, 0}, e[kBins] = {0, 0, 0}, m = 0;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += nthreads) {
        const long long d = off[v + 1] - off[v];
        if (d <= 0) continue;
        const int b = d < t_small ? 0 : (d < t_large ? 1 : 2);
        c[b] += 1;
        e[b] += (unsigned long long)d;
        m = d > (long long)m ? (unsigned long long)d : m;
    }
    for (int b = 0; b < kBins; ++b) {
        atomicAdd(&s_c[b], c[b]);
        atomicAdd(&s_e[b], e[b]);
    }
    atomicMax(&s_m, m);
    __syncthreads();
    if (threadIdx.x < kBins) {
        atomicAdd(&counts[threadIdx.x], s_c[threadIdx.x]);
        atomicAdd(&edges[threadIdx.x], s_e[threadIdx.x]);
    }
    if (threadIdx.x == 0) atomicMax(maxdeg, s_m);
}

// -------------------------------------------------------- host wrappers
// Kernels are instantiated for 2, 3 and 4 resident CTAs per SM (register
// cap 128, 80 or 64; batched kernels 2 and 3: at 4 their spills cost more
// than the extra warps gain); the graph's occupancy option picks one.
const void* plain_persistent_fn(int mb, bool staged) {
    if (staged)
        return mb >= 4 ? (const void*)bfs_plain_persistent<4, true>
             : mb == 3 ? (const void*)bfs_plain_persistent<3, true>
                       : (const void*)bfs_plain_persistent<2, true>;
    return mb >= 4 ? (const void*)bfs_plain_persistent<4, false>
         : mb == 3 ? (const void*)bfs_plain_persistent<3, false>
                   : (const void*)bfs_plain_persistent<2, false>;
}
const void* plain_step_fn(int mb, bool staged) {
    if (staged)
        return mb >= 4 ? (const void*)bfs_plain_step<4, true>
             : mb == 3 ? (const void*)bfs_plain_step<3, true> : (const void*)bfs_plain_step<2, true>;
    return mb >= 4 ? (const void*)bfs_plain_step<4, false>
         : mb == 3 ? (const void*)bfs_plain_step<3, false> : (const void*)bfs_plain_step<2, false>;
}
const void* batch_persistent_fn(int mb) {
    return mb >= 3 ? (const void*)bfs_batch_persistent<3> : (const void*)bfs_batch_persistent<2>;
}
const void* batch_step_fn(int mb) {
    return mb >= 3 ? (const void*)bfs_batch_step<3> : (const void*)bfs_batch_step<2>;
}

// int8 rows from int32 distances, 16 per thread and step (16-byte loads and
// stores when both arrays are 16-byte aligned, else one at a time).
__global__ void dist_to_int8_kernel(const int32_t* __restrict__ src, int8_t* __restrict__ dst,
                                    long long count, DevStats* stats, bool vec) {
    const long long nthreads = (long long)gridDim.x * blockDim.x;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long n16 = vec ? count / 16 : 0;   // 16-byte accesses need aligned ends
    bool deep = false;
    for (long long i = tid; i < n16; i += nthreads) {
        const int4* s4 = reinterpret_cast<const int4*>(src + 16 * i);
        unsigned w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int4 x = __ldcs(s4 + k);
            const int v[4] = {x.x, x.y, x.z, x.w};
            unsigned b = 0;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                int y = v[c];
                if (y > 126) { deep = true; y = -2; }
                b |= (unsigned)(uint8_t)(int8_t)y << (8 * c);
            }
            w[k] = b;
        }
        reinterpret_cast<uint4*>(dst)[i] = make_uint4(w[0], w[1], w[2], w[3]);
    }
    for (long long i = 16 * n16 + tid; i < count; i += nthreads) {
        int y = src[i];
        if (y > 126) { deep = true; y = -2; }
        dst[i] = (int8_t)y;
    }
    if (deep && stats) atomicCAS(&stats->status, 0, (int)kDevDepth);
}

cudaError_t launch_dist_to_int8(const int32_t* src, int8_t* dst, long long count, DevStats* stats,
                                int sms, cudaStream_t s) {
    const bool vec = ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15u) == 0;
    dist_to_int8_kernel<<<sms * 4, 256, 0, s>>>(src, dst, count, stats, vec);
    return cudaGetLastError();
}

cudaError_t launch_csr_check(const int64_t* off, const int32_t* col, long long n, long long nnz,
                             int* flags, int sms, cudaStream_t s) {
    csr_check_kernel<<<sms * 4, 512, 0, s>>>(off, col, n, nnz, flags);
    return cudaGetLastError();
}

cudaError_t launch_symmetry_hash(const int64_t* off, const int32_t* col, long long n,
                                 unsigned long long* sums, int sms, cudaStream_t s) {
    symmetry_hash_kernel<<<sms * 4, 256, 0, s>>>(off, col, n, sums);
    return cudaGetLastError();
}

cudaError_t launch_degree_bins(const int64_t* off, long long n, int t_small, int t_large,
                               unsigned long long* counts, unsigned long long* edges,
                               unsigned long long* maxdeg, int sms, cudaStream_t s) {
    degree_bins_kernel<<<sms * 2, 512, 0, s>>>(off, n, t_small, t_large, counts, edges, maxdeg);
    return cudaGetLastError();
}

}  // namespace bfs
