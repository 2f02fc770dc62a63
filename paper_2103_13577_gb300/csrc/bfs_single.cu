// bfs_single.cu -- the default single-source traversal: one cooperative
// persistent launch, every level top-down (Algorithm 1 / Algorithm 2 Phase
// 1 with one compute node).
//
// A level runs in one of two ways, chosen by the entries its frontier
// holds:
//  * sparse: every probe round's candidates are staged, claimed, written
//    and queued by the warp that found them (bfs_device.cuh);
//  * dense: the expansion only marks -- a target whose visited bit is clear
//    gets the bit set by a reduction whose result nobody waits for, and its
//    parent stored -- and, after a grid barrier, a sweep over the bitmap
//    writes the distances of the vertices marked since the previous level
//    and queues them.
// The kernel has a form without dense levels for graphs that cannot have one
// (may_run_dense) and for bfs_run_static.  Runs that ask for direction-optimizing
// levels, bitmap-order levels or one of the tuning options use bfs_kernels.cu.
#define BFS_LEAN_PATHS 1
#include "bfs_device.cuh"

namespace bfs {

namespace {

// ---------------------------------------------------------- row gathering
// A warp's rows (one column segment [a, b) per lane) laid end to end, and
// which row an entry of that sequence belongs to.  The non-empty segments
// are compacted into shared memory; each round every lane whose segment
// starts inside the round's 32-slot window sets one bit of a warp-wide word
// (redux.or), and the owner of slot l is the number of starts at or before
// it -- a popcount and one shared-memory read where a shuffle binary search
// took five dependent steps and six more shuffles for the segment's fields.
struct __align__(16) Segment {
    long long cb;   // column index minus the sequence position (in entries)
    int lo, hi;     // units only: valid entries, as positions of the sequence
};

struct WarpSegments {
    Segment s[32];
    int32_t v[32];   // the rows' vertices
};

__device__ __forceinline__ unsigned lanemask_le() {
    unsigned m;
    asm volatile("mov.u32 %0, %%lanemask_le;" : "=r"(m));
    return m;
}

// Lanes whose value d lies in [0, 32) set bit d.
__device__ __forceinline__ unsigned start_bits(bool live, int d) {
    return __reduce_or_sync(FULL_MASK, (live && (unsigned)d < 32u) ? 1u << d : 0u);
}

// Long rows: 16-byte units (4 columns, the first rounded down to a 16-byte
// boundary), two per lane and round, one 128-bit load each.
template <class Visit>
__device__ __forceinline__ void gather_units(const int32_t* col, WarpSegments& W, long long a,
                                             long long b, int32_t v, Visit&& visit) {
    const unsigned lane = lane_id();
    const bool live = b > a;
    const unsigned ne = __ballot_sync(FULL_MASK, live);
    if (ne == 0u) return;
    const long long a4 = a & ~3ll;
    const int units = live ? (int)((b - a4 + 3) >> 2) : 0;
    const int incl = warp_incl_scan(units);
    const int excl = incl - units;
    const int total = __shfl_sync(FULL_MASK, incl, 31);
    __syncwarp();
    if (live) {
        const int k = __popc(ne & lanemask_lt());
        W.s[k].cb = a4 - 4ll * excl;
        W.s[k].lo = (int)(a - a4) + 4 * excl;
        W.s[k].hi = (int)(b - a4) + 4 * excl;
        W.v[k] = v;
    }
    __syncwarp();
    int before = -1;  // segments that start before the round, minus one
    for (int q0 = 0; q0 < total; q0 += 64) {
        int32_t u[8];
        unsigned okm = 0u;
        int32_t v2[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const unsigned m = start_bits(live, excl - (q0 + 32 * h));
            const int o = before + __popc(m & lanemask_le());
            before += __popc(m);
            const int q = q0 + 32 * h + (int)lane;
            const Segment s = W.s[o];
            int4 x = make_int4(0, 0, 0, 0);
            if (q < total) x = __ldcs(reinterpret_cast<const int4*>(col + s.cb + 4ll * q));
            const int c0 = min(max(s.lo - 4 * q, 0), 4), c1 = min(max(s.hi - 4 * q, 0), 4);
            okm |= (((1u << c1) - 1u) & ~((1u << c0) - 1u)) << (4 * h);
            u[4 * h + 0] = x.x;
            u[4 * h + 1] = x.y;
            u[4 * h + 2] = x.z;
            u[4 * h + 3] = x.w;
            v2[h] = W.v[o];
        }
        visit(okm, u, [&](int j) { return v2[j / 4]; });
    }
}

// Light rows: single columns, 256 entries per round.
template <class Visit>
__device__ __forceinline__ void gather_entries(const int32_t* col, WarpSegments& W, long long a,
                                               int deg, int32_t v, Visit&& visit) {
    const unsigned lane = lane_id();
    const bool live = deg > 0;
    const unsigned ne = __ballot_sync(FULL_MASK, live);
    if (ne == 0u) return;
    const int incl = warp_incl_scan(deg);
    const int excl = incl - deg;
    const int total = __shfl_sync(FULL_MASK, incl, 31);
    __syncwarp();
    if (live) {
        const int k = __popc(ne & lanemask_lt());
        W.s[k].cb = a - excl;
        W.v[k] = v;
    }
    __syncwarp();
    int before = -1;
    for (int e0 = 0; e0 < total; e0 += 256) {
        int32_t u[8];
        unsigned okm = 0u;
        unsigned own[2] = {0u, 0u};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            u[j] = 0;
            if (e0 + 32 * j < total) {  // the same for the whole warp
                const unsigned m = start_bits(live, excl - (e0 + 32 * j));
                const int o = before + __popc(m & lanemask_le());
                before += __popc(m);
                const int e = e0 + 32 * j + (int)lane;
                own[j / 4] |= (unsigned)o << (8 * (j % 4));
                if (e < total) {
                    okm |= 1u << j;
                    u[j] = __ldcs(col + W.s[o].cb + e);
                }
            }
        }
        // the entries' rows by number, one byte each, instead of 8 registers
        visit(okm, u, [&](int j) { return W.v[(own[j / 4] >> (8 * (j % 4))) & 0xffu]; });
    }
}

// ------------------------------------------------------------- work items
// Bins 1 and 2 are cut into equal runs of 2^shift entries, one per warp item
// (bin 2 rows span many items); bin 0 into groups of 32 rows.  Warp 0 of each
// CTA works a level's shape out once, in shared memory: done by every warp,
// its arithmetic was a fixed cost of 2 us per level (an almost empty level of
// a scale-22 traversal: 7.7 -> 5.2 us).
struct RunBin {               // bins 1 and 2
    const int32_t* chunk;
    const int64_t* eoff;
    const int32_t* v;
    int cnt, n;               // queue entries, runs
    int sh, down;             // log2 of a run's entries; chunk = run >> down
};

struct Level {
    LevelShape shape;         // of a sparse level
    RunBin bin[2];
    const int32_t* v0;        // bin 0
    int cnt0, n0;             // its queue entries, groups of 32
    int nonempty, dense, parts;
    int sync, look;           // `queued` is behind; the prefix is worth looking for
    // the graph's arrays: kept here, not in registers across the loops
    const int64_t* off;
    const int32_t* col;
    const int32_t* name;      // dense levels that write parents: the caller's numbers
    const uint16_t* cut;      // entries at the front of each row that lead to visited vertices
                              // (nullptr: unknown)
    long long edges;          // entries of its rows
    // carried from level to level
    long long prefix;         // vertices [0, prefix) are all visited
    unsigned long long reached, edges_seen;
};

// Runs of a bin whose chunk-start table has one slot per 2^chunk_shift
// entries.  A run starts at the entry its chunk's slot names and skips the
// rows that end before it, so a run is at least 1/32 of a chunk.
__device__ __forceinline__ long long bin_items(const BinQueue& Q, long long edges, int chunk_shift,
                                               int& sh) {
    sh = max(sh, chunk_shift - 5);
    const long long chunks =
        min((edges + (1ll << chunk_shift) - 1) >> chunk_shift, (long long)Q.chunk_cap);
    const long long runs = (edges + (1ll << sh) - 1) >> sh;
    const long long most = sh <= chunk_shift ? chunks << (chunk_shift - sh)
                                             : (chunks + (1ll << (sh - chunk_shift)) - 1) >>
                                                   (sh - chunk_shift);
    return min(runs, most);
}

// A dense level of a graph with hubs that are still unvisited runs in two
// parts: the first sixteenth of its items reaches nearly every heavy vertex,
// so the rows of the rest skip the entries that lead to them -- more than
// half of all entries when the degrees are skewed.
constexpr int kFirstPart = 4;                     // part 0 ends at n / 16
constexpr int kHubClass = 1;                      // hubs: degree >= 256

// Warp 0: vertices [0, prefix) are visited.
__device__ __forceinline__ void set_prefix(const TraversalParams& P, Level& L, long long prefix) {
    const int lane = (int)lane_id();
    const long long bound = lane < kCutClasses ? P.cut_bound[lane < kCutClasses ? lane : 0] : 0;
    const unsigned m =
        __ballot_sync(FULL_MASK, P.cut != nullptr && bound > 0 && bound <= prefix);
    if (lane == 0) {
        L.prefix = prefix;
        L.cut = m != 0u ? P.cut + (31 - __clz(m)) * P.n : nullptr;
    }
}

// The whole CTA: how many vertices from the front of the order are visited
// (at least `known`; looks 32 K vertices at a time, at most 512 K).
__device__ long long visited_prefix(const TraversalParams& P, long long known) {
    constexpr int kStep = 4 * kBlock;             // words per step
    __shared__ unsigned s_first;
    if (threadIdx.x == 0) s_first = 0xffffffffu;
    __syncthreads();
    const long long words = (P.sweep_limit + 31) / 32;
    long long w0 = known / 32 / kStep * kStep;
    for (int step = 0; step < 16 && w0 < words; ++step, w0 += kStep) {
        const long long w = w0 + 4 * threadIdx.x;
        if (w < words) {   // the bitmap is padded: 16-byte reads stay inside
            const uint4 x = __ldcg(reinterpret_cast<const uint4*>(P.visited + w));
            const uint32_t y[4] = {x.x, x.y, x.z, x.w};
            for (int k = 3; k >= 0; --k)
                if (y[k] != 0xffffffffu) atomicMin(&s_first, (unsigned)(w + k));
        }
        __syncthreads();
        if (s_first != 0xffffffffu) return min(32ll * s_first, P.sweep_limit);
        __syncthreads();
    }
    return min(32 * w0, P.sweep_limit);
}

// The whole CTA: brings the level's prefix and row cuts up to date.
__device__ __forceinline__ void refresh_prefix(const TraversalParams& P, Level& L) {
    const long long prefix = visited_prefix(P, L.prefix);
    __syncthreads();
    if (threadIdx.x < 32) set_prefix(P, L, prefix);
    __syncthreads();
}

// Warp 0: shape of the level about to be expanded, lane b working out bin b
// (as one thread's serial code it took 3 us of every level); block 0 books it.
template <bool kDense>
__device__ __forceinline__ void open_level(const TraversalParams& P, Level& L, int level) {
    const int lane = (int)lane_id();
    const int slot = level % 3, cur = level & 1;
    const int b = lane < kBins ? lane : 0;
    const unsigned long long p = ld_cg_u64(&P.ctl[slot].packed[b]);
    const unsigned discovered = __ldcg(&P.ctl[slot].discovered);
    const unsigned clear = kDense ? __ldcg(&P.ctl[slot].clear_word) : 0u;
    const BinQueue& Q = P.q[cur][b];
    // clamped so that a recorded overflow cannot turn into a bad read
    const int cnt = (int)min((long long)(p >> kCountShift), (long long)Q.cap);
    const long long edges = (long long)(p & kEdgeMask);
    const long long E1 = __shfl_sync(FULL_MASK, edges, 1), E2 = __shfl_sync(FULL_MASK, edges, 2);
    const long long E = __shfl_sync(FULL_MASK, edges, 0) + E1 + E2;
    const long long n = (long long)__shfl_sync(FULL_MASK, cnt, 0) + __shfl_sync(FULL_MASK, cnt, 1) +
                        __shfl_sync(FULL_MASK, cnt, 2);
    const int fit = (63 - __clzll(E1 + E2 + 1)) - (31 - __clz(gridDim.x * kWarps));
    const unsigned long long reached = L.reached + discovered;
    // Dense pays from 8 M entries on; from 1 M on where the targets are spread (no
    // hubs) or a quarter of the vertices is reached, so that most entries lead
    // nowhere new, and the rows' class counts are kept, so that they skip them.
    // (Without the counts, as in a caller's arena, the lower limit took the skewed
    // graph of 262 k vertices from 108 to 120 us and a uniform one of a million
    // from 261 to 240: left out.)  Below that, and on a skewed graph's early
    // levels, the marks crowd into the few bitmap lines of the hubs (a reduction
    // takes ~2.3 ns of its 128-byte line's time) and the extra barrier and sweep
    // are not won back: 200 k vertices, 4.5 M entries: sparse 42 us, dense 56; a
    // million vertices, 6.1 M entries: 70 and 75; 18 M: 89 and 88; scale 22, 67 M:
    // 190 and 180.  With most vertices reached 13 M entries take 50 and 37 us;
    // uniform, 20 M entries: 121 and 100.
    const bool hubs = P.cut != nullptr && P.cut_bound[kHubClass] > 0;
    const bool late = 4 * (long long)reached > P.sweep_limit;
    const bool dense = kDense && (E >= P.dense_min ||
                                  (8 * E >= P.dense_min && P.cut != nullptr && (!hubs || late)));
    // Dense levels: runs of 32 to 2048 entries, two to eight per warp, so that
    // the last round of the static deal leaves few warps idle, but 512
    // entries as soon as two such runs per warp can be had.
    const int run_shift = max(min(max(fit - 2, 5), 11), min(fit - 1, 9));
    if (kDense && lane < kBins) {
        if (lane == 0) {
            L.v0 = Q.v;
            L.cnt0 = cnt;
            L.n0 = (cnt + 31) / 32;
        } else {
            RunBin& R = L.bin[lane - 1];
            const int chunk_shift = __ffs(lane == 1 ? P.chunk_warp : P.chunk_cta) - 1;
            int sh = run_shift;
            R.n = (int)bin_items(Q, edges, chunk_shift, sh);
            R.sh = sh;
            R.down = chunk_shift - sh;
            R.chunk = Q.chunk;
            R.eoff = Q.eoff;
            R.v = Q.v;
            R.cnt = cnt;
        }
    }
    if (lane == 31 && !dense) L.shape = read_level(P, level);
    const bool swept = kDense && L.dense != 0;   // the previous level's sweep looked at every word
    long long prefix = L.prefix;
    if (swept) prefix = clear == 0u ? P.sweep_limit : 32ll * (0xffffffffu - clear);
    __syncwarp();
    if (kDense) set_prefix(P, L, prefix);
    if (blockIdx.x == 0 && lane >= 8 && lane < 8 + (int)(sizeof(LevelCtl) / 8))
        // clear the slot that the level after next will fill
        reinterpret_cast<unsigned long long*>(P.ctl + (level + 2) % 3)[lane - 8] = 0ull;
    if (lane == 0) {
        L.nonempty = n > 0;
        L.reached = reached;
        L.edges = E;
        L.edges_seen += (unsigned long long)E;
        if (kDense) {
            L.dense = dense;
            L.sync = dense && !swept;
            L.look = dense && P.cut != nullptr && late && !swept;
            L.parts = dense && hubs && P.cut_bound[kHubClass] > prefix && !late ? 2 : 1;
        }
        if (blockIdx.x == 0) {
            if (discovered > 0) P.stats->levels = level + 1;
            P.stats->reached = (long long)L.reached;
            P.stats->edges = (long long)L.edges_seen;
        }
    }
}

// The rows of one item, one per lane: offsets as read, not yet used, so that
// the loads can be in flight while another item is visited.
struct RowRead {
    long long base, end;
    int skip;
};
__device__ __forceinline__ RowRead read_row(const Level& L, int32_t v) {
    RowRead r = {0, 0, 0};
    if (v >= 0) {
        r.base = __ldg(L.off + v);
        r.end = __ldg(L.off + v + 1);
        if (L.cut) r.skip = __ldg(L.cut + v);
    }
    return r;
}

// Expands runs [begin, end) of bin B with `visit(okm, u, row)` for every round
// of 8 entries per lane (bit j of okm: u[j] is an entry of vertex row(j)).
// Rows go by the caller's numbers when L.name is set.
//
// A row is found through three dependent reads (chunk start -> queue entry
// -> row offsets) before its columns can be asked for.  A warp reads the
// chunk starts of its next 32 runs at once, and while one run is visited the
// row offsets of the next and the queue entries of the one after are in
// flight.
template <class Visit>
__device__ __forceinline__ void expand_runs(const Level& L, WarpSegments& W, const RunBin& B, int warp_at,
                                            int begin, int end, Visit&& visit) {
    const int lane = (int)lane_id();
    const int nwarps = (int)gridDim.x * kWarps;
    int it = begin + warp_at;
    if (it >= end) return;
    auto starts_from = [&](int from) -> int {
        const int k = from + lane * nwarps;
        return k < end ? __ldcg(B.chunk + (B.down >= 0 ? (long long)k >> B.down
                                                       : (long long)k << -B.down))
                       : 0;
    };
    // this lane's entry of the batch that starts at queue entry i: its vertex
    // (-1: none) and where its row starts relative to the run
    auto entry = [&](int run, int i, int& rel) -> int32_t {
        rel = 0;
        if (run >= end || i + lane >= B.cnt) return -1;
        const long long d = __ldcg(B.eoff + i + lane) - ((long long)run << B.sh);
        const int32_t v = __ldcg(B.v + i + lane);
        rel = (int)max(d, -0x7fffffffll);
        return d < (1ll << B.sh) ? v : -1;
    };
    auto work = [&](int32_t v, int rel, const RowRead& r) {
        const int32_t x = L.name && v >= 0 ? __ldg(L.name + v) : v;
        const int len = 1 << B.sh;
        gather_units(L.col, W, r.base + max(-rel, r.skip), min(r.end, r.base + (len - rel)), x,
                     visit);
    };
    int starts = starts_from(it), k = 0;   // k: runs done of those in `starts`
    int i = -1, rel, rel1;                 // i: queue entry of the batch, -1 for a run's first
    int32_t v = entry(it, __shfl_sync(FULL_MASK, starts, 0), rel);
    int32_t v1 = entry(it + nwarps, __shfl_sync(FULL_MASK, starts, 1), rel1);
    RowRead r = read_row(L, v);
    for (;;) {
        RowRead r1;
        int32_t v2 = -1;
        int rel2 = 0;
        if (i < 0) {
            if (k == 30) {
                starts = starts_from(it);
                k = 0;
            }
            v2 = entry(it + 2 * nwarps, __shfl_sync(FULL_MASK, starts, k + 2), rel2);
            r1 = read_row(L, v1);
        }
        const bool full = __ballot_sync(FULL_MASK, v >= 0) == FULL_MASK;
        work(v, rel, r);
        if (full) {
            // more than 32 rows in the run: the next 32, without lookahead
            i = (i < 0 ? __shfl_sync(FULL_MASK, starts, k) : i) + 32;
            v = entry(it, i, rel);
            r = read_row(L, v);
            continue;
        }
        it += nwarps;
        if (it >= end) break;
        if (i < 0) {
            ++k;
            v = v1;
            rel = rel1;
            r = r1;
            v1 = v2;
            rel1 = rel2;
        } else {
            // what was read ahead went with the batches: start over
            i = -1;
            starts = starts_from(it);
            k = 0;
            v = entry(it, __shfl_sync(FULL_MASK, starts, 0), rel);
            v1 = entry(it + nwarps, __shfl_sync(FULL_MASK, starts, 1), rel1);
            r = read_row(L, v);
        }
    }
}

// Expands groups [begin, end) of 32 rows of bin 0, the next group's rows in
// flight while one is visited.
template <class Visit>
__device__ __forceinline__ void expand_groups(const Level& L, WarpSegments& W, int warp_at,
                                              int begin, int end,
                                              Visit&& visit) {
    const int lane = (int)lane_id();
    const int nwarps = (int)gridDim.x * kWarps;
    int it = begin + warp_at;
    if (it >= end) return;
    auto entry = [&](int g) -> int32_t {
        const int i = g * 32 + lane;
        return g < end && i < L.cnt0 ? __ldcg(L.v0 + i) : -1;
    };
    auto work = [&](int32_t v, const RowRead& r) {
        const int32_t x = L.name && v >= 0 ? __ldg(L.name + v) : v;
        gather_entries(L.col, W, r.base + r.skip, (int)(r.end - r.base) - r.skip, x, visit);
    };
    int32_t v = entry(it), v1 = entry(it + nwarps);
    RowRead r = read_row(L, v);
    for (; it < end; it += nwarps) {
        const int32_t v2 = entry(it + 2 * nwarps);
        const RowRead r1 = read_row(L, v1);
        work(v, r);
        v = v1;
        r = r1;
        v1 = v2;
    }
}

// One part of a level: its share of each bin's items, dealt round robin over
// all warps of the grid as one sequence.
template <class Visit>
__device__ __forceinline__ void expand_part(const Level& L, WarpSegments& W, int part,
                                            Visit&& visit) {
    const int nwarps = (int)gridDim.x * kWarps;
    int at = (int)blockIdx.x * kWarps + (int)(threadIdx.x >> 5);
    const int sh0 = part > 0 ? kFirstPart : 31;
    const int sh1 = part + 1 < L.parts ? kFirstPart : 0;
    for (int b = 0; b < 2; ++b) {
        const int begin = L.bin[b].n >> sh0, end = L.bin[b].n >> sh1;
        expand_runs(L, W, L.bin[b], at, begin, end, visit);
        at -= (end - begin) % nwarps;
        if (at < 0) at += nwarps;
    }
    expand_groups(L, W, at, L.n0 >> sh0, L.n0 >> sh1, visit);
}

// --------------------------------------------------------------- marking
// Dense levels: marks the targets whose visited bit is clear.  A plain
// (L1-cacheable) read can only show clear a bit that is set since, never the
// reverse, and marking a vertex again changes nothing: every row that marks
// it at this level is a valid parent.  (About one mark in six is such a
// repetition at scale 22.)
template <class Row>
__device__ __forceinline__ void mark_round(uint32_t* visited, int32_t* parent,
                                           const int32_t* new2old, unsigned okm,
                                           const int32_t (&u)[8], Row&& row) {
    uint32_t w[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = ((okm >> j) & 1u) ? visited[u[j] >> 5] : 0xffffffffu;
    unsigned cand = 0u;
#pragma unroll
    for (int j = 0; j < 8; ++j)
        if (!((w[j] >> (u[j] & 31)) & 1u)) cand |= 1u << j;
    if (__ballot_sync(FULL_MASK, cand != 0u) == 0u) return;
    int32_t cu[8];
    if (parent != nullptr) {
        // all the caller numbers before the first store: one round trip
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            cu[j] = u[j];
            if (new2old != nullptr && ((cand >> j) & 1u)) cu[j] = __ldg(new2old + u[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
        if ((cand >> j) & 1u) atomicOr(visited + (u[j] >> 5), 1u << (u[j] & 31));
    if (parent != nullptr) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if ((cand >> j) & 1u) parent[cu[j]] = row(j);
    }
}

// One part of a dense level's expansion.  What the loops use of P is read
// before their first store.
__device__ __forceinline__ void dense_part(const TraversalParams& P, WarpSegments& W, const Level& L,
                                        int part) {
    uint32_t* const visited = P.visited;
    int32_t* const parent = P.parent;
    const int32_t* const new2old = P.new2old;
    expand_part(L, W, part,
                      [&](unsigned okm, const int32_t(&u)[8], auto&& row) {
                          mark_round(visited, parent, new2old, okm, u, row);
                      });
}

// --------------------------------------------------------------- enqueue
constexpr int kPerThread = 8;
constexpr int kListMax = kPerThread * kBlock;    // vertices queued at a time

struct QueueShared {
    unsigned long long at[kBins][kWarps];  // per bin and warp: entries << 34 | degree sum, then
                                           // where the warp's entries start in the queue
};

// The whole CTA: writes the distances of the tile's new vertices (list[0,
// total) in shared memory: bitmap word of the tile << 5 | bit; word k of the
// tile is word tile + k * tiles of the bitmap) and appends them to the
// frontier queues of parity `par`, counted in slot `slot`.  Queue slots and
// edge ranges are reserved with one atomicAdd per bin.
__device__ __forceinline__ void enqueue_tile(const TraversalParams& P, QueueShared& X,
                                             const uint16_t* list, int total, long long tile,
                                             long long tiles, int slot, int par, int dist_value) {
    const unsigned lane = lane_id();
    const int warp = threadIdx.x >> 5;
    const int64_t* const off = P.off;
    const int32_t* const new2old = P.new2old;
    int32_t* const dist = P.dist;
    const int t_small = P.t_small, t_large = P.t_large;
    const int sh_warp = __ffs(P.chunk_warp) - 1, sh_cta = __ffs(P.chunk_cta) - 1;
    unsigned long long* const packed = P.ctl[slot].packed;
    bool overflow = false;
    const int per = (total + kBlock - 1) / kBlock;
    const int i0 = (int)threadIdx.x * per;
    int32_t u[kPerThread];
    int deg[kPerThread];
#pragma unroll
    for (int h = 0; h < kPerThread; ++h) {
        u[h] = -1;
        deg[h] = 0;
        if (h < per && i0 + h < total) {
            const int x = list[i0 + h];
            u[h] = (int32_t)((tile + (x >> 5) * tiles) * 32 + (x & 31));
            deg[h] = (int)(__ldg(off + u[h] + 1) - __ldg(off + u[h]));
        }
    }
    // per bin: this thread's entries << 34 | degree sum
    unsigned long long at[kBins] = {0ull, 0ull, 0ull}, incl[kBins];
#pragma unroll
    for (int h = 0; h < kPerThread; ++h) {
        if (u[h] < 0) continue;
        dist[new2old ? __ldg(new2old + u[h]) : u[h]] = dist_value;
        const unsigned long long x = (1ull << kCountShift) + (unsigned long long)deg[h];
        if (deg[h] > 0) {
            if (deg[h] < t_small) at[0] += x;
            else if (deg[h] < t_large) at[1] += x;
            else at[2] += x;
        }
    }
#pragma unroll
    for (int b = 0; b < kBins; ++b) {
        incl[b] = 0ull;
        if (__ballot_sync(FULL_MASK, at[b] != 0ull) != 0u) incl[b] = warp_incl_scan(at[b]);
        if (lane == 31) X.at[b][warp] = incl[b];
    }
    __syncthreads();
    if (warp == 0) {
        // lane = bin * 8 + warp: exclusive scan over the warps, and the
        // bin's slots and edge range from one atomicAdd
        const int b = (int)lane / kWarps, k = (int)lane % kWarps;
        const bool on = b < kBins;
        const unsigned long long x = on ? X.at[on ? b : 0][k] : 0ull;
        unsigned long long y = x;
#pragma unroll
        for (int d = 1; d < kWarps; d <<= 1) {
            const unsigned long long z = __shfl_up_sync(FULL_MASK, y, d);
            if (k >= d) y += z;
        }
        unsigned long long base = 0ull;
        if (on && k == kWarps - 1 && y != 0ull) base = atomicAdd(packed + b, y);
        base = __shfl_sync(FULL_MASK, base, (int)lane | (kWarps - 1));
        if (on) X.at[b][k] = base + y - x;
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < kBins; ++b) at[b] = X.at[b][warp] + incl[b] - at[b];
#pragma unroll
    for (int h = 0; h < kPerThread; ++h) {
        long long c0 = 0;
        int nc = 0;   // chunks whose first entry lies in this row
        int32_t pos = 0;
        const int b = deg[h] < t_small ? 0 : (deg[h] < t_large ? 1 : 2);
        if (deg[h] > 0) {
            const unsigned long long x = b == 0 ? at[0] : b == 1 ? at[1] : at[2];
            const unsigned long long next = x + (1ull << kCountShift) + (unsigned long long)deg[h];
            if (b == 0) at[0] = next;
            else if (b == 1) at[1] = next;
            else at[2] = next;
            const BinQueue& Q = P.q[par][b];
            pos = (int32_t)(x >> kCountShift);
            if (pos >= Q.cap) {
                overflow = true;
            } else {
                Q.v[pos] = u[h];
                if (b > 0) {
                    const long long eo = (long long)(x & kEdgeMask);
                    Q.eoff[pos] = eo;
                    const int cshift = b == 1 ? sh_warp : sh_cta;
                    c0 = (eo + (1ll << cshift) - 1) >> cshift;
                    const long long c_end = (eo + deg[h] - 1) >> cshift;
                    const long long last = Q.chunk_cap - 1;
                    if (c_end > last) overflow = true;
                    nc = (int)(min(c_end, last) - c0 + 1);
                }
            }
        }
        // chunk starts: each lane its own row's, a run of more than 32 by the
        // whole warp
        if (nc > 0 && nc <= 32) {
            int32_t* const qc = P.q[par][b].chunk + c0;
            for (int c = 0; c < nc; ++c) qc[c] = pos;
        }
        for (unsigned m = __ballot_sync(FULL_MASK, nc > 32); m != 0u; m &= m - 1u) {
            const int src = __ffs(m) - 1;
            const long long cc = __shfl_sync(FULL_MASK, c0, src);
            const int ncc = __shfl_sync(FULL_MASK, nc, src);
            const int32_t p = __shfl_sync(FULL_MASK, pos, src);
            int32_t* const qc = P.q[par][__shfl_sync(FULL_MASK, b, src)].chunk;
            for (int c = (int)lane; c < ncc; c += 32) qc[cc + c] = p;
        }
    }
    if (overflow) raise_status(P, kDevOverflow);
    __syncthreads();
}

// ----------------------------------------------------------------- sweep
constexpr int kPerWarp = 8;                      // bitmap words per warp
constexpr int kTileWords = kPerWarp * kWarps;
static_assert(kTileWords * 32 <= kListMax, "a tile's vertices fit in one list");

struct SweepShared {
    uint16_t list[kListMax];    // new vertices of the tile
    int warp_new[kWarps];
    QueueShared queue;
};

// After a dense level: every vertex whose visited bit was set during the level
// (it is not in `queued` yet) gets distance level + 1 and a place in the next
// frontier.  A CTA takes 64 bitmap words at a time, spread evenly over the
// bitmap: in degree order the heavy vertices, whose chunk-start runs are the
// longest, would otherwise all fall to a few CTAs (sweep of a scale-22
// traversal's level 2: 49 us with consecutive words, 40 spread).  A word's 32
// row offsets and caller numbers are read in order.  The first word with a
// vertex still unvisited bounds the prefix of the order that the next level's
// rows may skip.
__device__ void sweep_level(const TraversalParams& P, SweepShared& X, int level) {
    const unsigned lane = lane_id();
    const int warp = threadIdx.x >> 5;
    const int nslot = (level + 1) % 3, nxt = (level & 1) ^ 1;
    const long long words = (P.sweep_limit + 31) / 32;
    const long long tiles = (words + kTileWords - 1) / kTileWords;
    int found = 0;
    unsigned clear = 0u;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        uint32_t fresh = 0u;
        const long long w = t + (warp * kPerWarp + lane) * tiles;
        if (lane < kPerWarp && w < words) {
            const uint32_t now = __ldcg(P.visited + w), old = __ldcg(P.queued + w);
            fresh = now & ~old;
            if (fresh) P.queued[w] = now;
            const long long past = 32 * (w + 1) - P.sweep_limit;
            const uint32_t all = past > 0 ? 0xffffffffu >> past : 0xffffffffu;
            if ((now & all) != all) clear = max(clear, 0xffffffffu - (unsigned)w);
        }
        const int cnt = __popc(fresh);
        int incl = cnt;
#pragma unroll
        for (int d = 1; d < kPerWarp; d <<= 1) {
            const int y = __shfl_up_sync(FULL_MASK, incl, d);
            if (lane >= (unsigned)d) incl += y;
        }
        if (lane == kPerWarp - 1) X.warp_new[warp] = incl;
        __syncthreads();
        int before = 0, total = 0;
#pragma unroll
        for (int k = 0; k < kWarps; ++k) {
            const int x = X.warp_new[k];
            if (k < warp) before += x;
            total += x;
        }
#pragma unroll
        for (int k = 0; k < kPerWarp; ++k) {
            const uint32_t word = __shfl_sync(FULL_MASK, fresh, k);
            const int at = before + __shfl_sync(FULL_MASK, incl - cnt, k);
            if ((word >> lane) & 1u)
                X.list[at + __popc(word & lanemask_lt())] =
                    (uint16_t)((warp * kPerWarp + k) * 32 + lane);
        }
        __syncthreads();
        found += total;
        if (total > 0) enqueue_tile(P, X.queue, X.list, total, t, tiles, nslot, nxt, level + 1);
    }
    clear = __reduce_max_sync(FULL_MASK, clear);
    if (threadIdx.x == 0 && found > 0) atomicAdd(&P.ctl[nslot].discovered, (unsigned)found);
    if (lane == 0 && clear > 0u) atomicMax(&P.ctl[nslot].clear_word, clear);
}

// ------------------------------------------------------------------ init
// Clears the state with the root already marked, so that level 0 (its row,
// which every CTA finds by itself) needs no launch-wide step of its own.
__device__ void init_single(const TraversalParams& P, int32_t root, long long tid,
                            long long nthreads) {
    if (blockIdx.x == 0 && threadIdx.x < 3 * (int)(sizeof(LevelCtl) / 8))
        reinterpret_cast<unsigned long long*>(P.ctl)[threadIdx.x] = 0ull;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        P.stats->levels = 0;
        P.stats->reached = 0;
        P.stats->edges = 0;
        P.stats->status = 0;
        P.stats->max_level = 0;
        P.stats->bu_levels = 0;
    }
    fill_bytes(P.dist, P.n * 4, 0xff, tid, nthreads);
    if (P.parent) fill_bytes(P.parent, P.n * 4, 0xff, tid, nthreads);
    // the bitmap is 16-byte aligned and padded
    const long long quads = ((P.n + 31) / 32 + 3) / 4;
    for (long long i = tid; i < quads; i += nthreads) {
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        if (i == root >> 7) w[(root >> 5) & 3] = 1u << (root & 31);
        const uint4 x = make_uint4(w[0], w[1], w[2], w[3]);
        reinterpret_cast<uint4*>(P.visited)[i] = x;
    }
}

// Level 0: the entries of the root's row, in runs of 32 to 512 per warp.
__device__ __forceinline__ void expand_root(const TraversalParams& P, Stage<false>& S,
                                            const Level& L, int32_t root) {
    const int nwarps = (int)gridDim.x * kWarps;
    const long long base = __ldg(L.off + root), E = L.edges;
    const int sh = min(max((63 - __clzll(E + 1)) - (31 - __clz(nwarps)), 5), 9);
    for (long long cs = ((long long)blockIdx.x * kWarps + (threadIdx.x >> 5)) << sh; cs < E;
         cs += (long long)nwarps << sh)
        expand_segment<false>(P, S, base + cs, base + min(cs + (1ll << sh), E), root, 0ull, 0, 1, 1,
                              0, 256);
}

// One level's working memory, by the way it runs.
template <bool kDense>
struct LevelMemory {
    union {
        struct {
            Stage<false> stage[kWarps];
            WarpSegments seg[kWarps];
        } expand;
        SweepShared sweep;
    };
    __device__ LevelMemory() {}
};
template <>
struct LevelMemory<false> {
    struct {
        Stage<false> stage[kWarps];
    } expand;
};

// A dense level; false when a barrier was given up.
__device__ __forceinline__ bool dense_level(const TraversalParams& P, LevelMemory<true>& s, Level& L,
                                            int level, unsigned long long& epoch, long long tid,
                                            long long nthreads) {
    if (L.sync) {
        // the levels before ran sparse: take note of what they queued
        const long long quads = ((P.sweep_limit + 31) / 32 + 3) / 4;
        for (long long i = tid; i < quads; i += nthreads)
            reinterpret_cast<uint4*>(P.queued)[i] =
                __ldcg(reinterpret_cast<const uint4*>(P.visited) + i);
        if (!grid_barrier(P, epoch)) return false;
    }
    if (L.look) refresh_prefix(P, L);
    for (int part = 0; part < L.parts; ++part) {
        dense_part(P, s.expand.seg[threadIdx.x >> 5], L, part);
        if (!grid_barrier(P, epoch, true)) return false;
        if (part + 1 < L.parts) refresh_prefix(P, L);
    }
    sweep_level(P, s.sweep, level);
    return true;
}

}  // namespace

template <int MB, bool kDense>
__global__ void __launch_bounds__(kBlock, MB)
bfs_single_persistent(const __grid_constant__ TraversalParams P) {
    __shared__ LevelMemory<kDense> s;
    __shared__ unsigned long long epoch;
    __shared__ Level L;
    __shared__ int s_disc;
    Stage<false>& S = s.expand.stage[threadIdx.x >> 5];
    const long long nthreads = (long long)gridDim.x * kBlock;
    const long long tid = (long long)blockIdx.x * kBlock + threadIdx.x;
    // a failed validation launch (same stream, so its result is visible to
    // every CTA) ends the traversal before anything reads the graph
    if (P.pre_status && ld_volatile_i32(P.pre_status) != 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) raise_status(P, ld_volatile_i32(P.pre_status));
        kernel_exit(P);
        return;
    }
    stamp(P, 0);
    const int32_t root = P.old2new ? __ldg(P.old2new + P.root_caller) : P.root_caller;
    init_single(P, root, tid, nthreads);
    if (threadIdx.x == 0) {
        epoch = 0ull;
        s_disc = 0;
        L.off = P.off;
        L.col = P.col;
        L.name = P.parent != nullptr ? P.new2old : nullptr;
        L.cut = nullptr;
        L.prefix = 0;
        L.dense = 0;
        L.edges = __ldg(P.off + root + 1) - __ldg(P.off + root);
        L.reached = 1ull;
        L.edges_seen = (unsigned long long)L.edges;
    }
    if (grid_barrier(P, epoch)) {
        stamp(P, 1);
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            P.dist[P.root_caller] = 0;
            if (P.parent) P.parent[P.root_caller] = P.root_caller;
            P.stats->levels = 1;
            P.stats->reached = 1;
            P.stats->edges = L.edges;
            stamp(P, 2);
        }
        for (int level = 0;;) {
            if (level > 0) {
                if (threadIdx.x < 32) open_level<kDense>(P, L, level);
                if (threadIdx.x == 0) s_disc = 0;
                __syncthreads();
                if (!L.nonempty) break;
            }
            const int nslot = (level + 1) % 3, nxt = (level & 1) ^ 1;
            bool dense = false;
            if constexpr (kDense) {
                dense = L.dense != 0;
                if (dense && !dense_level(P, s, L, level, epoch, tid, nthreads)) break;
            }
            if (!dense) {
                stage_init(S);
                if (level == 0) expand_root(P, S, L, root);
                else expand_top_down<false>(P, S, L.shape, level);
                stage_flush<false>(P, S, level, nxt, nslot);
                if (lane_id() == 0 && S.disc > 0) atomicAdd(&s_disc, S.disc);
                __syncthreads();
                if (threadIdx.x == 0 && s_disc > 0)
                    atomicAdd(&P.ctl[nslot].discovered, (unsigned)s_disc);
            }
            if (!grid_barrier(P, epoch)) break;
            stamp(P, 3 + level);
            ++level;
        }
    }
    kernel_exit(P);
}

const void* single_persistent_fn(int mb, bool dense) {
    if (dense)
        return mb >= 4 ? (const void*)bfs_single_persistent<4, true>
             : mb == 3 ? (const void*)bfs_single_persistent<3, true>
                       : (const void*)bfs_single_persistent<2, true>;
    return mb >= 4 ? (const void*)bfs_single_persistent<4, false>
         : mb == 3 ? (const void*)bfs_single_persistent<3, false>
                   : (const void*)bfs_single_persistent<2, false>;
}

}  // namespace bfs
