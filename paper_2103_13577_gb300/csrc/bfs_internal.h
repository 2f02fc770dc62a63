// bfs_internal.h -- structures shared by the kernels and the host runtime.
#pragma once

#include <cstddef>
#include <cstdint>

namespace bfs {

constexpr int kBlock = 256;               // threads per CTA of every traversal kernel
constexpr int kWarps = kBlock / 32;
constexpr int kBins = 3;                  // 0: warp-gather, 1: warp-per-vertex, 2: CTA chunks
constexpr int kCountShift = 34;           // packed bin counter: (count << 34) | edges
constexpr unsigned long long kEdgeMask = (1ull << kCountShift) - 1ull;
constexpr int64_t kMaxVertices = (1ll << 30) - 1;    // count field holds 30 bits
constexpr int64_t kMaxEdges = (1ll << kCountShift) - 1;

// Device status codes (mirrors of BFS_ERR_* that the kernels can raise).
enum DevStatus : int { kDevOk = 0, kDevTimeout = 1, kDevOverflow = 2, kDevDepth = 3,
                       kDevInvalidGraph = 4 };

// One slot of the per-level control block; three slots rotate by level so
// that the slot being written (next frontier), the slot being read (current
// frontier) and the slot being cleared never coincide.
struct LevelCtl {
    unsigned long long packed[kBins];  // per bin: (entries << 34) | sum of degrees
    unsigned int work;                  // dynamic work-item counter of this level
    unsigned int discovered;            // vertices claimed at this level (any degree)
    unsigned long long new_lanes;       // batched: (vertex, lane) pairs discovered
    unsigned long long front_lanes;     // batched: lanes with a non-empty frontier
    unsigned int clear_word;            // 2^32 - 1 - first bitmap word with an unvisited vertex,
                                        // batched: with one some live lane lacks (0: none)
    unsigned int full_count;            // batched: vertices every live lane has reached
};

struct GridBarrier {
    unsigned long long arrived;   // arrivals since the launch began; bit 63: a CTA gave up
    unsigned int exited;          // CTAs that have left the launch
    unsigned int pad[29];
};

struct DevStats {
    long long levels;
    long long reached;
    long long edges;
    int status;       // sticky result of the launch (read by the host)
    int max_level;
    int abort;        // set with status; tells waiting CTAs to leave; cleared at kernel exit
    int bu_levels;    // levels run bottom-up
    int pad[2];
    // graph-captured level loop: the state the device-side loop keeps in
    // registers, carried between the loop body's launches
    long long graph_seen;  // edges of all frontiers so far
    int graph_level;       // level the next body launch expands
    int graph_prev_bu;     // the previous level ran bottom-up
    int graph_dir;         // direction of the level just expanded
    int graph_pad;
    long long full_edges;  // batched: degree sum of the vertices every lane has reached
};

// Frontier queue of one bin (one of two ping-pong copies).
struct BinQueue {
    int32_t* v;            // vertex (device numbering)
    int64_t* eoff;         // exclusive prefix of degrees inside the bin (bins 1, 2)
    int32_t* chunk;        // first entry of each edge chunk (bins 1, 2)
    uint64_t* mask;        // batched traversal: source-lane bitset of the entry
    int64_t cap;           // entries
    int64_t chunk_cap;     // chunk-start slots
};

// Rows of a degree-ordered graph list their entries by the target's degree
// class, heaviest first; class c holds the targets of degree >= kCutDegree[c]
// that no lighter-numbered class holds, the rest come last.
constexpr int kCutClasses = 8;
constexpr int kCutDegree[kCutClasses] = {1024, 256, 128, 64, 32, 16, 8, 4};
struct CutBounds {
    long long below[kCutClasses];   // ids of the vertices of degree >= kCutDegree[c] are below
    long long reach;                // ids of the vertices that some row leads to are below
};

// Entries from which a level of the default single-source kernel runs dense
// (an eighth of it where the level suits, see open_level).
constexpr long long kDenseMin = 1ll << 23;

// Entries from which a batched top-down run looks for vertices that every live
// lane has reached.  A graph of fewer gives a warp a few hundred entries per
// level at most, and the counters cost its levels more than the entries spared
// (64 lanes, 50 k vertices, 0.8 M entries: 151 us with them, 147 without; 131 k,
// 2 M: 190 either way; 600 k, 9 M: 386 with them, 412 before there were any).
constexpr long long kFilterMin = 1ll << 20;

// Whether a level of a graph of nnz entries can run dense (a level never holds
// more entries than the graph; open_level has the rule for one level).  Where
// none can, the form of the default kernel without that path is launched: its
// sparse levels keep 64 registers with 112 / 148 bytes of spills and 14.2 KB of
// shared memory per CTA where the form with both has 388 / 532 and 19.3 KB
// (65 k vertices, 2.1 M entries: 96 us in the form with both, 77 without).
inline bool may_run_dense(long long nnz, bool has_cut, long long dense_min) {
    return (has_cut ? 8 * nnz : nnz) >= dense_min;
}

struct TraversalParams {
    // graph (device numbering)
    int64_t n;
    const int64_t* off;
    const int32_t* col;
    const int32_t* new2old;   // device -> caller numbering (nullptr: identity)
    const int32_t* old2new;   // caller -> device numbering (nullptr: identity)
    // degree bins
    int32_t t_small;
    int32_t t_large;
    int32_t chunk_warp;
    int32_t chunk_cta;
    // workspace
    uint32_t* visited;        // plain: 1 bit per vertex
    uint32_t* queued;         // default single-source kernel: vertices already in a frontier
                              // (a dense level's sweep takes visited & ~queued)
    long long dense_min;      // default single-source kernel: a level whose frontier has at
                              // least this many entries runs dense
    const uint16_t* cut;      // nullable, [kCutClasses][n]: entries of each row in classes 0..c
                              // (at most 65535)
    long long cut_bound[kCutClasses];  // vertices of degree >= kCutDegree[c]: their ids are below
    long long sweep_limit;    // vertices that some row leads to are below this (the default
                              // single-source kernel's sweeps, the batched full bitmap)
    BinQueue q[2][kBins];
    LevelCtl* ctl;            // [3]
    GridBarrier* bar;
    DevStats* stats;
    // batched traversal state
    uint64_t* lane_vn;        // [n][2]: lanes that reached v (visited), lanes reaching v next
    uint64_t* lane_front;     // [n]: lanes for which v is in the current frontier (dir_mode != 0)
    uint32_t* full;           // bitmap of the vertices every live lane has reached (nullptr:
                              // not looked for; else the buffer of lane_front)
    uint8_t* lane_level;      // [n][64 bytes]: 8 bit planes of 64 lanes' levels at each vertex
    int32_t nlanes;
    int32_t dist_int8;
    int32_t roots[64];        // caller numbering, [nlanes]
    // outputs (caller numbering)
    int32_t* dist;            // plain: [n]; batched: [nlanes][n] (int32 or int8)
    int32_t* parent;          // plain only, nullable
    int32_t root_caller;      // plain: caller numbering
    // control
    int32_t level;            // host-loop mode: the level this launch runs
    int32_t phase;            // host-loop mode: 0 init, 1 seed, 2 level (batched: 3 sweep)
    long long timeout_ns;
    int32_t debug_stall;
    int32_t use_match_any;    // warp-aggregated atomicOr on the visited bitmap
    int32_t hot_words;        // visited words copied to shared memory on large levels (0: off)
    long long hot_min_edges;  // a level is large when its frontier has this many edges
    // frontier bitmaps and the bottom-up step (plain traversal)
    uint32_t* fb[3];          // frontier of level L in fb[L % 3]; nullptr: not kept
    long long nnz;
    long long bu_limit;       // bottom-up scans vertices [0, bu_limit)
    int32_t dir_mode;         // 0 top-down, 1 direction-optimizing, 2 bottom-up on every level
    int32_t do_alpha;         // top-down -> bottom-up when frontier edges * alpha > unvisited edges
    int32_t do_beta;          // bottom-up -> top-down when frontier vertices * beta < n
    int32_t dir_override;     // host-loop launches: direction chosen by the host (-1: device)
    int32_t bitmap_div;       // top-down levels with more than n / bitmap_div frontier
                              // vertices walk the frontier bitmap (0: never)
    long long bitmap_from;    // first vertex that can be light (degree-ordered graphs)
    int32_t l2_prefetch;      // bulk L2 prefetch of the heavy bins' column segments
    int32_t tma_stage;        // bin-2 column blocks staged in shared memory by TMA bulk copies
    int32_t tma_offset;       // byte offset of the staging buffers in dynamic shared memory
    int32_t timeline_cap;     // entries of timeline
    unsigned long long* timeline;  // nullable: %globaltimer after init, seed and each level
    unsigned long long graph_cond; // graph-captured loop: conditional handle of the while node
    const int* pre_status;    // nullable: a status written by an earlier launch on the same
                              // stream (CSR validation); non-zero ends the traversal before
                              // its first access to the graph
};

// Direction of level L (Beamer, Asanovic, Patterson, "Direction-optimizing
// breadth-first search", SC 2012): 0 = top-down over the frontier queues,
// 1 = top-down over the frontier bitmap, 2 = bottom-up.  m_f: edges of the
// frontier, m_u: edges of the vertices not yet visited, n_f: frontier
// vertices.
__host__ __device__ inline int choose_direction(int mode, bool prev_bu, long long m_f,
                                                long long m_u, long long n_f, long long n,
                                                int alpha, int beta, int bitmap_div) {
    const int td = (bitmap_div > 0 && n_f * (long long)bitmap_div > n) ? 1 : 0;
    if (mode == 0) return td;
    if (mode == 2) return 2;
    if (!prev_bu) return (m_f * (long long)alpha > m_u) ? 2 : td;
    return (n_f * (long long)beta < n) ? td : 2;
}

}  // namespace bfs
