// bfs_device.cuh -- device code the traversal kernels share: warp helpers,
// the bounded grid barrier, the per-warp stage of candidate vertices with
// its flush into the binned next frontier, and the probe of a round of edges.
//
// Included by bfs_kernels.cu (every optional path, the batched kernels, the
// host- and graph-driven level loops) and, with BFS_LEAN_PATHS = 1, by
// bfs_single.cu (the default single-source kernel), where the paths only
// bfs_kernels.cu offers -- frontier bitmaps kept by the flush, the
// shared-memory copy of the hot bitmap, warp-aggregated claims -- are
// compiled out: they cost the probe loops registers even when not taken.
#pragma once

#include <cuda_runtime.h>
#include <cstdint>

#include "bfs_internal.h"

#ifndef BFS_LEAN_PATHS
#define BFS_LEAN_PATHS 0
#endif

namespace bfs {
// one set of functions per including file: they differ in the paths compiled in
#if BFS_LEAN_PATHS
inline namespace device_default {
#else
inline namespace device_optional {
#endif

constexpr bool kLean = BFS_LEAN_PATHS != 0;

#define FULL_MASK 0xffffffffu

// ---------------------------------------------------------------- helpers

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }
__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm volatile("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}
__device__ __forceinline__ unsigned long long global_timer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ int ld_volatile_i32(const int* p) { return *(const volatile int*)p; }
__device__ __forceinline__ unsigned long long ld_cg_u64(const unsigned long long* p) {
    return __ldcg(p);
}

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T x) {
    const unsigned lane = lane_id();
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        T y = __shfl_up_sync(FULL_MASK, x, d);
        if (lane >= (unsigned)d) x += y;
    }
    return x;
}

__device__ __forceinline__ void raise_status(const TraversalParams& P, int code) {
    atomicCAS(&P.stats->status, 0, code);
}

// One bulk request that brings col[a, b) into L2 (cp.async.bulk.prefetch:
// no shared memory, no completion to wait for).  Start and size must be
// multiples of 16 bytes; col is padded past its last entry, so rounding the
// end up stays inside the allocation.
__device__ __forceinline__ void prefetch_cols_l2(const int32_t* col, long long a, long long b) {
    if (b <= a) return;
    const long long a4 = a & ~3ll, b4 = (b + 3) & ~3ll;
    const unsigned bytes = (unsigned)((b4 - a4) * 4);
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(col + a4), "r"(bytes)
                 : "memory");
}

// Prefetch distance of the heavy bins, in column entries (32 KiB).
constexpr long long kPrefetchAhead = 8192;

// Level timeline (diagnostics): block 0, thread 0 records %globaltimer.
__device__ __forceinline__ void stamp(const TraversalParams& P, int i) {
    if (P.timeline && i < P.timeline_cap && blockIdx.x == 0 && threadIdx.x == 0)
        P.timeline[i] = global_timer_ns();
}

// ------------------------------------------------- TMA bulk copies (1D)
__device__ __forceinline__ unsigned smem_u32(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}
// Arrive on bar and expect `bytes` of asynchronous transfers in this phase.
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}"
                 ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// One bulk copy global -> shared (16-byte aligned ends, size a multiple of
// 16), completing `bytes` transactions on bar.
__device__ __forceinline__ void tma_load_1d(void* dst, const void* src, unsigned bytes,
                                            unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Waits for phase `parity` of bar, giving up after the traversal's wait
// limit (%globaltimer) or when another CTA has aborted the launch.
__device__ __forceinline__ bool mbar_wait_bounded(const TraversalParams& P,
                                                  unsigned long long* bar, unsigned parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_timer_ns();
    for (unsigned it = 0;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 15u) == 15u) {
            if (global_timer_ns() - t0 > (unsigned long long)P.timeout_ns) return false;
            if (ld_volatile_i32(&P.stats->abort) != 0) return false;
        }
    }
}

// ------------------------------------------------------------ grid barrier
// All CTAs are co-resident (cooperative launch).  Thread 0 of each CTA adds
// its arrival to one 64-bit word that only grows during a launch: the k-th
// barrier is complete once the word reaches k * gridDim.x, so an arrival is a
// fire-and-forget reduction and the wait is a loop of acquire loads (no reset
// or generation step that the last arrival would have to publish with further
// round trips).  An acquire load throws away the SM's L1: where some CTAs of
// an SM wait long while others still expand (long_wait, the dense levels), the
// loop polls with relaxed loads and fences once at its end (scale 22, level 2:
// 222 -> 196 us; on short waits the fence costs 0.3 us).  Bit 63 of the word
// says that a CTA gave up: a wait longer than timeout_ns of %globaltimer
// records kDevTimeout, sets the bit and returns false, and every CTA that
// reads the bit returns false too. `epoch` (thread 0's, in shared memory: no
// register held across the level loop) counts the barriers this CTA has passed
// in the launch, the same in every CTA; the last CTA to leave the launch
// clears the word.
constexpr unsigned long long kBarGaveUp = 1ull << 63;

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Tells every CTA waiting at (or arriving at) a grid barrier to leave.
__device__ __forceinline__ void give_up(const TraversalParams& P) {
    atomicExch(&P.stats->abort, 1);
    atomicOr(&P.bar->arrived, kBarGaveUp);
}

__device__ bool grid_barrier(const TraversalParams& P, unsigned long long& epoch,
                             bool long_wait = false) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long* const word = &P.bar->arrived;
        const unsigned long long target =
            ++epoch * gridDim.x + (P.debug_stall ? 1ull : 0ull);
        __threadfence();
        asm volatile("red.relaxed.gpu.global.add.u64 [%0], 1;" ::"l"(word) : "memory");
        int ok = 1;
        unsigned long long t0 = 0ull;
        for (;;) {
            const unsigned long long a = long_wait ? ld_relaxed_u64(word) : ld_acquire_u64(word);
            if (a & kBarGaveUp) { ok = 0; break; }
            if (a >= target) break;
            const unsigned long long t = global_timer_ns();
            if (t0 == 0ull) {
                t0 = t;
            } else if (t - t0 > (unsigned long long)P.timeout_ns) {
                raise_status(P, kDevTimeout);
                give_up(P);
                ok = 0;
                break;
            }
        }
        if (long_wait) asm volatile("fence.acq_rel.gpu;" ::: "memory");
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// Last CTA to leave a persistent launch clears the barrier and abort flag,
// so the next launch starts clean even after a timed-out wait.
__device__ void kernel_exit(const TraversalParams& P) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned done = atomicAdd(&P.bar->exited, 1u) + 1u;
        if (done == gridDim.x) {
            atomicExch(&P.bar->arrived, 0ull);
            atomicExch(&P.bar->exited, 0u);
            atomicExch(&P.stats->abort, 0);
            __threadfence();
        }
    }
}

// --------------------------------------------------------------- enqueue
// Candidate vertices (claimed or still to claim) are staged per warp in
// shared memory and appended to the next frontier up to 64 at a time
// (measured faster than 32, 128 and 256 on GB300).  The flush claims the
// unclaimed ones, does the per-vertex work that needs random reads (degree
// from the row offsets, caller numbering) for the whole group at once,
// writes the distances and parents, bins the group by degree, and reserves
// queue slots and edge ranges with one 64-bit atomicAdd per bin (the bin
// counter packs entries << 34 | edge prefix).
#ifndef BFS_STAGE_CAP
#define BFS_STAGE_CAP 64
#endif
constexpr int kStageCap = BFS_STAGE_CAP;
// A probe round whose warp holds at least this many candidates claims them
// at once (one atomic round trip shared by all of them); rounds with fewer
// leave the claim to the stage flush.
#ifndef BFS_CLAIM_NOW
#define BFS_CLAIM_NOW 16
#endif
constexpr int kClaimNow = BFS_CLAIM_NOW;
// Parent field flag of a staged entry that is already claimed.
constexpr uint32_t kClaimed = 0x80000000u;

template <bool kBatch>
struct Stage {
    int32_t u[kStageCap];
    int32_t v[kBatch ? 1 : kStageCap];                 // plain: parent of u
    unsigned long long mask[kBatch ? kStageCap : 1];   // batched: new lanes of u
    int cnt;
    unsigned long long edges;                          // batched: sum deg * lanes
    const uint32_t* hot;                               // plain: shared copy of visited[0, hot_bits);
                                                       // batched: bitmap of the vertices every live
                                                       // lane has reached, nullptr while few have
    const uint16_t* cut;                               // batched: entries at the front of each row
                                                       // that lead to such vertices (nullable)
    int hot_bits;                                      // 0 when the copy is off for this level
    int disc;                                          // plain: vertices this warp claimed
    uint4* tma_buf;                  // plain, BFS_OPT_TMA_STAGE: two 1 KB staging buffers
    unsigned long long* tma_bar;     // their mbarriers
    unsigned tma_ph;                 // bit b: parity of buffer b's next phase
    int tma_ok;                      // 0 after a staging wait gave up
};

// Warp-collective flush of the staged entries into the next frontier.
// Lane l owns entries [H l, H l + H): all their random reads (row offsets,
// caller numbering) are issued together; one packed atomicAdd per bin,
// issued by lanes 0..2 at once, places the lane's entries at consecutive
// queue slots.
//
// The flush is inlined at every call site: as an out-of-line call it made
// the callers save their live registers around it (spills on the probe
// loops' critical path).  Launch parameters are still read into registers
// before the stores that follow them: P is a reference, and a parameter read
// after a global store through a generic pointer cannot be moved above it
// (the compiler cannot rule out that the store changed the parameter), which
// would put a round trip on every chunk-table iteration.
template <bool kBatch>
__device__ __forceinline__ void stage_flush(const TraversalParams& P, Stage<kBatch>& S, int level,
                                         int nxt, int nslot) {
    constexpr int H = kStageCap / 32;
    const unsigned lane = lane_id();
    const int n = S.cnt;
    if (n == 0) return;
    const int64_t* const off = P.off;
    const int32_t* const new2old = P.new2old;
    int32_t* const dist = P.dist;
    int32_t* const parent = P.parent;
    uint32_t* const fbn = (!kLean && P.fb[0]) ? P.fb[(level + 1) % 3] : nullptr;
    const int t_small = P.t_small, t_large = P.t_large;
    const int sh_warp = __ffs(P.chunk_warp) - 1, sh_cta = __ffs(P.chunk_cta) - 1;
    unsigned long long* const packed = P.ctl[nslot].packed;
    bool overflow = false;

    const int i0 = (int)lane * H;
    int32_t u[H];
    int deg[H];
#pragma unroll
    for (int h = 0; h < H; ++h) u[h] = (i0 + h < n) ? S.u[i0 + h] : -1;
    // The random reads that do not depend on the claim (row offsets, caller
    // numbering) are issued before it, so that their round trip overlaps the
    // atomics' instead of following it.
#pragma unroll
    for (int h = 0; h < H; ++h) {
        deg[h] = -1;
        if (u[h] >= 0) deg[h] = (int)(__ldg(off + u[h] + 1) - __ldg(off + u[h]));
    }
    int32_t cu[H], cv[H];
    // Plain entries are candidates (their target looked unvisited when it
    // was probed): the claim -- an atomicOr on the visited bitmap whose old
    // value says who set the bit first -- happens here, for all of a flush's
    // entries at once, instead of one round trip per probe round.
    uint32_t old[H];
    uint32_t pv[H];  // plain: staged parent with the claimed flag
    if constexpr (!kBatch) {
        uint32_t* const visited = P.visited;
#pragma unroll
        for (int h = 0; h < H; ++h) {
            pv[h] = u[h] >= 0 ? (uint32_t)S.v[i0 + h] : 0u;
            cu[h] = u[h];
            cv[h] = (u[h] >= 0) ? (int32_t)(pv[h] & ~kClaimed) : 0;
            if (new2old && u[h] >= 0) {
                cu[h] = __ldg(new2old + u[h]);
                cv[h] = __ldg(new2old + cv[h]);
            }
        }
        if (!kLean && P.use_match_any) {
            // lanes claiming bits of the same word merge them: one atomicOr
            // per word, the first lane holding a vertex wins it
#pragma unroll
            for (int h = 0; h < H; ++h) {
                old[h] = (u[h] >= 0 && (pv[h] & kClaimed)) ? 0u : 0xffffffffu;
                const bool need = u[h] >= 0 && !(pv[h] & kClaimed);
                const unsigned needm = __ballot_sync(FULL_MASK, need);
                if (need) {
                    const uint32_t bit = 1u << (u[h] & 31);
                    const unsigned peers = __match_any_sync(needm, u[h] >> 5);
                    const uint32_t bits = __reduce_or_sync(peers, bit);
                    const int leader = __ffs(peers) - 1;
                    uint32_t o = 0u;
                    if ((int)lane == leader) o = atomicOr(visited + (u[h] >> 5), bits);
                    o = __shfl_sync(peers, o, leader);
                    const unsigned same = __match_any_sync(peers, u[h]);
                    if ((o & bit) == 0u && (int)lane == __ffs(same) - 1) old[h] = 0u;
                }
            }
        } else {
#pragma unroll
            for (int h = 0; h < H; ++h) {
                old[h] = 0xffffffffu;
                if (u[h] >= 0)
                    old[h] = (pv[h] & kClaimed) ? 0u : atomicOr(visited + (u[h] >> 5), 1u << (u[h] & 31));
            }
        }
    }
    if constexpr (kBatch) {
        unsigned long long e = 0;
#pragma unroll
        for (int h = 0; h < H; ++h)
            if (u[h] >= 0) e += (unsigned long long)deg[h] * __popcll(S.mask[i0 + h]);
        if (e) atomicAdd(&S.edges, e);
    } else {
        // entries whose claim lost are dropped
        int won = 0;
#pragma unroll
        for (int h = 0; h < H; ++h) {
            if (u[h] >= 0 && ((old[h] >> (u[h] & 31)) & 1u)) {
                u[h] = -1;
                deg[h] = -1;
            }
            won += __popc(__ballot_sync(FULL_MASK, u[h] >= 0));
        }
        if (lane == 0) S.disc += won;
#pragma unroll
        for (int h = 0; h < H; ++h) {
            if (u[h] < 0) continue;
            dist[cu[h]] = level + 1;
            if (parent) parent[cu[h]] = cv[h];
            if (fbn) atomicOr(fbn + (u[h] >> 5), 1u << (u[h] & 31));
        }
    }
    // Reserve queue slots and edge ranges for all bins in one round trip:
    // per bin one warp scan of (entries << 48 | degree sum) -- a lane holds
    // at most H entries and degrees stay below 2^31, so the sum fits in 48
    // bits -- then lanes 0..2 issue the bins' atomicAdds together.
    int bh[H];
#pragma unroll
    for (int h = 0; h < H; ++h)
        bh[h] = deg[h] <= 0 ? -1 : (deg[h] < t_small ? 0 : (deg[h] < t_large ? 1 : 2));
    unsigned long long incl[kBins], mine[kBins];
    unsigned long long add = 0ull;
#pragma unroll
    for (int b = 0; b < kBins; ++b) {
        unsigned long long x = 0ull;
#pragma unroll
        for (int h = 0; h < H; ++h)
            if (bh[h] == b) x += (1ull << 48) + (unsigned long long)deg[h];
        mine[b] = x;
        incl[b] = 0ull;
        if (__ballot_sync(FULL_MASK, x != 0ull) == 0u) continue;
        incl[b] = warp_incl_scan(x);
        const unsigned long long tot = __shfl_sync(FULL_MASK, incl[b], 31);
        if (lane == (unsigned)b)
            add = ((tot >> 48) << kCountShift) + (tot & ((1ull << 48) - 1ull));
    }
    unsigned long long basep = 0ull;
    if (add != 0ull) basep = atomicAdd(packed + lane, add);
#pragma unroll
    for (int b = 0; b < kBins; ++b) {
        const unsigned long long base = __shfl_sync(FULL_MASK, basep, b);
        if (mine[b] == 0ull) continue;
        const unsigned long long excl = incl[b] - mine[b];
        long long pos = (long long)(base >> kCountShift) + (long long)(excl >> 48);
        long long eo = (long long)(base & kEdgeMask) + (long long)(excl & ((1ull << 48) - 1ull));
        // chunk sizes are powers of two: chunk c starts at edge c << cshift
        const int cshift = b == 1 ? sh_warp : sh_cta;
        const BinQueue& Q = P.q[nxt][b];
        int32_t* const qv = Q.v;
        int64_t* const qe = Q.eoff;
        int32_t* const qc = Q.chunk;
        uint64_t* const qm = kBatch ? Q.mask : nullptr;
        const long long qcap = Q.cap, qccap = Q.chunk_cap;
#pragma unroll
        for (int h = 0; h < H; ++h) {
            if (bh[h] != b) continue;
            if (pos < qcap) {
                qv[pos] = u[h];
                if (kBatch) qm[pos] = S.mask[kBatch ? i0 + h : 0];
                if (b > 0) {
                    qe[pos] = eo;
                    // chunks whose first edge lies in [eo, eo + deg) start here
                    const long long c_end = (eo + deg[h] - 1) >> cshift;
                    const long long c0 = (eo + (1ll << cshift) - 1) >> cshift;
                    if (c_end >= qccap) overflow = true;
                    for (long long c = c0; c <= c_end && c < qccap; ++c) qc[c] = (int32_t)pos;
                }
            } else {
                overflow = true;
            }
            ++pos;
            eo += deg[h];
        }
    }
    if (overflow) raise_status(P, kDevOverflow);
    __syncwarp();
    if (lane == 0) S.cnt = 0;
    __syncwarp();
}

// Warp-collective: lanes with ok stage u (with its parent v, or its new
// lanes mask).
template <bool kBatch>
__device__ __forceinline__ void stage_push(const TraversalParams& P, Stage<kBatch>& S, bool ok,
                                           int32_t u, int32_t v, uint64_t mask, int level,
                                           int nxt, int nslot) {
    const unsigned m = __ballot_sync(FULL_MASK, ok);
    if (m == 0u) return;
    int n0 = S.cnt;
    const int k = __popc(m);
    if (n0 + k > kStageCap) {
        stage_flush<kBatch>(P, S, level, nxt, nslot);
        n0 = 0;
    }
    if (ok) {
        const int i = n0 + __popc(m & lanemask_lt());
        S.u[i] = u;
        if constexpr (kBatch) S.mask[i] = mask;
        else S.v[i] = v;
    }
    __syncwarp();
    if (lane_id() == 0) S.cnt = n0 + k;
    __syncwarp();
}

template <bool kBatch>
__device__ __forceinline__ void stage_init(Stage<kBatch>& S) {
    if (lane_id() == 0) {
        S.cnt = 0;
        S.edges = 0ull;
        S.hot = nullptr;
        S.cut = nullptr;
        S.hot_bits = 0;
        S.disc = 0;
        S.tma_buf = nullptr;
        S.tma_bar = nullptr;
        S.tma_ph = 0u;
        S.tma_ok = 0;
    }
    __syncwarp();
}

// Staging buffers and mbarriers of this warp (plain kernels with
// BFS_OPT_TMA_STAGE): two 1 KB buffers in dynamic shared memory after the
// hot bitmap prefix, two mbarriers with one arrival per phase.
__device__ void tma_setup(const TraversalParams& P, Stage<false>& S, uint4* s_dyn) {
    __shared__ __align__(8) unsigned long long s_tma_bar[kWarps * 2];
    if (!P.tma_stage) return;
    const int warp = threadIdx.x >> 5;
    if (lane_id() == 0) {
        unsigned long long* bar = s_tma_bar + 2 * warp;
        mbar_init(bar, 1u);
        mbar_init(bar + 1, 1u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        S.tma_buf = s_dyn + P.tma_offset / 16 + warp * 128;
        S.tma_bar = bar;
        S.tma_ph = 0u;
        S.tma_ok = 1;
    }
    __syncwarp();
}

// ----------------------------------------------------------------- visits
// Stages each lane's candidates (bit j of candm: u[j] with parent v(j),
// flag kClaimed when already claimed) in one pass: a warp scan of the
// per-lane counts places them; a full stage is flushed and the rest placed
// after it.
template <int K, class Row>
__device__ __forceinline__ void stage_push_multi(const TraversalParams& P, Stage<false>& S,
                                                 unsigned candm, const int32_t (&u)[K], Row&& v,
                                                 uint32_t flag, int level, int nxt, int nslot) {
    const int c = __popc(candm);
    if (__ballot_sync(FULL_MASK, c != 0) == 0u) return;
    const int incl = warp_incl_scan(c);
    const int total = __shfl_sync(FULL_MASK, incl, 31);
    const int excl = incl - c;
    for (int done = 0; done < total;) {
        int n0 = S.cnt;
        if (n0 == kStageCap) {
            stage_flush<false>(P, S, level, nxt, nslot);
            n0 = 0;
        }
        const int take = min(kStageCap - n0, total - done);
        int k = excl - done;  // stage offset of this lane's next candidate
#pragma unroll
        for (int j = 0; j < K; ++j) {
            if ((candm >> j) & 1u) {
                if (k >= 0 && k < take) {
                    S.u[n0 + k] = u[j];
                    S.v[n0 + k] = (int32_t)((uint32_t)v(j) | flag);
                }
                ++k;
            }
        }
        __syncwarp();
        if (lane_id() == 0) S.cnt = n0 + take;
        __syncwarp();
        done += take;
    }
}

// K edges per lane at once: all K visited-bitmap probes are issued before
// any result is used, so a warp keeps K random reads in flight instead of
// one.  A probe that finds the bit clear makes the edge a candidate.  The
// claim (the atomicOr whose old value decides which edge discovers the
// vertex) is made here when the round has many candidates -- discovery-
// heavy levels, where claiming early also keeps other warps from staging
// the same vertex -- and otherwise left to the stage flush, which claims a
// whole stage in one round trip instead of one per probe round.  A stale
// cached word can only show clear a bit that is already set (bits are never
// cleared during a traversal), and the claim then rejects the candidate.
template <int K, class Row>
__device__ __forceinline__ void visit_plain_k(const TraversalParams& P, Stage<false>& S,
                                              unsigned okm, const int32_t (&u)[K], Row&& v,
                                              int level, int nxt, int nslot) {
    // pass 1 (shared memory only): drop edges whose target was visited before
    // the level and lies in the hot prefix copied at level start
    const int hot_bits = S.hot_bits;
    if (!kLean && hot_bits > 0) {
        const uint32_t* hot = S.hot;
#pragma unroll
        for (int j = 0; j < K; ++j)
            if (((okm >> j) & 1u) && u[j] < hot_bits && ((hot[u[j] >> 5] >> (u[j] & 31)) & 1u))
                okm &= ~(1u << j);
    }
    // pass 2: independent global probes for the rest
    uint32_t w[K];
#pragma unroll
    for (int j = 0; j < K; ++j) w[j] = ((okm >> j) & 1u) ? P.visited[u[j] >> 5] : 0xffffffffu;
    unsigned candm = 0u;
#pragma unroll
    for (int j = 0; j < K; ++j)
        if (((w[j] >> (u[j] & 31)) & 1u) == 0u) candm |= 1u << j;
    const int total = __reduce_add_sync(FULL_MASK, (unsigned)__popc(candm));
    if (total == 0) return;
    uint32_t flag = 0u;
    if (total >= kClaimNow) {
#pragma unroll
        for (int j = 0; j < K; ++j)
            if ((candm >> j) & 1u) w[j] = atomicOr(P.visited + (u[j] >> 5), 1u << (u[j] & 31));
#pragma unroll
        for (int j = 0; j < K; ++j)
            if (((w[j] >> (u[j] & 31)) & 1u) != 0u) candm &= ~(1u << j);
        flag = kClaimed;
    }
    stage_push_multi<K>(P, S, candm, u, v, flag, level, nxt, nslot);
}

// Batched traversal, phase A: OR the lanes of the frontier entry that u has
// not seen yet into next[u].  visited only changes in phase B, so a cached
// value is a safe filter; next[u] is read first so that lanes already
// present skip the atomic (a fire-and-forget red.or otherwise).
// The K pairs are read in groups of 4 (8 would keep 32 registers of pairs
// live, which spills at 3 CTAs per SM).
// Once many vertices have been reached by every live lane, their bitmap
// (n / 8 bytes, mostly L1 hits in degree order) is read first: it spares two
// thirds of a scale-20 launch's level 3 entries and nearly all of level 4's
// the 16-byte read through L2 (scale 22, with the row cuts: level 4 258 -> 87
// us, level 3 552 -> 510).
template <int K>
__device__ __forceinline__ void visit_batch_k(const TraversalParams& P, const uint32_t* full,
                                              unsigned okm, const int32_t (&u)[K],
                                              const uint64_t (&mask)[K]) {
    constexpr int G = K < 4 ? K : 4;
    if (full != nullptr) {
        uint32_t w[K];
#pragma unroll
        for (int j = 0; j < K; ++j) w[j] = ((okm >> j) & 1u) ? full[u[j] >> 5] : 0u;
#pragma unroll
        for (int j = 0; j < K; ++j)
            if ((w[j] >> (u[j] & 31)) & 1u) okm &= ~(1u << j);
        if (__ballot_sync(FULL_MASK, okm != 0u) == 0u) return;
    }
#pragma unroll
    for (int j0 = 0; j0 < K; j0 += G) {
        // visited and next of a vertex are adjacent: one 16-byte load each
        ulonglong2 vn[G];
#pragma unroll
        for (int j = 0; j < G; ++j)
            vn[j] = ((okm >> (j0 + j)) & 1u)
                        ? *reinterpret_cast<const ulonglong2*>(P.lane_vn + 2 * (long long)u[j0 + j])
                        : make_ulonglong2(~0ull, ~0ull);
#pragma unroll
        for (int j = 0; j < G; ++j) {
            const uint64_t m = mask[j0 + j] & ~vn[j].x;
            if ((m & ~vn[j].y) != 0ull)
                atomicOr(reinterpret_cast<unsigned long long*>(P.lane_vn + 2 * (long long)u[j0 + j] + 1),
                         (unsigned long long)m);
        }
    }
}

template <bool kBatch, int K>
__device__ __forceinline__ void visit_k(const TraversalParams& P, Stage<kBatch>& S, unsigned okm,
                                        const int32_t (&u)[K], const int32_t (&v)[K],
                                        const uint64_t (&mask)[K], int level, int nxt, int nslot) {
    if constexpr (kBatch) visit_batch_k<K>(P, S.hot, okm, u, mask);
    else visit_plain_k<K>(P, S, okm, u, [&](int j) { return v[j]; }, level, nxt, nslot);
}

// ------------------------------------------------------------ expansion
#if !BFS_LEAN_PATHS
// bfs_kernels.cu
__device__ void expand_segment_staged(const TraversalParams& P, Stage<false>& S, long long a4,
                                      int lo, int hi, int32_t v, int level, int nxt, int nslot,
                                      int wbase);
__device__ void expand_bitmap_tile(const TraversalParams& P, Stage<false>& S, long long tile,
                                   int level, int nxt, int nslot);
#endif

// One column segment col[a, b) of vertex v, read by a group of warps with
// 128-bit loads (start rounded down to 16 bytes; col is padded so the
// rounded reads stay inside the allocation).  wbase/wstride place this
// warp's 256-entry blocks; a segment that fits in 128 entries uses one
// 128-bit load per lane.
template <bool kBatch, bool kStaged = false>
__device__ __forceinline__ void expand_segment(const TraversalParams& P, Stage<kBatch>& S,
                                               long long a, long long b, int32_t v, uint64_t mask,
                                               int level, int nxt, int nslot, long long wbase,
                                               long long wstride) {
    const unsigned lane = lane_id();
    const long long a4 = a & ~3ll;
    const int lo = (int)(a - a4);                 // valid entries: [lo, hi) relative to a4
    const int hi = (int)(b - a4);
#if !BFS_LEAN_PATHS
    if constexpr (!kBatch && kStaged) {
        if (S.tma_buf != nullptr && wstride == 256ll * kWarps) {
            expand_segment_staged(P, S, a4, lo, hi, v, level, nxt, nslot, (int)wbase);
            return;
        }
    }
#endif
    const int32_t* colp = P.col + a4;
    int32_t vv[8];
    uint64_t mm[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        vv[j] = v;
        mm[j] = mask;
    }
    if (wbase == 0 && wstride == 256 && hi <= 128) {
        const int r0 = 4 * (int)lane;
        int4 x0 = make_int4(0, 0, 0, 0);
        if (r0 < hi) x0 = __ldcs(reinterpret_cast<const int4*>(colp + r0));
        unsigned okm = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (r0 + j >= lo && r0 + j < hi) okm |= 1u << j;
        const int32_t u[4] = {x0.x, x0.y, x0.z, x0.w};
        const int32_t v4[4] = {v, v, v, v};
        const uint64_t m4[4] = {mask, mask, mask, mask};
        visit_k<kBatch, 4>(P, S, okm, u, v4, m4, level, nxt, nslot);
        return;
    }
    for (int rw = (int)wbase; rw < hi; rw += (int)wstride) {
        if (!kLean && P.l2_prefetch && lane == 0 && rw + kPrefetchAhead < hi)
            prefetch_cols_l2(P.col, a4 + rw + kPrefetchAhead,
                             a4 + min((long long)hi, rw + kPrefetchAhead + 256));
        const int r0 = rw + 4 * (int)lane;
        const int r1 = r0 + 128;
        int4 x0 = make_int4(0, 0, 0, 0), x1 = make_int4(0, 0, 0, 0);
        if (r0 < hi) x0 = __ldcs(reinterpret_cast<const int4*>(colp + r0));
        if (r1 < hi) x1 = __ldcs(reinterpret_cast<const int4*>(colp + r1));
        unsigned okm = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (r0 + j >= lo && r0 + j < hi) okm |= 1u << j;
            if (r1 + j >= lo && r1 + j < hi) okm |= 1u << (4 + j);
        }
        const int32_t u[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
        visit_k<kBatch, 8>(P, S, okm, u, vv, mm, level, nxt, nslot);
    }
}

// Bin 0: 32 frontier vertices per warp, one per lane; their edges are laid
// end to end by an exclusive scan and consumed 256 per round, lane l taking
// edges l + 32 j (j < 8) and finding each edge's owner vertex in a
// per-round owner table in shared memory that each lane fills for its own
// edges (cheaper than a shuffle binary search per edge: a lane writes at
// most its degree's slots).
template <bool kBatch>
__device__ void expand_small_group(const TraversalParams& P, Stage<kBatch>& S, int cur,
                                   long long grp, long long cnt, int level, int nxt, int nslot) {
    const BinQueue& Q = P.q[cur][0];
    const unsigned lane = lane_id();
    const long long i = grp * 32 + lane;
    int32_t v = 0;
    long long base = 0;
    int deg = 0;
    uint64_t mask = 0ull;
    if (i < cnt) {
        v = __ldcg(Q.v + i);
        base = __ldg(P.off + v);
        deg = (int)(__ldg(P.off + v + 1) - base);
        if (kBatch && S.cut) {
            const int skip = __ldg(S.cut + v);
            base += skip;
            deg -= skip;
        }
        if (kBatch) mask = __ldcg(reinterpret_cast<const unsigned long long*>(Q.mask) + i);
    }
    const int incl = warp_incl_scan(deg);
    const int excl = incl - deg;
    const int total = __shfl_sync(FULL_MASK, incl, 31);
    // owner of each of the round's 256 edge slots, written by the owning lane
    __shared__ uint8_t s_owner[kWarps][256];
    uint8_t* const own = s_owner[threadIdx.x >> 5];
    for (int e0 = 0; e0 < total; e0 += 256) {
        unsigned okm = 0u;
        int32_t u[8], vv[8];
        uint64_t mm[8];
        {
            const int a = max(excl, e0), b = min(excl + deg, e0 + 256);
            __syncwarp();
            for (int e = a; e < b; ++e) own[e - e0] = (uint8_t)lane;
            __syncwarp();
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int e = e0 + 32 * j + (int)lane;
            u[j] = 0;
            vv[j] = 0;
            mm[j] = 0ull;
            // slots past the round's last edge (the same for the whole warp)
            // need no owner lookup
            if (e0 + 32 * j < total) {
                const int o = e < total ? own[32 * j + lane] : 0;
                const long long bo = __shfl_sync(FULL_MASK, base, o);
                const int xo = __shfl_sync(FULL_MASK, excl, o);
                vv[j] = __shfl_sync(FULL_MASK, v, o);
                mm[j] = kBatch ? __shfl_sync(FULL_MASK, (unsigned long long)mask, o) : 0ull;
                if (e < total) {
                    okm |= 1u << j;
                    u[j] = __ldcs(P.col + bo + (e - xo));
                }
            }
        }
        visit_k<kBatch, 8>(P, S, okm, u, vv, mm, level, nxt, nslot);
    }
}

// Valid columns of the 16-byte unit holding row-relative columns [r, r + 4)
// of a row whose valid columns are [lo, hi): bits [lo - r, hi - r) of 4.
__device__ __forceinline__ unsigned unit_mask(int r, int lo, int hi) {
    const int a = min(max(lo - r, 0), 4), b = min(max(hi - r, 0), 4);
    return ((1u << b) - 1u) & ~((1u << a) - 1u);
}

// Bins 1 and 2 as warp items: edges [cs, ce) of bin b's level sequence
// (a bin-1 chunk of chunk_warp edges, or, on small levels, a 32-edge slice
// of either bin).  The range's vertex segments (up to 32 at a time, from the
// entry that holds the first edge of its base chunk) are cut into 16-byte
// units (4 columns, the first rounded down to a 16-byte boundary) laid end
// to end by a scan; each round a lane takes two units, finds their segments
// by a shuffle binary search, and reads each with one 128-bit load -- short
// and long segments alike keep every lane busy.
template <bool kBatch>
__device__ void expand_warp_range(const TraversalParams& P, Stage<kBatch>& S, const BinQueue& Q,
                                  int cshift, long long cs, long long ce, long long cnt, int level,
                                  int nxt, int nslot) {
    const unsigned lane = lane_id();
    long long i = __ldcg(Q.chunk + (cs >> cshift));
    for (;;) {
        const long long ij = i + lane;
        long long eo = 0x7fffffffffffffffll;
        if (ij < cnt) eo = __ldcg(Q.eoff + ij);
        const bool ok = eo < ce;
        bool live = false;  // the segment overlaps [cs, ce) (a slice's first
                            // entries may end before cs)
        int32_t v = 0;
        long long a = 0, b = 0;
        uint64_t mask = 0ull;
        if (ok) {
            v = __ldcg(Q.v + ij);
            const long long base = __ldg(P.off + v), end = __ldg(P.off + v + 1);
            const long long skip = kBatch && S.cut ? (long long)__ldg(S.cut + v) : 0ll;
            const long long lo = max(eo + skip, cs), hi = min(eo + (end - base), ce);
            live = hi > lo;
            a = base + (lo - eo);
            b = base + (hi - eo);
            if (kBatch) mask = __ldcg(reinterpret_cast<const unsigned long long*>(Q.mask) + ij);
            if (!kLean && P.l2_prefetch && live) prefetch_cols_l2(P.col, a, min(b, a + kPrefetchAhead));
        }
        const unsigned okb = __ballot_sync(FULL_MASK, ok);
        const long long a4 = a & ~3ll;
        const int rlo = (int)(a - a4), rhi = (int)(b - a4);  // valid columns, relative to a4
        const int units = live ? (rhi + 3) >> 2 : 0;
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
                int o = 0;
#pragma unroll
                for (int st = 16; st > 0; st >>= 1) {
                    const int c = o + st;
                    if (__shfl_sync(FULL_MASK, excl, c & 31) <= q) o = c;
                }
                const long long a4o = __shfl_sync(FULL_MASK, a4, o);
                const int lo_o = __shfl_sync(FULL_MASK, rlo, o);
                const int hi_o = __shfl_sync(FULL_MASK, rhi, o);
                const int xo = __shfl_sync(FULL_MASK, excl, o);
                const int32_t vo = __shfl_sync(FULL_MASK, v, o);
                const uint64_t mo = kBatch ? __shfl_sync(FULL_MASK, (unsigned long long)mask, o) : 0ull;
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
                    mm[4 * h + c] = mo;
                }
            }
            visit_k<kBatch, 8>(P, S, okm, u, vv, mm, level, nxt, nslot);
        }
        if (__popc(okb) < 32) break;
        i += 32;
    }
}

// Bin 2: one CTA per chunk of chunk_cta edges (a heavy vertex spans many
// chunks, hence many CTAs); the CTA's warps interleave over each segment.
template <bool kBatch, bool kStaged = false>
__device__ void expand_cta_chunk(const TraversalParams& P, Stage<kBatch>& S, int cur,
                                 long long item, int k, long long cnt, long long E, int level,
                                 int nxt, int nslot) {
    __shared__ long long s_eo[kBlock], s_base[kBlock], s_end[kBlock];
    __shared__ int32_t s_v[kBlock];
    __shared__ unsigned long long s_mask[kBatch ? kBlock : 1];
    __shared__ uint16_t s_skip[kBatch ? kBlock : 1];
    const BinQueue& Q = P.q[cur][2];
    const int warp = threadIdx.x >> 5;
    const long long cs = item * k * (long long)P.chunk_cta;
    const long long ce = min(cs + k * (long long)P.chunk_cta, E);
    long long i = __ldcg(Q.chunk + item * k);
    for (;;) {
        const long long ij = i + threadIdx.x;
        long long eo = 0x7fffffffffffffffll;
        if (ij < cnt) eo = __ldcg(Q.eoff + ij);
        const bool ok = eo < ce;
        if (ok) {
            const int32_t v = __ldcg(Q.v + ij);
            s_v[threadIdx.x] = v;
            s_eo[threadIdx.x] = eo;
            const long long base = __ldg(P.off + v), end = __ldg(P.off + v + 1);
            s_base[threadIdx.x] = base;
            s_end[threadIdx.x] = end;
            if (!kLean && P.l2_prefetch) {
                const long long a = base + (max(eo, cs) - eo);
                const long long b = base + (min(eo + (end - base), ce) - eo);
                prefetch_cols_l2(P.col, a, min(b, a + kPrefetchAhead));
            }
            if (kBatch) s_skip[kBatch ? threadIdx.x : 0] = S.cut ? __ldg(S.cut + v) : (uint16_t)0;
            if (kBatch)
                s_mask[kBatch ? threadIdx.x : 0] =
                    __ldcg(reinterpret_cast<const unsigned long long*>(Q.mask) + ij);
        }
        const int nent = __syncthreads_count(ok);
        for (int k = 0; k < nent; ++k) {
            const long long eok = s_eo[k], bk = s_base[k];
            const long long lo = max(eok + (kBatch ? s_skip[kBatch ? k : 0] : 0), cs);
            const long long hi = min(eok + (s_end[k] - bk), ce);
            if (kBatch && hi <= lo) continue;
            expand_segment<kBatch, kStaged>(P, S, bk + (lo - eok), bk + (hi - eok), s_v[k],
                                   kBatch ? s_mask[kBatch ? k : 0] : 0ull, level, nxt, nslot,
                                   (long long)warp * 256, 256ll * kWarps);
        }
        __syncthreads();
        if (nent < kBlock) break;
        i += kBlock;
    }
}

struct LevelShape {
    long long cnt[kBins], edges[kBins];
    long long n_cta;            // CTA items (bin 2)
    long long items_w1, items_w2;  // warp items of bins 1 and 2
    long long groups_small;     // light groups (bin 0)
    int k_cta;                  // base chunks per CTA item
    int sh_w1, sh_w2;           // log2 of the edges of a warp item of bins 1 and 2
    unsigned discovered;
};

__device__ __forceinline__ int pow2_floor_clamped(long long x, int kmax) {
    if (x <= 1) return 1;
    const int p = 63 - __clzll((unsigned long long)x);
    return p >= 31 ? kmax : min(1 << p, kmax);
}

// Shape of level `level` (frontier in slot level % 3, queues level & 1).
// Counts are clamped to the queue capacities so that a recorded overflow
// can never turn into an out-of-bounds read.
__device__ __forceinline__ LevelShape read_level(const TraversalParams& P, int level) {
    LevelShape s;
    const int slot = level % 3, cur = level & 1;
#pragma unroll
    for (int b = 0; b < kBins; ++b) {
        const unsigned long long p = ld_cg_u64(&P.ctl[slot].packed[b]);
        s.cnt[b] = min((long long)(p >> kCountShift), (long long)P.q[cur][b].cap);
        s.edges[b] = (long long)(p & kEdgeMask);
    }
    s.discovered = __ldcg(&P.ctl[slot].discovered);
    // base chunks (the granularity of the chunk tables), then work items of k
    // base chunks: small levels keep k = 1 so that every CTA / warp gets work,
    // large levels aim at ~4 items per CTA (or warp) to bound per-item costs
    const int sh_cta = __ffs(P.chunk_cta) - 1, sh_warp = __ffs(P.chunk_warp) - 1;
    const long long base_cta =
        min((s.edges[2] + P.chunk_cta - 1) >> sh_cta, (long long)P.q[cur][2].chunk_cap);
    const long long base_warp =
        min((s.edges[1] + P.chunk_warp - 1) >> sh_warp, (long long)P.q[cur][1].chunk_cap);
    s.k_cta = pow2_floor_clamped(base_cta / (4ll * gridDim.x), 32);
    const int k_warp = pow2_floor_clamped(base_warp / (4ll * gridDim.x * kWarps), 16);
    s.n_cta = (base_cta + s.k_cta - 1) / s.k_cta;
    s.items_w1 = (base_warp + k_warp - 1) / k_warp;
    s.sh_w1 = sh_warp + __ffs(k_warp) - 1;
    s.items_w2 = 0;
    s.sh_w2 = sh_cta;
    s.groups_small = (s.cnt[0] + 31) / 32;
    // Small levels: bins 1 and 2 cut into 32-edge warp slices when that,
    // with the light groups, still gives no warp more than one item.  The
    // level then costs one slice's chain of dependent accesses, where a
    // CTA chunk (1024 edges on 4 warps) or a warp chunk chained a probe
    // round and several flushes of its discoveries.
    const long long f1 = min((s.edges[1] + 31) >> 5, base_warp << (sh_warp - 5));
    const long long f2 = min((s.edges[2] + 31) >> 5, base_cta << (sh_cta - 5));
    if (f1 + f2 > 0 && f1 + f2 + s.groups_small <= (long long)gridDim.x * kWarps) {
        s.n_cta = 0;
        s.items_w1 = f1;
        s.items_w2 = f2;
        s.sh_w1 = s.sh_w2 = 5;
    }
    return s;
}

// Top-down work of one level: CTA chunks of bin 2 pulled from a counter
// (heavy vertices spread over whichever CTAs are free), then warp items
// (bin 1 chunks, bin 0 groups) dealt round robin over all warps of the grid.
template <bool kBatch, bool kStaged = false>
__device__ void expand_top_down(const TraversalParams& P, Stage<kBatch>& S, const LevelShape& L,
                                int level, bool bitmap = false) {
    __shared__ long long s_item;
    const int slot = level % 3, nslot = (level + 1) % 3;
    const int cur = level & 1, nxt = cur ^ 1;
    const int warp = threadIdx.x >> 5;
    if (L.n_cta > 0) {
        for (;;) {
            if (threadIdx.x == 0) s_item = (long long)atomicAdd(&P.ctl[slot].work, 1u);
            __syncthreads();
            const long long item = s_item;
            __syncthreads();
            if (item >= L.n_cta) break;
            expand_cta_chunk<kBatch, kStaged>(P, S, cur, item, L.k_cta, L.cnt[2], L.edges[2], level, nxt,
                                     nslot);
        }
    }
    const long long nwarps = (long long)gridDim.x * kWarps;
    const long long gw = (long long)blockIdx.x * kWarps + warp;
    // bitmap mode: the light bin's groups are replaced by bitmap tiles
    // starting at the first tile that can hold a light vertex
    long long tile0 = 0, tiles = 0;
    if (!kLean && !kBatch && bitmap) {
        tile0 = P.bitmap_from / 1024;
        tiles = ((P.n + 31) / 32 + 31) / 32 - tile0;
    }
    const long long small_items = (!kLean && !kBatch && bitmap) ? tiles : L.groups_small;
    const long long w1 = L.items_w1, w12 = w1 + L.items_w2;
    const long long witems = w12 + small_items;
    const int sh_warp = __ffs(P.chunk_warp) - 1, sh_cta = __ffs(P.chunk_cta) - 1;
    for (long long it = gw; it < witems; it += nwarps) {
        if (it < w12) {
            const bool b2 = it >= w1;
            const int shw = b2 ? L.sh_w2 : L.sh_w1;
            const long long cs = (b2 ? it - w1 : it) << shw;
            const long long E = b2 ? L.edges[2] : L.edges[1];
            expand_warp_range<kBatch>(P, S, P.q[cur][b2 ? 2 : 1], b2 ? sh_cta : sh_warp, cs,
                                      min(cs + (1ll << shw), E), b2 ? L.cnt[2] : L.cnt[1], level,
                                      nxt, nslot);
        } else if constexpr (!kBatch) {
#if !BFS_LEAN_PATHS
            if (bitmap)
                expand_bitmap_tile(P, S, tile0 + (it - w12), level, nxt, nslot);
            else
#endif
                expand_small_group<kBatch>(P, S, cur, it - w12, L.cnt[0], level, nxt, nslot);
        } else {
            expand_small_group<kBatch>(P, S, cur, it - w12, L.cnt[0], level, nxt, nslot);
        }
    }
}

// Byte-uniform fill (0x00 or 0xff patterns): scalar bytes up to a 16-byte
// boundary, 16-byte stores for the body, scalar bytes for the tail.
__device__ void fill_bytes(void* ptr, long long nbytes, unsigned char value, long long tid,
                           long long nthreads) {
    unsigned char* p = static_cast<unsigned char*>(ptr);
    const long long head = min(nbytes, (long long)((16 - ((uintptr_t)p & 15)) & 15));
    for (long long i = tid; i < head; i += nthreads) p[i] = value;
    const long long nvec = (nbytes - head) / 16;
    int4* pv = reinterpret_cast<int4*>(p + head);
    const int w = (int)(value * 0x01010101u);
    const int4 v4 = make_int4(w, w, w, w);
    for (long long i = tid; i < nvec; i += nthreads) pv[i] = v4;
    for (long long i = head + nvec * 16 + tid; i < nbytes; i += nthreads) p[i] = value;
}

}  // inline namespace
}  // namespace bfs
