// bfs_relabel.cu -- degree-ordered renumbering of an uploaded graph.
//
// Vertices are ordered by logarithmic degree bucket, heaviest first (bucket
// = floor(log2 deg) + 1, 0 for isolated vertices: the same log2 classes as
// the paper's Logarithmic Radix Binning, used here for layout), stable by
// the caller's id inside a bucket.  Hubs then get the smallest ids, so the
// visited-bitmap words, row offsets and distances that most edges touch
// sit together at the front of each array.  Results are always written in
// the caller's numbering (new2old on every dist/parent write).
//
// Steps (all on the device):
//   1. per tile of 1024 vertices, count vertices per bucket
//   2. exclusive scan of the bucket-major count table -> tile offsets
//   3. stable scatter: new2old[pos] = v, old2new[v] = pos
//   4. new offsets = exclusive scan of deg[new2old[i]]
//   5. new columns: row of new2old[i] copied with old2new applied, heavy
//      neighbours first
#include <cuda_runtime.h>

#include <cstdint>

#include "bfs_internal.h"

namespace bfs {

constexpr int kRelTile = 1024;
constexpr int kRelThreads = 256;
constexpr int kBuckets = 33;  // deg 0, [1,2), [2,4), ..., [2^31, ...)

__device__ __forceinline__ int rel_key(long long deg) {
    // ascending key = descending degree bucket
    const int bucket = deg <= 0 ? 0 : 64 - __clzll((unsigned long long)deg);  // floor(log2)+1
    return (kBuckets - 1) - min(bucket, kBuckets - 1);
}

__global__ void rel_count_kernel(const int64_t* off, long long n, long long ntiles,
                                 unsigned long long* counts) {
    __shared__ unsigned s_cnt[kBuckets];
    for (int i = threadIdx.x; i < kBuckets; i += blockDim.x) s_cnt[i] = 0;
    __syncthreads();
    const long long t = blockIdx.x;
    for (int k = threadIdx.x; k < kRelTile; k += blockDim.x) {
        const long long v = t * kRelTile + k;
        if (v < n) atomicAdd(&s_cnt[rel_key(off[v + 1] - off[v])], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kBuckets; i += blockDim.x) counts[(long long)i * ntiles + t] = s_cnt[i];
}

// Stable scatter of one tile: sub-batches of 256 vertices in order; inside a
// sub-batch, warps in order; inside a warp, lanes in order.
__global__ void rel_scatter_kernel(const int64_t* off, long long n, long long ntiles,
                                   const unsigned long long* offsets, int32_t* new2old,
                                   int32_t* old2new) {
    __shared__ unsigned long long s_base[kBuckets];
    __shared__ unsigned s_warp[kRelThreads / 32][kBuckets];
    const long long t = blockIdx.x;
    const int warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < kBuckets; i += blockDim.x) s_base[i] = offsets[(long long)i * ntiles + t];
    __syncthreads();
    for (int sub = 0; sub < kRelTile; sub += kRelThreads) {
        const long long v = t * kRelTile + sub + threadIdx.x;
        const bool ok = v < n;
        const int key = ok ? rel_key(off[v + 1] - off[v]) : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        unsigned lt;
        asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt));
        const int rank_in_warp = __popc(peers & lt);
        for (int i = threadIdx.x; i < (kRelThreads / 32) * kBuckets; i += blockDim.x)
            (&s_warp[0][0])[i] = 0;
        __syncthreads();
        if (ok && rank_in_warp == 0) s_warp[warp][key] = __popc(peers);
        __syncthreads();
        if (ok) {
            unsigned before = 0;
            for (int w = 0; w < warp; ++w) before += s_warp[w][key];
            const long long pos = (long long)s_base[key] + before + rank_in_warp;
            new2old[pos] = (int32_t)v;
            old2new[v] = (int32_t)pos;
        }
        __syncthreads();
        if (threadIdx.x < kBuckets) {
            unsigned tot = 0;
            for (int w = 0; w < kRelThreads / 32; ++w) tot += s_warp[w][threadIdx.x];
            s_base[threadIdx.x] += tot;
        }
        __syncthreads();
    }
}

__global__ void rel_newdeg_kernel(const int64_t* off, const int32_t* new2old, long long n,
                                  int64_t* out) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const int32_t o = new2old[i];
        out[i] = off[o + 1] - off[o];
    }
}

// Vertices of each cut class come first in the new order: below[c] of them
// (key = 32 - bucket, bucket = floor(log2 deg) + 1: deg >= 2^k <=> key <= 31 - k).
// `reach` starts at none; rel_columns_kernel raises it.
__global__ void rel_bounds_kernel(const unsigned long long* key_start, long long ntiles,
                                  CutBounds* out) {
    if (threadIdx.x < kCutClasses) {
        constexpr int deg[kCutClasses] = {kCutDegree[0], kCutDegree[1], kCutDegree[2], kCutDegree[3],
                                          kCutDegree[4], kCutDegree[5], kCutDegree[6], kCutDegree[7]};
        const int lg = 31 - __clz(deg[threadIdx.x]);
        out->below[threadIdx.x] = (long long)key_start[(long long)(32 - lg) * ntiles];
    }
    if (threadIdx.x == 0) out->reach = 0;
}

// One warp per new row; columns renamed through old2new and each row stably
// partitioned by the degree class of the neighbour, heaviest first (new ids
// are in decreasing degree-bucket order, so the classes are id ranges).  A
// bottom-up level checks neighbours in row order, and the heavy ones are the
// most likely in the frontier; a top-down level that knows every vertex
// below a class's bound to be visited skips the row's entries up to that
// class -- cut[c][row], when asked for, says how many they are.  The largest
// target of all rows bounds the vertices that a traversal can reach.
//
// Bound by the random reads of old2new and, on long rows, by the chain of one
// warp: 128 entries are read together, and the 9 classes of a chunk are told
// apart by the ballots of their number's 4 bits (a ballot per class and one
// chunk at a time: upload of scale 22, 16 edges per vertex, 13.3 ms, of a star
// of 2 M vertices 113; now 8.3 and 49).
constexpr int kStep = 4;   // 32-entry chunks of a row in flight
__device__ __forceinline__ void read_entries(const int32_t* old2new, const int32_t* row, unsigned d,
                                             unsigned k, int32_t (&x)[kStep]) {
    int32_t c[kStep];
#pragma unroll
    for (int s = 0; s < kStep; ++s) c[s] = k + 32 * s < d ? row[k + 32 * s] : 0;
#pragma unroll
    for (int s = 0; s < kStep; ++s) x[s] = k + 32 * s < d ? old2new[c[s]] : 0;
}
__global__ void rel_columns_kernel(const int64_t* off, const int32_t* col, const int32_t* new2old,
                                   const int32_t* old2new, const int64_t* new_off, long long n,
                                   CutBounds* bounds, uint16_t* cut, int32_t* new_col) {
    static_assert(kCutClasses + 1 < 16, "a class and \"no entry\" fit in 4 bits");
    int bound[kCutClasses];
#pragma unroll
    for (int c = 0; c < kCutClasses; ++c) bound[c] = (int)bounds->below[c];
    int reach = 0;
    const long long nwarps = (long long)gridDim.x * (blockDim.x / 32);
    const int lane = threadIdx.x & 31;
    unsigned lt;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt));
    auto class_of = [&](int32_t x, bool ok) -> int {
        int g = 0;
#pragma unroll
        for (int c = 0; c < kCutClasses; ++c) g += x >= bound[c] ? 1 : 0;
        return ok ? g : 15;
    };
    // the lanes whose class has the bits of `like`, from the ballots of the 4 bits
    auto lanes_like = [](const unsigned (&bit)[4], int like) -> unsigned {
        unsigned m = 0xffffffffu;
#pragma unroll
        for (int k = 0; k < 4; ++k) m &= (like >> k) & 1 ? bit[k] : ~bit[k];
        return m;
    };
    auto ballots = [](int g, unsigned (&bit)[4]) {
#pragma unroll
        for (int k = 0; k < 4; ++k) bit[k] = __ballot_sync(0xffffffffu, (g >> k) & 1);
    };
    for (long long i = (long long)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); i < n;
         i += nwarps) {
        const int32_t o = new2old[i];
        const long long b = off[o], nb = new_off[i];
        // (rows of 2^31 and more entries are refused after the renumbering)
        const unsigned d = (unsigned)min((long long)off[o + 1] - b, 0x7fffffffll);
        if (d == 0 && cut == nullptr) continue;
        // lane c counts class c, then holds where its next entry goes in the row
        int mine = 0;
        int32_t x[kStep];
        unsigned bit[4];
        for (unsigned k0 = 0; k0 < d; k0 += 32 * kStep) {
            read_entries(old2new, col + b, d, k0 + lane, x);
#pragma unroll
            for (int s = 0; s < kStep; ++s) {
                if (k0 + 32 * s >= d) break;
                const bool ok = k0 + 32 * s + lane < d;
                if (ok) reach = max(reach, x[s] + 1);
                ballots(class_of(x[s], ok), bit);
                mine += __popc(lanes_like(bit, lane));
            }
        }
        if (lane > kCutClasses) mine = 0;   // lane 15 counted what is no entry
        int incl = mine;
#pragma unroll
        for (int s = 1; s < 16; s <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, s);
            if (lane >= s) incl += y;
        }
        if (cut && lane < kCutClasses)
            cut[lane * n + i] = (uint16_t)(incl < 65535 ? incl : 65535);
        int at = incl - mine;
        for (unsigned k0 = 0; k0 < d; k0 += 32 * kStep) {
            // a row of one step still holds its entries
            if (d > 32 * kStep) read_entries(old2new, col + b, d, k0 + lane, x);
#pragma unroll
            for (int s = 0; s < kStep; ++s) {
                if (k0 + 32 * s >= d) break;
                const bool ok = k0 + 32 * s + lane < d;
                const int g = class_of(x[s], ok);
                ballots(g, bit);
                const int base = __shfl_sync(0xffffffffu, at, g);
                if (ok) new_col[nb + base + __popc(lanes_like(bit, g) & lt)] = x[s];
                at += __popc(lanes_like(bit, lane));
            }
        }
    }
    reach = __reduce_max_sync(0xffffffffu, reach);
    if (lane == 0 && reach > 0) atomicMax(&bounds->reach, (long long)reach);
}

// ---------------------------------------------------- exclusive scan (int64)
// Three passes: per-block sums, scan of the block sums in one block, then
// each block scans its segment and adds its base.  out may alias in.
constexpr int kScanThreads = 512;
constexpr int kScanPerThread = 8;
constexpr long long kScanBlock = (long long)kScanThreads * kScanPerThread;

__device__ __forceinline__ long long block_excl_scan(long long x, long long* total) {
    __shared__ long long s_w[kScanThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long incl = x;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) s_w[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        long long w = lane < kScanThreads / 32 ? s_w[lane] : 0;
        long long wi = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, wi, d);
            if (lane >= d) wi += y;
        }
        if (lane < kScanThreads / 32) s_w[lane] = wi - w;
        if (lane == kScanThreads / 32 - 1) *total = wi;
    }
    __syncthreads();
    const long long r = s_w[warp] + incl - x;
    __syncthreads();
    return r;
}

__global__ void scan_block_sums(const int64_t* in, long long n, int64_t* sums) {
    __shared__ long long s_tot;
    const long long base = (long long)blockIdx.x * kScanBlock + (long long)threadIdx.x * kScanPerThread;
    long long acc = 0;
    for (int k = 0; k < kScanPerThread; ++k)
        if (base + k < n) acc += in[base + k];
    block_excl_scan(acc, &s_tot);
    if (threadIdx.x == 0) sums[blockIdx.x] = s_tot;
}

__global__ void scan_sums_single(int64_t* sums, long long nblocks) {
    __shared__ long long s_tot;
    long long carry = 0;
    for (long long start = 0; start < nblocks; start += kScanThreads) {
        const long long i = start + threadIdx.x;
        const long long x = i < nblocks ? sums[i] : 0;
        const long long ex = block_excl_scan(x, &s_tot);
        if (i < nblocks) sums[i] = carry + ex;
        __syncthreads();
        carry += s_tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) sums[nblocks] = carry;
}

__global__ void scan_apply(const int64_t* in, long long n, const int64_t* sums, int64_t* out) {
    __shared__ long long s_tot;
    const long long base = (long long)blockIdx.x * kScanBlock + (long long)threadIdx.x * kScanPerThread;
    long long v[kScanPerThread];
    long long acc = 0;
    for (int k = 0; k < kScanPerThread; ++k) {
        v[k] = base + k < n ? in[base + k] : 0;
        acc += v[k];
    }
    long long run = block_excl_scan(acc, &s_tot) + sums[blockIdx.x];
    for (int k = 0; k < kScanPerThread; ++k) {
        if (base + k < n) out[base + k] = run;
        run += v[k];
    }
}

// Exclusive scan of n int64 values; out[n] receives the total.  tmp needs
// ceil(n / 4096) + 1 int64.
cudaError_t exclusive_scan_i64(const int64_t* in, long long n, int64_t* out, int64_t* tmp,
                               cudaStream_t s) {
    const long long nb = (n + kScanBlock - 1) / kScanBlock;
    if (nb > 0) {
        scan_block_sums<<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, tmp);
        scan_sums_single<<<1, kScanThreads, 0, s>>>(tmp, nb);
        scan_apply<<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, tmp, out);
    } else {
        cudaMemsetAsync(tmp, 0, sizeof(int64_t), s);
    }
    // out[n] = total
    return cudaMemcpyAsync(out + n, tmp + nb, sizeof(int64_t), cudaMemcpyDeviceToDevice, s);
}

// Scratch sizes (bytes) the relabel needs beyond the new graph arrays; the
// first 16 n of them hold the rows' class counts when those are kept.
size_t relabel_scratch_bytes(long long n) {
    const long long ntiles = (n + kRelTile - 1) / kRelTile;
    const long long table = (long long)kBuckets * ntiles;
    const long long big = table > n ? table : n;
    return (size_t)(2 * (big + 1) * 8 + ((big + kScanBlock - 1) / kScanBlock + 2) * 8) + 1024;
}

// Builds new2old/old2new and the renumbered CSR (new_off[n+1], new_col[nnz]).
// With keep_cut the rows' class counts, uint16[kCutClasses][n], are left at
// the start of scratch, which the caller then keeps; bounds (host) are written
// when the stream has been waited for.
cudaError_t relabel_graph(const int64_t* off, const int32_t* col, long long n, long long nnz,
                          int sms, int32_t* new2old, int32_t* old2new, int64_t* new_off,
                          int32_t* new_col, void* scratch, bool keep_cut, CutBounds* bounds,
                          cudaStream_t s) {
    static_assert(kCutClasses * sizeof(uint16_t) <= 2 * sizeof(int64_t), "the counts fit in a and b");
    static_assert(sizeof(CutBounds) <= 1024, "the bounds fit in tmp");
    const long long ntiles = (n + kRelTile - 1) / kRelTile;
    const long long table = (long long)kBuckets * ntiles;
    const long long big = table > n ? table : n;
    int64_t* a = static_cast<int64_t*>(scratch);
    int64_t* b = a + big + 1;
    int64_t* tmp = b + big + 1;
    rel_count_kernel<<<(unsigned)ntiles, kRelThreads, 0, s>>>(off, n, ntiles,
                                                               reinterpret_cast<unsigned long long*>(a));
    cudaError_t e = exclusive_scan_i64(a, table, b, tmp, s);
    if (e != cudaSuccess) return e;
    rel_scatter_kernel<<<(unsigned)ntiles, kRelThreads, 0, s>>>(
        off, n, ntiles, reinterpret_cast<const unsigned long long*>(b), new2old, old2new);
    rel_newdeg_kernel<<<sms * 4, 256, 0, s>>>(off, new2old, n, a);
    e = exclusive_scan_i64(a, n, new_off, tmp, s);
    if (e != cudaSuccess) return e;
    // the scan's scratch is free again: the class bounds go there; after them
    // a and b are free too, for the class counts
    CutBounds* d_bounds = reinterpret_cast<CutBounds*>(tmp);
    uint16_t* cut = keep_cut ? static_cast<uint16_t*>(scratch) : nullptr;
    rel_bounds_kernel<<<1, 32, 0, s>>>(reinterpret_cast<const unsigned long long*>(b), ntiles, d_bounds);
    rel_columns_kernel<<<sms * 8, 256, 0, s>>>(off, col, new2old, old2new, new_off, n, d_bounds, cut,
                                                new_col);
    (void)nnz;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return cudaMemcpyAsync(bounds, d_bounds, sizeof(CutBounds), cudaMemcpyDeviceToHost, s);
}

}  // namespace bfs
