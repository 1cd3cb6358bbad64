// Seed cleaning and the quality filter with duplicate removal (Sec. 2.2: seeds are processed in
// parallel, so hits consumed by earlier tracks cannot be masked; duplicates are removed from the
// resulting tracks).
//
// Both compare items (rows of hit ids; < 0 = none) that share hits.  An index of the items on
// each hit (counting sort by hit id: ranks, scan, fill) lists, for every hit of an item, the
// other items on it; one thread per item walks those lists and counts, for every other item it
// meets, the hits on which it met it.  The decision is an OR over the better items, so it does not
// depend on the order in which the index lists them.
//   seeds: a seed is dropped if a seed of lower index shares at least two of its three hits;
//   tracks: a track with fewer than min_hits hits is dropped, and a track is dropped if a better
//   track (higher score, equal score and lower index) shares at least frac x the smaller hit
//   count.  Every item is judged against all others (not transitively).
#include "internal.h"

namespace mk {

namespace {

constexpr int kThreads = 256;

// Counts the items on every hit; rank gets each entry's place among them, so that the fill needs
// no second pass of atomics.
__global__ void k_item_hit_count(int64_t n_entries, const int* __restrict__ hits, int64_t n_hits, int* cnt,
                                 int* __restrict__ rank) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n_entries; q += (int64_t)gridDim.x * blockDim.x) {
        const int h = hits[q];
        if (h >= 0 && h < n_hits) rank[q] = atomicAdd(cnt + h, 1);
    }
}

__global__ void k_item_hit_fill(int64_t total, int width, const int* __restrict__ hits, int64_t n_hits,
                                const int* __restrict__ off, const int* __restrict__ rank, int* __restrict__ items) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const int h = hits[q];
        if (h >= 0 && h < n_hits) items[off[h] + rank[q]] = (int)(q / width);
    }
}

__device__ __forceinline__ int row_hits(const int* __restrict__ a, int width, int64_t n_hits) {
    int c = 0;
    for (int i = 0; i < width; ++i) c += (a[i] >= 0 && a[i] < n_hits);
    return c;
}

__device__ __forceinline__ int row_shared(const int* __restrict__ a, const int* __restrict__ b, int width,
                                          int64_t n_hits) {
    int s = 0;
    for (int i = 0; i < width; ++i) {
        const int h = a[i];
        if (h < 0 || h >= n_hits) continue;
        for (int j = 0; j < width; ++j)
            if (b[j] == h) {
                ++s;
                break;
            }
    }
    return s;
}

// Seeds: t is dropped if a seed of lower index shares at least two of its three hits.  Rows of three
// are compared where they are met, up to the first that drops t: 119 us for cleaning 192,000 seeds with 8
// to 64 of them on every hit, against 238 when the seeds met were counted to the end of the lists
// (20,000 seeds on the same two hits: 3.3 ms against 8.2).
__global__ void __launch_bounds__(kThreads) k_seed_decide(int n, int width, const int* __restrict__ hits,
                                                          int64_t n_hits, const int* __restrict__ off,
                                                          const int* __restrict__ items, int* keep) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const int* a = hits + (int64_t)t * width;
    bool drop = false;
    for (int i = 0; i < width && !drop; ++i) {
        const int h = a[i];
        if (h < 0 || h >= n_hits) continue;
        const int q1 = __ldg(off + h + 1);
        for (int q = __ldg(off + h); q < q1 && !drop; ++q) {
            const int u = __ldg(items + q);
            drop = u < t && row_shared(a, hits + (int64_t)u * width, width, n_hits) >= 2;
        }
    }
    keep[t] = drop ? 0 : 1;
}

// Whether track t (na hits) is dropped by the better track u, with s of t's hits on u.
__device__ __forceinline__ bool dropped_by(int u, int s, int na, int width, const int* __restrict__ hits,
                                           int64_t n_hits, float frac) {
    if ((double)s >= (double)frac * (double)na) return true;   // enough of t's own hits, whatever u has
    const int nb = row_hits(hits + (int64_t)u * width, width, n_hits);
    return nb < na && (double)s >= (double)frac * (double)nb;
}

// Tracks (score, frac, min_hits).
//
// The thread keeps the first kSeen tracks it meets in registers, with the number of its hits on
// each: the shared count comes from the index itself and no two rows are compared.  Better tracks
// beyond kSeen (a track on hits of many others) are compared row by row in a second walk, up to the
// first that drops t; a track on a hit of more than kCrowd goes to that walk at once.
// Bound by the gathers off[h] and items[...] (one 32-byte sector each per hit).  Comparing the rows
// at every meeting instead left 2.3 of 32 lanes active and took 451M warp instructions for 320k
// tracks of 22 layers; with it, and a second pass of atomics in the fill, cleaning 1.28M seeds and
// filtering 1.28M tracks (two per particle) took 2.96 ms, against 0.96 ms now.  With tens of tracks on
// every hit that comparison, which ends with the first better track, is the shorter way: 32 tracks per
// particle (20,000 in all) 1,178 us against 1,310, 64 (9,984) 908 against 1,189; kCrowd = 12 made 8 per
// particle 25% slower, 48 the 32 per particle 10%.
constexpr int kSeen = 6, kCrowd = 24;

__global__ void __launch_bounds__(kThreads) k_track_decide(int n, int width, const int* __restrict__ hits,
                                                           const float* __restrict__ score, int64_t n_hits,
                                                           int min_hits, float frac, const int* __restrict__ off,
                                                           const int* __restrict__ items, int* keep) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const int* a = hits + (int64_t)t * width;
    int first = 0;   // the row's hits, as far as min_hits
    for (int i = 0; i < width && first < min_hits; ++i) first += a[i] >= 0 && a[i] < n_hits;
    if (first < min_hits) {
        keep[t] = 0;
        return;
    }
    int na = 0;
    const float st = score[t];
    auto better = [&](int u) {
        const float su = __ldg(score + u);
        return su > st || (su == st && u < t);
    };
    int seen[kSeen], cnt[kSeen], last[kSeen];   // track, t's hits on it, the last of them (cnt < 0: not better)
#pragma unroll
    for (int k = 0; k < kSeen; ++k) {
        seen[k] = -1;
        cnt[k] = 0;
        last[k] = -1;
    }
    int n_seen = 0;
    bool more = false;
    for (int i = 0; i < width; ++i) {
        const int h = a[i];
        if (h < 0 || h >= n_hits) continue;
        ++na;
        const int q0 = __ldg(off + h), q1 = __ldg(off + h + 1);
        if (q1 - q0 > kCrowd) {
            na = row_hits(a, width, n_hits);
#pragma unroll
            for (int k = 0; k < kSeen; ++k) {
                seen[k] = -1;
                cnt[k] = 0;
            }
            more = true;
            break;
        }
        for (int q = q0; q < q1; ++q) {
            const int u = __ldg(items + q);
            if (u == t) continue;
            bool found = false;
#pragma unroll
            for (int k = 0; k < kSeen; ++k)
                if (seen[k] == u) {
                    found = true;
                    if (last[k] != i && cnt[k] >= 0) ++cnt[k];   // a track may list a hit twice
                    last[k] = i;
                }
            if (found) continue;
            const bool b = better(u);
            if (n_seen < kSeen) {
#pragma unroll
                for (int k = 0; k < kSeen; ++k)
                    if (k == n_seen) {
                        seen[k] = u;
                        cnt[k] = b ? 1 : -1;
                        last[k] = i;
                    }
                ++n_seen;
            } else {
                more = more || b;
            }
        }
    }
    bool drop = false;
#pragma unroll
    for (int k = 0; k < kSeen; ++k)
        if (!drop && cnt[k] > 0) drop = dropped_by(seen[k], cnt[k], na, width, hits, n_hits, frac);
    if (more && !drop) {
        for (int i = 0; i < width && !drop; ++i) {
            const int h = a[i];
            if (h < 0 || h >= n_hits) continue;
            const int q1 = off[h + 1];
            for (int q = off[h]; q < q1 && !drop; ++q) {
                const int u = items[q];
                if (u == t) continue;
                bool in_seen = false;
#pragma unroll
                for (int k = 0; k < kSeen; ++k) in_seen = in_seen || seen[k] == u;
                if (in_seen || !better(u)) continue;
                drop = dropped_by(u, row_shared(a, hits + (int64_t)u * width, width, n_hits), na, width, hits, n_hits,
                                  frac);
            }
        }
    }
    keep[t] = drop ? 0 : 1;
}

}  // namespace

size_t clean_scratch_ints(int n, int width, int64_t n_hits) {
    // counts/offsets (n_hits + 1), ranks and items (n x width each), scan scratch
    return (size_t)n_hits + 1 + 2 * (size_t)n * width + scan_tmp_ints(n_hits) + 64;
}

cudaError_t launch_item_decide(cudaStream_t st, int mode, int n, int width, const int* hits, const float* score,
                               int64_t n_hits, int min_hits, float frac, int* scratch, int* keep, int n_sms) {
    if (n == 0) return cudaSuccess;
    const int64_t entries = (int64_t)n * width;
    int* off = scratch;
    int* rank = off + (n_hits + 1);
    int* items = rank + entries;
    int* tmp = items + entries;
    cudaError_t e = cudaMemsetAsync(off, 0, 4 * ((size_t)n_hits + 1), st);
    if (e != cudaSuccess) return e;
    const int grid = 8 * n_sms;
    k_item_hit_count<<<grid, kThreads, 0, st>>>(entries, hits, n_hits, off, rank);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = exclusive_scan(st, off, off, n_hits, tmp)) != cudaSuccess) return e;   // off[n_hits] = total
    k_item_hit_fill<<<grid, kThreads, 0, st>>>(entries, width, hits, n_hits, off, rank, items);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int blocks = (n + kThreads - 1) / kThreads;
    if (mode == 0)
        k_seed_decide<<<blocks, kThreads, 0, st>>>(n, width, hits, n_hits, off, items, keep);
    else
        k_track_decide<<<blocks, kThreads, 0, st>>>(n, width, hits, score, n_hits, min_hits, frac, off, items, keep);
    return cudaGetLastError();
}

}  // namespace mk
