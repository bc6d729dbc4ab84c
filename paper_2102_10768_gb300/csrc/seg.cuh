// Segmented exclusive scans with decoupled look-back (prims.cuh): many
// independent index spaces ("segments": one per query vertex or query edge of
// a batch) in one launch.
//
// The tiles of all segments form one global tile sequence: segment s owns
// tiles tile_off[s] .. tile_off[s+1]-1 (at least one, so that an empty
// segment still reports a zero count).  Blocks of a persistent grid take
// tiles in that order from one counter.  A tile publishes its aggregate and
// looks back over the earlier tiles of its own segment only, stopping at the
// segment's first tile; every tile it waits on was taken before it by a
// block that is already running, so the wait ends.  It is still bounded by
// the same spin limit as the single-segment form, and running out sets the
// translation unit's look-back error flag.
#pragma once

#include <vector>

#include "prims.cuh"

namespace fast {

// last s with tile_off[s] <= t (the segment owning tile t; the empty
// segments before it share its offset)
__device__ __forceinline__ int seg_of_tile(const int64_t* __restrict__ tile_off, int nseg, int64_t t) {
    int lo = 0, hi = nseg;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (tile_off[mid] <= t) lo = mid; else hi = mid;
    }
    return lo;
}

// The same by the 32 lanes of a warp together, which all pass the same t: 33
// parts per round, so that ten thousand segments take three rounds of one
// load each instead of fourteen dependent loads.
__device__ __forceinline__ int warp_seg_of(const int64_t* __restrict__ tile_off, int nseg, int64_t t) {
    const int lane = threadIdx.x & 31;
    int lo = 0, hi = nseg;
    while (hi - lo > 1) {
        const int p = lo + (int)(((int64_t)(hi - lo) * (lane + 1)) / 33);      // in [lo, hi), ascending in the lane
        const int c = __popc(__ballot_sync(0xffffffffu, tile_off[p] <= t));    // those probes form a prefix
        const int plo = __shfl_sync(0xffffffffu, p, c > 0 ? c - 1 : 0);
        const int phi = __shfl_sync(0xffffffffu, p, c < 32 ? c : 31);
        if (c > 0) lo = plo;
        if (c < 32) hi = phi;
    }
    return lo;
}

// Host side: tile_off[0..nseg] for segments of n_s indices, tiles of `tile`
// indices, at least one tile per segment.
inline std::vector<int64_t> seg_tile_offsets(const std::vector<int64_t>& n, int64_t tile) {
    std::vector<int64_t> off(n.size() + 1, 0);
    for (size_t i = 0; i < n.size(); i++) off[i + 1] = off[i] + std::max<int64_t>(1, ceil_div(n[i], tile));
    return off;
}

// ------------------------------------------------------------------- scan

// Exclusive scan of every segment, with what is scanned and where it goes
// given by F:
//   int64_t n(int s)                              items of segment s
//   T load(int s, int64_t i)                      item i (each is loaded once)
//   void values(int s, const T (&x)[kScanItems])  a thread's items (zeros past the end), by whole warps
//   void store(int s, int64_t i, T excl, T v)     its exclusive prefix and itself
//   void total(int s, T tot)                      the segment's sum
// st: one status word per tile, tile_ctr after them, all zero at launch.
template <class T, class F>
__device__ __forceinline__ void seg_scan(F& f, const int64_t* __restrict__ tile_off, int nseg, unsigned long long* st,
                                         unsigned int* tile_ctr) {
    __shared__ T tmp[kScanBlock / 32 + 1];
    __shared__ int64_t s_t, s_excl, s_first;
    __shared__ int s_seg;
    const int64_t total = tile_off[nseg];
    for (;;) {
        if (threadIdx.x < 32) {
            int64_t t = 0;
            if (threadIdx.x == 0) t = (int64_t)atomicAdd(tile_ctr, 1u);
            t = __shfl_sync(0xffffffffu, t, 0);
            const int sg = t < total ? warp_seg_of(tile_off, nseg, t) : 0;
            if (threadIdx.x == 0) {
                s_t = t;
                s_seg = sg;
                s_first = tile_off[sg];
            }
        }
        __syncthreads();
        const int64_t t = s_t;
        if (t >= total) break;
        const int sg = s_seg;
        const int64_t lt = t - s_first, n = f.n(sg);
        const int64_t tb = lt * kScanTile;
        if (tb >= n) {                                     // empty segment
            if (lt == 0 && threadIdx.x == 0) f.total(sg, T(0));
            __syncthreads();
            continue;
        }
        const int64_t base = tb + (int64_t)threadIdx.x * kScanItems;
        T v[kScanItems], x[kScanItems];
#pragma unroll
        for (int i = 0; i < kScanItems; i++) x[i] = v[i] = base + i < n ? f.load(sg, base + i) : T(0);
        f.values(sg, x);
        const T tot = block_exclusive_scan<T, kScanBlock, kScanItems>(v, tmp);
        if (threadIdx.x < 32) {
            const int64_t excl = tile_publish(st + s_first, lt, (int64_t)tot);
            if (threadIdx.x == 0) {
                s_excl = excl;
                if (tb + kScanTile >= n) f.total(sg, (T)(excl + (int64_t)tot));
            }
        }
        __syncthreads();
        const T off = (T)s_excl;
#pragma unroll
        for (int i = 0; i < kScanItems; i++)
            if (base + i < n) f.store(sg, base + i, v[i] + off, x[i]);
        __syncthreads();
    }
}

}  // namespace fast
