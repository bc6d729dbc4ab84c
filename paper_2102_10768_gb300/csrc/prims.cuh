// Device-wide building blocks written for this library: exclusive scan,
// ordered predicate compaction over an index space (two passes: the output's
// size is known between them), the decoupled look-back of the segmented
// scans, and a stable LSD radix sort of 64-bit keys.  All are stream-ordered and take
// their scratch through dalloc on the caller's stream.
#pragma once

#include <algorithm>
#include <type_traits>
#include <utility>

#include "common.cuh"

namespace fast {

constexpr int kScanBlock = 512;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanBlock * kScanItems;

// Block-wide exclusive scan of ITEMS values per thread (blocked layout:
// thread t holds tile positions t*ITEMS .. t*ITEMS+ITEMS-1).  Returns the
// block total.  `warp_tmp` needs BLOCK/32 entries of shared memory.
template <class T, int BLOCK, int ITEMS>
__device__ __forceinline__ T block_exclusive_scan(T (&v)[ITEMS], T* warp_tmp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T local = 0;
#pragma unroll
    for (int i = 0; i < ITEMS; i++) { T x = v[i]; v[i] = local; local += x; }
    T incl = local;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        T t = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += t;
    }
    if (lane == 31) warp_tmp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        constexpr int NW = BLOCK / 32;
        T x = lane < NW ? warp_tmp[lane] : T(0);
        T y = x;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            T t = __shfl_up_sync(0xffffffffu, y, off);
            if (lane >= off) y += t;
        }
        if (lane < NW) warp_tmp[lane] = y - x;       // exclusive
        if (lane == NW - 1) warp_tmp[NW] = y;         // total
    }
    __syncthreads();
    T base = warp_tmp[warp] + (incl - local);
#pragma unroll
    for (int i = 0; i < ITEMS; i++) v[i] += base;
    T total = warp_tmp[BLOCK / 32];
    __syncthreads();
    return total;
}

template <class T>
__global__ void k_scan_partials(const T* __restrict__ in, int64_t n, T* __restrict__ partials) {
    __shared__ T tmp[kScanBlock / 32 + 1];
    int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    T v[kScanItems];
#pragma unroll
    for (int i = 0; i < kScanItems; i++) v[i] = (base + i < n) ? in[base + i] : T(0);
    T tot = block_exclusive_scan<T, kScanBlock, kScanItems>(v, tmp);
    if (threadIdx.x == 0) partials[blockIdx.x] = tot;
}

template <class T>
__global__ void k_scan_apply(const T* __restrict__ in, T* __restrict__ out, int64_t n,
                             const T* __restrict__ partials, T* __restrict__ total) {
    __shared__ T tmp[kScanBlock / 32 + 1];
    int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    T v[kScanItems];
#pragma unroll
    for (int i = 0; i < kScanItems; i++) v[i] = (base + i < n) ? in[base + i] : T(0);
    T tot = block_exclusive_scan<T, kScanBlock, kScanItems>(v, tmp);
    T off = partials ? partials[blockIdx.x] : T(0);
#pragma unroll
    for (int i = 0; i < kScanItems; i++)
        if (base + i < n) out[base + i] = v[i] + off;
    if (total && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total = off + tot;
}

// out[i] = in[0] + ... + in[i-1]; *total (device, nullable) = sum of all.
// in and out may alias.
template <class T>
int scan_exclusive(const T* in, T* out, int64_t n, T* total, cudaStream_t s) {
    if (n <= 0) {
        if (total) FAST_CUDA(cudaMemsetAsync(total, 0, sizeof(T), s));
        return FAST_OK;
    }
    int64_t nb = ceil_div(n, kScanTile);
    if (nb == 1) {
        k_scan_apply<T><<<1, kScanBlock, 0, s>>>(in, out, n, (const T*)nullptr, total);
        note_launch();
        FAST_CUDA(cudaGetLastError());
        return FAST_OK;
    }
    T* part = nullptr;
    FAST_TRY(dalloc(&part, nb, s));
    k_scan_partials<T><<<(unsigned)nb, kScanBlock, 0, s>>>(in, n, part);
    note_launch();
    int rc = cudaGetLastError() == cudaSuccess ? FAST_OK : set_error(FAST_ERR_CUDA, "scan partials launch");
    if (rc == FAST_OK) rc = scan_exclusive<T>(part, part, nb, (T*)nullptr, s);
    if (rc == FAST_OK) {
        k_scan_apply<T><<<(unsigned)nb, kScanBlock, 0, s>>>(in, out, n, part, total);
        note_launch();
        if (cudaGetLastError() != cudaSuccess) rc = set_error(FAST_ERR_CUDA, "scan apply launch");
    }
    dfree(part, s);
    return rc;
}

// ---------------------------------------------------------------- compaction
//
// Ordered compaction over indices [0, n): F::eval(i, val) says whether index
// i is kept and what to write; kept values land in out[] in index order.
// F::begin(i0) is called once per thread before it evaluates indices i0,
// i0+1, ... in increasing order.

constexpr int kCompBlock = 128;
constexpr int kComp2Items = 8;
constexpr int kComp2Tile = kCompBlock * kComp2Items;

template <class F>
__global__ void k_compact_count(F f, int64_t n, int64_t* __restrict__ counts) {
    __shared__ int64_t tmp[kCompBlock / 32 + 1];
    int64_t base = (int64_t)blockIdx.x * kComp2Tile + (int64_t)threadIdx.x * kComp2Items;
    int64_t v[kComp2Items];
    F g = f;
    g.begin(base);
#pragma unroll
    for (int i = 0; i < kComp2Items; i++) {
        typename F::value_type x;
        v[i] = (base + i < n && g.eval(base + i, x)) ? 1 : 0;
    }
    int64_t tot = block_exclusive_scan<int64_t, kCompBlock, kComp2Items>(v, tmp);
    if (threadIdx.x == 0) counts[blockIdx.x] = tot;
}

template <class F>
__global__ void k_compact_write(F f, int64_t n, const int64_t* __restrict__ offs,
                                typename F::value_type* __restrict__ out, int64_t* __restrict__ count) {
    __shared__ int64_t tmp[kCompBlock / 32 + 1];
    int64_t base = (int64_t)blockIdx.x * kComp2Tile + (int64_t)threadIdx.x * kComp2Items;
    int64_t v[kComp2Items];
    typename F::value_type val[kComp2Items];
    F g = f;
    g.begin(base);
#pragma unroll
    for (int i = 0; i < kComp2Items; i++) {
        v[i] = (base + i < n && g.eval(base + i, val[i])) ? 1 : 0;
    }
    int64_t hit[kComp2Items];
#pragma unroll
    for (int i = 0; i < kComp2Items; i++) hit[i] = v[i];
    int64_t tot = block_exclusive_scan<int64_t, kCompBlock, kComp2Items>(v, tmp);
    int64_t off = offs[blockIdx.x];
#pragma unroll
    for (int i = 0; i < kComp2Items; i++) {
        if (hit[i]) out[off + v[i]] = val[i];
    }
    if (count && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *count = off + tot;
}

// Decoupled look-back (segmented scans, seg.cuh).  Blocks take tiles in order
// from a counter.  Each tile publishes its sum (flag AGG), finds its
// exclusive offset by summing predecessors back to the first one whose
// inclusive prefix is known (flag PRE) and publishes its own prefix.  A tile
// only waits on tiles taken before it, by blocks that are already running, so
// the wait ends; it is still bounded, and running out sets g_lookback_err
// (never expected), which the caller turns into an error.
constexpr unsigned long long kLbAgg = 1ull << 62, kLbPre = 2ull << 62, kLbVal = (1ull << 62) - 1;
constexpr int kLbSpins = 1 << 24;
static __device__ int g_lookback_err;

// The exclusive prefix of tile t >= 1, by the 32 lanes of one warp: each
// round reads the status words of the 32 tiles before the window's end at
// once, waits (bounded) until each has published, and stops at the nearest
// one whose inclusive prefix is known, summing the aggregates after it.
__device__ __forceinline__ int64_t lookback_prefix_warp(unsigned long long* st, int64_t t) {
    const int lane = threadIdx.x & 31;
    int64_t excl = 0;
    for (int64_t hi = t - 1;; hi -= 32) {
        const int64_t p = hi - lane;
        unsigned long long w = kLbPre;                 // before tile 0: a prefix of 0
        if (p >= 0) {
            int spins = 0;
            for (;;) {
                w = *(volatile unsigned long long*)(st + p);
                if (w >> 62) break;
                if (++spins > kLbSpins) { atomicExch(&g_lookback_err, 1); w = kLbPre; break; }
                __nanosleep(32);
            }
        }
        const unsigned pre = __ballot_sync(0xffffffffu, (w >> 62) == 2);
        const int stop = pre ? __ffs(pre) - 1 : 31;    // the nearest prefix (lane 0 is tile hi)
        int64_t v = lane <= stop ? (int64_t)(w & kLbVal) : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        excl += v;
        if (pre) break;
    }
    return excl;
}

// Warp 0 of a block: publish tile t's count `tot` (t relative to its
// index space's first tile, status words st), find its exclusive offset and
// publish its inclusive prefix.  Returns the offset on every lane of warp 0.
__device__ __forceinline__ int64_t tile_publish(unsigned long long* st, int64_t t, int64_t tot) {
    const int lane = threadIdx.x & 31;
    int64_t excl = 0;
    if (t == 0) {
        if (lane == 0) atomicExch(st, kLbPre | (unsigned long long)tot);
    } else {
        if (lane == 0) atomicExch(st + t, kLbAgg | (unsigned long long)tot);
        excl = lookback_prefix_warp(st, t);
        if (lane == 0) atomicExch(st + t, kLbPre | (unsigned long long)(excl + tot));
    }
    return excl;
}

// The rows of two indices i <= j (the last r in [0, rows) with e_off[r] <= i,
// and with e_off[r] <= j; e_off non-decreasing, e_off[0] <= i, j <
// e_off[rows]), by the 32 lanes of a warp together: each round probes 32
// points of both intervals at once and keeps the 1/33 between two of them, so
// a search over a million rows takes four rounds of parallel loads instead of
// twenty dependent ones.  A search that has finished keeps probing its own
// row, which leaves it where it is.
__device__ __forceinline__ void warp_rows_of(const int64_t* __restrict__ e_off, int64_t rows, int64_t i, int64_t j,
                                             int64_t* ri, int64_t* rj) {
    const int lane = threadIdx.x & 31;
    int64_t alo = 0, ahi = rows, blo = 0, bhi = rows;
    while (ahi - alo > 1 || bhi - blo > 1) {
        const int64_t pa = alo + ((ahi - alo) * (lane + 1)) / 33;
        const int64_t pb = blo + ((bhi - blo) * (lane + 1)) / 33;
        const int64_t va = e_off[pa], vb = e_off[pb];
        const int ca = __popc(__ballot_sync(0xffffffffu, va <= i));
        const int cb = __popc(__ballot_sync(0xffffffffu, vb <= j));
        const int64_t alo2 = __shfl_sync(0xffffffffu, pa, ca > 0 ? ca - 1 : 0);
        const int64_t ahi2 = __shfl_sync(0xffffffffu, pa, ca < 32 ? ca : 31);
        const int64_t blo2 = __shfl_sync(0xffffffffu, pb, cb > 0 ? cb - 1 : 0);
        const int64_t bhi2 = __shfl_sync(0xffffffffu, pb, cb < 32 ? cb : 31);
        if (ca > 0) alo = alo2;
        if (ca < 32) ahi = ahi2;
        if (cb > 0) blo = blo2;
        if (cb < 32) bhi = bhi2;
    }
    *ri = alo;
    *rj = blo;
}

template <class F>
int compact_alloc(const F& f, int64_t n, typename F::value_type** out, int64_t* kept_host, cudaStream_t s) {
    *out = nullptr;
    *kept_host = 0;
    if (n <= 0) return FAST_OK;
    int64_t nb = ceil_div(n, kComp2Tile);
    int64_t* offs = nullptr;
    int64_t* tot = nullptr;
    FAST_TRY(dalloc(&offs, nb + 1, s));
    tot = offs + nb;
    int rc = FAST_OK;
    k_compact_count<F><<<(unsigned)nb, kCompBlock, 0, s>>>(f, n, offs);
    note_launch();
    if (cudaGetLastError() != cudaSuccess) rc = set_error(FAST_ERR_CUDA, "compact count launch");
    if (rc == FAST_OK) rc = scan_exclusive<int64_t>(offs, offs, nb, tot, s);
    if (rc == FAST_OK) {
        cudaError_t e = cudaMemcpyAsync(kept_host, tot, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) rc = cuda_status(e, "compaction size readback", __FILE__, __LINE__);
    }
    if (rc == FAST_OK) rc = dalloc(out, (size_t)(*kept_host), s);
    if (rc == FAST_OK) {
        k_compact_write<F><<<(unsigned)nb, kCompBlock, 0, s>>>(f, n, offs, *out, (int64_t*)nullptr);
        note_launch();
        if (cudaGetLastError() != cudaSuccess) rc = set_error(FAST_ERR_CUDA, "compact write launch");
    }
    dfree(offs, s);
    if (rc != FAST_OK) dfree(*out, s);
    return rc;
}

// --------------------------------------------------------------- radix sort
//
// Stable LSD radix sort of uint64 keys, 8-bit digits, over the digit
// positions listed in `shifts`.  Three kernels per pass: per-tile digit
// histograms, a digit-major exclusive scan of them, and a stable scatter.

constexpr int kSortBlock = 256;
constexpr int kSortRounds = 8;
constexpr int kSortTile = kSortBlock * kSortRounds;

static __global__ void k_radix_hist(const uint64_t* __restrict__ keys, int64_t n, int shift, int64_t nblocks,
                             uint32_t* __restrict__ hist) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    int64_t base = (int64_t)blockIdx.x * kSortTile;
    uint64_t key[kSortRounds];            // all loads in flight at once
#pragma unroll
    for (int r = 0; r < kSortRounds; r++) {
        const int64_t i = base + (int64_t)r * kSortBlock + threadIdx.x;
        key[r] = i < n ? keys[i] : 0;
    }
#pragma unroll
    for (int r = 0; r < kSortRounds; r++)
        if (base + (int64_t)r * kSortBlock + threadIdx.x < n) atomicAdd(&h[(key[r] >> shift) & 255u], 1u);
    __syncthreads();
    hist[(int64_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// A warp ranks its own 256 keys, 32 at a time: the lanes with one digit are
// found by eight ballots, and its counts lie in its own row of shared memory,
// so no block barrier stands between two steps.  One scan over the warps and
// the digits gives every key its place in the tile; the tile is put in order
// in shared memory and leaves it digit by digit, so that neighbouring lanes
// write neighbouring keys.  Bound by the ranking's instructions (a pass over
// 32 M keys moves 512 MB).  With a block barrier per step and keys written
// from where they were read, such a pass took 245 us; the loader of a 16M-edge
// graph on the device 3.56 -> 2.94 ms (3.12 with 4096 keys a tile and three
// blocks per SM, 2.98 with 3072 and four).
static __global__ void __launch_bounds__(kSortBlock, 6) k_radix_scatter(const uint64_t* __restrict__ in,
                                uint64_t* __restrict__ out, int64_t n,
                                int shift, int64_t nblocks, const uint32_t* __restrict__ offs) {
    constexpr int NW = kSortBlock / 32;
    __shared__ uint64_t tile[kSortTile];
    __shared__ uint32_t wcnt[NW][256];    // each warp's counts, then the keys of the digit in the warps before it
    __shared__ uint32_t start[256];       // where each digit begins in the tile
    __shared__ uint32_t wsum[NW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t goff = offs[(int64_t)threadIdx.x * nblocks + blockIdx.x];   // global start of this tile's digit run
#pragma unroll
    for (int w = 0; w < NW; w++) wcnt[w][threadIdx.x] = 0;
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
    const int count = (int)(n - base < kSortTile ? n - base : kSortTile);
    const int first = warp * 32 * kSortRounds + lane;
    uint64_t key[kSortRounds];
#pragma unroll
    for (int r = 0; r < kSortRounds; r++) key[r] = first + 32 * r < count ? in[base + first + 32 * r] : 0;
    __syncthreads();
    uint32_t rank[kSortRounds];           // among the warp's keys of the digit
#pragma unroll
    for (int r = 0; r < kSortRounds; r++) {
        const bool valid = first + 32 * r < count;
        const uint32_t d = (uint32_t)(key[r] >> shift) & 255u;
        uint32_t peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
        for (int b = 0; b < 8; b++) {
            const uint32_t m = __ballot_sync(0xffffffffu, (d >> b) & 1u);
            peers &= (d >> b) & 1u ? m : ~m;
        }
        const uint32_t before = __popc(peers & lanemask_lt());
        uint32_t c = 0;
        if (valid) c = wcnt[warp][d];
        __syncwarp();
        if (valid && before == 0) wcnt[warp][d] = c + __popc(peers);
        __syncwarp();
        rank[r] = c + before;
    }
    __syncthreads();
    uint32_t total = 0;                   // of digit threadIdx.x
#pragma unroll
    for (int w = 0; w < NW; w++) {
        const uint32_t c = wcnt[w][threadIdx.x];
        wcnt[w][threadIdx.x] = total;
        total += c;
    }
    uint32_t incl = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    uint32_t s0 = incl - total;
#pragma unroll
    for (int w = 0; w < NW; w++) s0 += w < warp ? wsum[w] : 0u;
    start[threadIdx.x] = s0;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortRounds; r++)
        if (first + 32 * r < count) {
            const uint32_t d = (uint32_t)(key[r] >> shift) & 255u;
            tile[start[d] + wcnt[warp][d] + rank[r]] = key[r];
        }
    __syncthreads();
    wcnt[0][threadIdx.x] = goff - s0;     // what to add to a place in the tile
    __syncthreads();
    for (int i = threadIdx.x; i < count; i += kSortBlock) {
        const uint64_t k = tile[i];
        out[wcnt[0][(k >> shift) & 255u] + (uint32_t)i] = k;
    }
}

// Sorts keys[0..n) in place (tmp: caller scratch of n keys, or null to
// allocate).  n must be below 2^32.
inline int radix_sort_u64(uint64_t* keys, int64_t n, const int* shifts, int npass, cudaStream_t s) {
    if (n <= 1 || npass == 0) return FAST_OK;
    if (n >= (int64_t)0xFFFFFFFFll) return set_error(FAST_ERR_INVALID, "radix sort: too many keys (%lld)", (long long)n);
    int64_t nb = ceil_div(n, kSortTile);
    uint64_t* tmp = nullptr;
    uint32_t* hist = nullptr;
    FAST_TRY(dalloc(&tmp, n, s));
    int rc = dalloc(&hist, 256 * nb, s);
    uint64_t* a = keys;
    uint64_t* b = tmp;
    for (int p = 0; p < npass && rc == FAST_OK; p++) {
        k_radix_hist<<<(unsigned)nb, kSortBlock, 0, s>>>(a, n, shifts[p], nb, hist);
        note_launch();
        if (cudaGetLastError() != cudaSuccess) { rc = set_error(FAST_ERR_CUDA, "radix hist launch"); break; }
        rc = scan_exclusive<uint32_t>(hist, hist, 256 * nb, (uint32_t*)nullptr, s);
        if (rc != FAST_OK) break;
        k_radix_scatter<<<(unsigned)nb, kSortBlock, 0, s>>>(a, b, n, shifts[p], nb, hist);
        note_launch();
        if (cudaGetLastError() != cudaSuccess) { rc = set_error(FAST_ERR_CUDA, "radix scatter launch"); break; }
        uint64_t* t = a; a = b; b = t;
    }
    if (rc == FAST_OK && a != keys) {
        cudaError_t e = cudaMemcpyAsync(keys, a, (size_t)n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess) rc = cuda_status(e, "radix copy back", __FILE__, __LINE__);
    }
    dfree(tmp, s);
    dfree(hist, s);
    return rc;
}

// Digit shifts covering bits [lo, hi) in 8-bit steps.
inline int digit_shifts(int lo, int hi, int* out, int max_out) {
    int n = 0;
    for (int sft = lo; sft < hi && n < max_out; sft += 8) out[n++] = sft;
    return n;
}

inline int bits_for(int64_t maxval) {
    int b = 0;
    while (b < 63 && (maxval >> b) > 0) b++;
    return b;
}

}  // namespace fast
