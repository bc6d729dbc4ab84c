// Data-graph loader (Sec. II-A data model) and the library's error plumbing.
//
// fast_load_graph turns an edge list into a device CSR of the simple
// undirected graph over positions: vertices ordered by (label, id), so that a
// label's vertices are one range, a row's neighbours with one label are one
// segment, and a set of vertices of one label is a bitmap over that range.  A
// radix sort on (label, id) gives the order; both directions of every edge
// become keys (position of src, position of dst), which a stable LSD radix
// sort orders; an ordered compaction drops self loops and repeats; a boundary
// pass writes the row offsets, and another the label segments.
//
// Sorting positions takes the place of sorting (src, dst) first and (src,
// label, dst) again after the repeats are gone: 5 instead of 10 digit passes
// over the 32 M entries of a 1M/16M graph.  The label segments are filled in
// parallel over the entries; a warp per row, as it was, walked the largest
// row (377,836 entries) alone, twice 7.6 ms.
#include <stdarg.h>

#include <atomic>
#include <cstring>

#include "internal.cuh"
#include "prims.cuh"

namespace fast {

static thread_local char g_err[512] = "";
static std::atomic<uint64_t> g_launches{0};

void note_launch(int n) { g_launches.fetch_add((uint64_t)n, std::memory_order_relaxed); }

int set_error(int code, const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return code;
}

int cuda_status(cudaError_t e, const char* what, const char* file, int line) {
    cudaGetLastError();
    int code = (e == cudaErrorMemoryAllocation) ? FAST_ERR_OOM : FAST_ERR_CUDA;
    const char* base = strrchr(file, '/');
    return set_error(code, "%s failed: %s (%s:%d)", what, cudaGetErrorString(e), base ? base + 1 : file, line);
}

}  // namespace fast

using namespace fast;

extern "C" const char* fast_last_error(void) { return g_err; }

extern "C" uint64_t fast_kernel_launches(void) { return g_launches.load(std::memory_order_relaxed); }

extern "C" void fast_config_default(fast_config* cfg) {
    if (!cfg) return;
    memset(cfg, 0, sizeof(*cfg));
    cfg->delta_w = 1ull << 20;
    cfg->sample_root = 0.0;
    cfg->sample_deep = 0.0;
    cfg->sample_seed = 0;
    cfg->max_chunks = 1ll << 16;
    cfg->warps_per_block = 8;
    cfg->blocks_per_sm = 4;
    cfg->time_budget_s = 0.0;
    cfg->limit = 0;
    cfg->queue_cells = 0;
    cfg->order_rule = 0;
    cfg->filter_rule = 0;
    cfg->build_rule = 0;
    cfg->refine_rule = 0;
    cfg->matcher_rule = 0;
    cfg->validators = 0;
}

namespace {


__global__ void k_check_edges(const int32_t* __restrict__ edges, int64_t m, int64_t n, int* __restrict__ bad) {
    const int2* e = (const int2*)edges;
    bool b = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int2 x = e[i];
        b |= x.x < 0 || x.y < 0 || x.x >= n || x.y >= n;
    }
    if (b) atomicOr(bad, 1);
}

__global__ void k_edge_keys(const int32_t* __restrict__ edges, int64_t m, const int32_t* __restrict__ pos, int nb,
                            uint64_t sent, uint64_t* __restrict__ keys) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= m) return;
    const int2 ab = ((const int2*)edges)[e];
    uint64_t x = sent, y = sent;                              // a loop: no entry
    if (ab.x != ab.y) {
        const uint64_t a = (uint32_t)pos[ab.x], b = (uint32_t)pos[ab.y];
        x = a << nb | b;
        y = b << nb | a;
    }
    keys[2 * e] = x;
    keys[2 * e + 1] = y;
}

__global__ void k_check_labels(const int32_t* __restrict__ lab, int64_t n, int* __restrict__ bad,
                               int* __restrict__ maxlab) {
    int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int32_t l = v < n ? lab[v] : 0;
    if (l < 0 || l >= (1 << 23)) { atomicOr(bad, 2); l = 0; }
    l = __reduce_max_sync(0xffffffffu, l);
    if ((threadIdx.x & 31) == 0 && l > *(volatile int*)maxlab) atomicMax(maxlab, l);
}

// keep key i iff it is a real edge and differs from its predecessor
struct DedupF {
    using value_type = uint64_t;
    const uint64_t* keys;
    uint64_t sent;
    __device__ void begin(int64_t) {}
    __device__ bool eval(int64_t i, uint64_t& v) const {
        uint64_t k = keys[i];
        v = k;
        return k != sent && (i == 0 || keys[i - 1] != k);
    }
};

// row_ptr[v] = first entry whose source is >= v, from sorted keys
__global__ void k_row_bounds(const uint64_t* __restrict__ kept, int64_t nadj, int64_t n, int nb, uint64_t dst_mask,
                             int64_t* __restrict__ row_ptr, int32_t* __restrict__ col) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p > nadj) return;
    int64_t hi = (p < nadj) ? (int64_t)(kept[p] >> nb) : n;      // rows (prev, hi] start at p
    int64_t lo = (p == 0) ? -1 : (int64_t)(kept[p - 1] >> nb);
    for (int64_t v = lo + 1; v <= hi; v++) row_ptr[v] = p;
    if (p < nadj) col[p] = (int32_t)(kept[p] & dst_mask);
}

__global__ void k_vertex_keys(const int32_t* __restrict__ lab, int64_t n, uint64_t* __restrict__ lkeys) {
    int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v < n) lkeys[v] = ((uint64_t)(uint32_t)lab[v] << 32) | (uint64_t)v;
}

// positions from the sorted (label, id) keys: label ranges, vertex and label
// of each position, position of each vertex
__global__ void k_label_bounds(const uint64_t* __restrict__ lkeys, int64_t n, int64_t L,
                               int64_t* __restrict__ lab_ptr, int32_t* __restrict__ lab_vtx,
                               int32_t* __restrict__ plab, int32_t* __restrict__ pos) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p > n) return;
    int64_t hi = (p < n) ? (int64_t)(lkeys[p] >> 32) : L;
    int64_t lo = (p == 0) ? -1 : (int64_t)(lkeys[p - 1] >> 32);
    for (int64_t l = lo + 1; l <= hi; l++) lab_ptr[l] = p;
    if (p < n) {
        const int32_t v = (int32_t)(lkeys[p] & 0xFFFFFFFFu);
        lab_vtx[p] = v;
        plab[p] = (int32_t)hi;
        pos[v] = (int32_t)p;
    }
}

// degree sums: out[l] = first entry of label l's rows; and the largest degree
__global__ void k_label_rows(const int64_t* __restrict__ row_ptr, const int64_t* __restrict__ lab_ptr, int64_t L,
                             int64_t* __restrict__ out) {
    int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (l <= L) out[l] = row_ptr[lab_ptr[l]];
}

__global__ void k_max_degree(const int64_t* __restrict__ row_ptr, int64_t n, unsigned long long* __restrict__ maxdeg) {
    uint32_t d = 0;                                           // a row has fewer than n < 2^31 entries
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        d = max(d, (uint32_t)(row_ptr[v + 1] - row_ptr[v]));
    d = __reduce_max_sync(0xffffffffu, d);
    if ((threadIdx.x & 31) == 0) atomicMax(maxdeg, (unsigned long long)d);
}

// ------------------------------------------------------------ label runs

// Where each row's neighbours with each label start, relative to the row:
// lrel[l * n + p] for row p and label l (plane L: the row's length), one
// plane per label so that a warp's 32 neighbouring rows read one line.  An
// entry that opens its label's segment writes it, and the empty segments of
// the labels before it; the row's last entry writes those after it.  Zeros
// (rows with no entries, first segments) come from the memset before.
__global__ void k_label_table(const int64_t* __restrict__ row_ptr, const uint64_t* __restrict__ kept, int64_t nadj,
                              int nb, uint64_t dst_mask, const int32_t* __restrict__ plab, int64_t n, int L,
                              uint32_t* __restrict__ lrel) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nadj) return;
    const uint64_t k = kept[i];
    const int64_t r = (int64_t)(k >> nb);
    const int32_t l = plab[k & dst_mask];
    const int64_t a = row_ptr[r], b = row_ptr[r + 1];
    const int32_t lp = i == a ? -1 : plab[kept[i - 1] & dst_mask];
    const uint32_t rel = (uint32_t)(i - a);
    if (rel)
        for (int32_t x = lp + 1; x <= l; x++) lrel[(int64_t)x * n + r] = rel;
    if (i == b - 1)
        for (int32_t x = l + 1; x <= L; x++) lrel[(int64_t)x * n + r] = (uint32_t)(b - a);
}

// warp per row: number of label runs (write = 0), or the runs themselves
template <bool WRITE>
__global__ void k_row_runs(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                           const int32_t* __restrict__ plab, int64_t n, int64_t* __restrict__ cnt,
                           const int64_t* __restrict__ run_ptr, int32_t* __restrict__ run_lab,
                           int64_t* __restrict__ run_beg) {
    const int lane = threadIdx.x & 31;
    int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = w; v < n; v += nw) {
        const int64_t a = row_ptr[v], b = row_ptr[v + 1];
        int64_t r = WRITE ? run_ptr[v] : 0;
        int64_t c = 0;
        for (int64_t base = a; base < b; base += 32) {
            int64_t i = base + lane;
            bool head = false;
            int32_t l = 0;
            if (i < b) {
                l = plab[col[i]];
                head = (i == a) || plab[col[i - 1]] != l;
            }
            uint32_t m = __ballot_sync(0xffffffffu, head);
            if (WRITE && head) {
                int64_t at = r + __popc(m & lanemask_lt());
                run_lab[at] = l;
                run_beg[at] = i;
            }
            r += __popc(m);
            c += __popc(m);
        }
        if (!WRITE && lane == 0) cnt[v] = c;
    }
}

// Adjacency entries per (label a of the row's vertex, label b of the
// neighbour), M[a * L + b]: blockIdx.y = b, a block sums the segments of
// kPairRows rows, label by label.
constexpr int kPairRows = 4096;

__global__ void __launch_bounds__(256) k_label_pairs(GraphSegs G, const int64_t* __restrict__ lab_ptr, int64_t n, int L,
                                                     unsigned long long* __restrict__ M) {
    const int b = blockIdx.y;
    const int64_t r0 = (int64_t)blockIdx.x * kPairRows, r1 = r0 + kPairRows < n ? r0 + kPairRows : n;
    int a = 0;
    {
        int hi = L;
        while (hi - a > 1) {                                  // last label with lab_ptr <= r0
            const int mid = (a + hi) >> 1;
            if (lab_ptr[mid] <= r0) a = mid; else hi = mid;
        }
    }
    for (; a < L && lab_ptr[a] < r1; a++) {
        const int64_t x0 = lab_ptr[a] > r0 ? lab_ptr[a] : r0, x1 = lab_ptr[a + 1] < r1 ? lab_ptr[a + 1] : r1;
        unsigned long long sum = 0;
        for (int64_t p = x0 + threadIdx.x; p < x1; p += blockDim.x) {
            uint32_t beg, len;
            label_segment(G, (int32_t)p, b, &beg, &len);
            sum += len;
        }
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if ((threadIdx.x & 31) == 0 && sum) atomicAdd(M + (int64_t)a * L + b, sum);
    }
}

int label_pair_counts(fast_graph* g, cudaStream_t s) {
    const int L = g->num_labels;
    if (L <= 0 || L > kLabelPairMax) return FAST_OK;
    unsigned long long* M = nullptr;
    FAST_TRY(dalloc(&M, (int64_t)L * L, s));
    cudaMemsetAsync(M, 0, (size_t)L * L * sizeof(unsigned long long), s);
    k_label_pairs<<<dim3((unsigned)ceil_div(g->n, kPairRows), (unsigned)L), 256, 0, s>>>(graph_segs(g), g->lab_ptr, g->n, L, M);
    note_launch();
    std::vector<int64_t> h((size_t)L * L);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(h.data(), M, h.size() * sizeof(int64_t), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    dfree(M, s);
    if (e != cudaSuccess) return cuda_status(e, "label pair counts", __FILE__, __LINE__);
    g->lab_pair_host.swap(h);
    return FAST_OK;
}

// The label segments of every row: the table when it takes at most 12 bytes
// per adjacency entry (every configuration of few labels: one line of loads
// per 32 rows), else a directory of the labels that a row has (one binary
// search per row; its size follows the entries, whatever the label count).
int build_label_segments(fast_graph* g, const uint64_t* kept, int nb, uint64_t dst_mask, const int32_t* plab,
                         cudaStream_t s) {
    const int64_t n = g->n, L = g->num_labels;
    const double table = 4.0 * (double)n * (double)(L + 1);
    if (table <= 12.0 * (double)g->nadj + (64 << 20)) {
        FAST_TRY(dalloc(&g->lrel, (size_t)n * (L + 1), s));
        FAST_CUDA(cudaMemsetAsync(g->lrel, 0, (size_t)n * (L + 1) * sizeof(uint32_t), s));
        if (g->nadj > 0) {
            k_label_table<<<(unsigned)ceil_div(g->nadj, 256), 256, 0, s>>>(g->row_ptr, kept, g->nadj, nb, dst_mask, plab, n,
                                                                         (int)L, g->lrel);
            note_launch();
            FAST_CUDA(cudaGetLastError());
        }
        return FAST_OK;
    }
    int64_t* cnt = nullptr;
    FAST_TRY(dalloc(&g->run_ptr, n + 1, s));
    FAST_TRY(dalloc(&cnt, n, s));
    unsigned blocks = (unsigned)std::min<int64_t>(ceil_div(n, 8), (int64_t)num_sms() * 32);
    k_row_runs<false><<<blocks, 256, 0, s>>>(g->row_ptr, g->col, plab, n, cnt, nullptr, nullptr, nullptr);
    note_launch();
    int rc = scan_exclusive<int64_t>(cnt, g->run_ptr, n, g->run_ptr + n, s);
    int64_t R = 0;
    if (rc == FAST_OK) {
        cudaError_t e = cudaMemcpyAsync(&R, g->run_ptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) rc = cuda_status(e, "label runs", __FILE__, __LINE__);
    }
    dfree(cnt, s);
    if (rc == FAST_OK) rc = dalloc(&g->run_lab, R, s);
    if (rc == FAST_OK) rc = dalloc(&g->run_beg, R, s);
    if (rc == FAST_OK) {
        k_row_runs<true><<<blocks, 256, 0, s>>>(g->row_ptr, g->col, plab, n, nullptr, g->run_ptr, g->run_lab, g->run_beg);
        note_launch();
        if (cudaGetLastError() != cudaSuccess) rc = set_error(FAST_ERR_CUDA, "label runs launch");
    }
    return rc;
}

void graph_release(fast_graph* g, cudaStream_t s) {
    if (!g) return;
    dfree(g->row_ptr, s); dfree(g->col, s);
    dfree(g->lab_ptr, s); dfree(g->lab_vtx, s);
    dfree(g->lrel, s); dfree(g->run_ptr, s); dfree(g->run_lab, s); dfree(g->run_beg, s);
    delete g;
}

int load_graph(int64_t n, int64_t m, const int32_t* edges, const int32_t* labels, int flags,
               cudaStream_t s, fast_graph** out) {
    if (!out) return set_error(FAST_ERR_INVALID, "fast_load_graph: out is NULL");
    *out = nullptr;
    if (n < 1 || n > 0x7FFFFFFFll) return set_error(FAST_ERR_INVALID, "fast_load_graph: n=%lld out of range", (long long)n);
    if (m < 0 || 2 * m >= 0xFFFFFFFFll) return set_error(FAST_ERR_INVALID, "fast_load_graph: m=%lld out of range", (long long)m);
    if ((m > 0 && !edges) || !labels) return set_error(FAST_ERR_INVALID, "fast_load_graph: NULL input");
    fast_graph* g = new fast_graph();
    g->n = n;
    int32_t* d_edges = nullptr;
    int32_t* d_lab = nullptr;
    uint64_t* keys = nullptr;
    uint64_t* kept = nullptr;
    int* flags_d = nullptr;
    uint64_t* lkeys = nullptr;
    int32_t* plab = nullptr;                                  // label of each position
    int32_t* pos = nullptr;                                   // position of each vertex
    int64_t* sums = nullptr;
    unsigned long long* maxdeg_d = nullptr;
    int rc = FAST_OK;
    const bool dev = (flags & FAST_PTR_DEVICE) != 0;
    do {
        const int32_t* l_dev = labels;
        const int32_t* e_dev = edges;
        if (!dev) {
            rc = dalloc(&d_lab, n, s); if (rc) break;
            if (cudaMemcpyAsync(d_lab, labels, n * sizeof(int32_t), cudaMemcpyHostToDevice, s) != cudaSuccess) { rc = set_error(FAST_ERR_CUDA, "label upload"); break; }
            l_dev = d_lab;
        }
        // the pairs are read 8 bytes at a time: a device array that does not
        // start on such a boundary is copied like a host one
        if (m > 0 && (!dev || ((uintptr_t)edges & 7))) {
            rc = dalloc(&d_edges, 2 * m, s); if (rc) break;
            if (cudaMemcpyAsync(d_edges, edges, 2 * m * sizeof(int32_t), cudaMemcpyDefault, s) != cudaSuccess) { rc = set_error(FAST_ERR_CUDA, "edge upload"); break; }
            e_dev = d_edges;
        }
        rc = dalloc(&flags_d, 2, s); if (rc) break;
        cudaMemsetAsync(flags_d, 0, 2 * sizeof(int), s);
        if (m > 0) {
            k_check_edges<<<(unsigned)std::min<int64_t>(ceil_div(m, 256), (int64_t)num_sms() * 8), 256, 0, s>>>(e_dev, m, n, flags_d);
            note_launch();
        }
        k_check_labels<<<(unsigned)ceil_div(n, 256), 256, 0, s>>>(l_dev, n, flags_d, flags_d + 1);
        note_launch();
        int hflags[2] = {0, 0};
        if (cudaMemcpyAsync(hflags, flags_d, sizeof(hflags), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess) { rc = set_error(FAST_ERR_CUDA, "loader validation"); break; }
        if (hflags[0] & 1) { rc = set_error(FAST_ERR_INVALID, "fast_load_graph: edge endpoint outside 0..n-1"); break; }
        if (hflags[0] & 2) { rc = set_error(FAST_ERR_INVALID, "fast_load_graph: label outside 0..2^23-1"); break; }
        g->num_labels = hflags[1] + 1;
        const int64_t L = g->num_labels;
        const int nb = bits_for(n - 1 > 0 ? n - 1 : 1);
        const int lbits = bits_for(L - 1 > 0 ? L - 1 : 1);
        g->csr_by_id = 2 * nb + lbits > 64;
        const uint64_t dst_mask = (1ull << nb) - 1;           // n < 2^31: nb <= 31
        const uint64_t sent = (1ull << (2 * nb)) - 1;         // a loop's key: no real entry has it
        int shifts[16];
        // ---- positions
        rc = dalloc(&lkeys, n, s); if (rc) break;
        k_vertex_keys<<<(unsigned)ceil_div(n, 256), 256, 0, s>>>(l_dev, n, lkeys);
        note_launch();
        int np = digit_shifts(32, 32 + lbits, shifts, 8);
        rc = radix_sort_u64(lkeys, n, shifts, np, s); if (rc) break;
        rc = dalloc(&g->lab_ptr, L + 1, s); if (rc) break;
        rc = dalloc(&g->lab_vtx, n, s); if (rc) break;
        rc = dalloc(&plab, n, s); if (rc) break;
        rc = dalloc(&pos, n, s); if (rc) break;
        k_label_bounds<<<(unsigned)ceil_div(n + 1, 256), 256, 0, s>>>(lkeys, n, L, g->lab_ptr, g->lab_vtx, plab, pos);
        note_launch();
        // ---- adjacency
        rc = dalloc(&keys, 2 * m, s); if (rc) break;
        if (m > 0) { k_edge_keys<<<(unsigned)ceil_div(m, 256), 256, 0, s>>>(e_dev, m, pos, nb, sent, keys); note_launch(); }
        np = digit_shifts(0, 2 * nb, shifts, 8);
        rc = radix_sort_u64(keys, 2 * m, shifts, np, s); if (rc) break;
        DedupF f{keys, sent};
        int64_t nadj = 0;
        rc = compact_alloc(f, 2 * m, &kept, &nadj, s); if (rc) break;
        g->nadj = nadj;
        dfree(keys, s);
        dfree(d_edges, s);
        rc = dalloc(&g->row_ptr, n + 1, s); if (rc) break;
        rc = dalloc(&g->col, nadj, s); if (rc) break;
        k_row_bounds<<<(unsigned)ceil_div(nadj + 1, 256), 256, 0, s>>>(kept, nadj, n, nb, dst_mask, g->row_ptr, g->col);
        note_launch();
        rc = build_label_segments(g, kept, nb, dst_mask, plab, s); if (rc) break;
        rc = dalloc(&maxdeg_d, 1, s); if (rc) break;
        cudaMemsetAsync(maxdeg_d, 0, sizeof(unsigned long long), s);
        k_max_degree<<<(unsigned)std::min<int64_t>(ceil_div(n, 256), (int64_t)num_sms() * 8), 256, 0, s>>>(g->row_ptr, n, maxdeg_d);
        note_launch();
        rc = dalloc(&sums, L + 1, s); if (rc) break;
        k_label_rows<<<(unsigned)ceil_div(L + 1, 256), 256, 0, s>>>(g->row_ptr, g->lab_ptr, L, sums);
        note_launch();
        std::vector<int64_t> hs(L + 1);
        g->lab_ptr_host.resize(L + 1);
        unsigned long long md = 0;
        if (cudaMemcpyAsync(hs.data(), sums, (L + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaMemcpyAsync(g->lab_ptr_host.data(), g->lab_ptr, (L + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaMemcpyAsync(&md, maxdeg_d, sizeof(md), cudaMemcpyDeviceToHost, s) != cudaSuccess) { rc = set_error(FAST_ERR_CUDA, "label index readback"); break; }
        cudaError_t e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) { rc = cuda_status(e, "fast_load_graph", __FILE__, __LINE__); break; }
        g->max_degree = (int64_t)md;
        g->lab_degsum_host.resize(L);
        for (int64_t l = 0; l < L; l++) g->lab_degsum_host[l] = hs[l + 1] - hs[l];
        rc = label_pair_counts(g, s); if (rc) break;
    } while (0);
    dfree(d_edges, s); dfree(d_lab, s); dfree(keys, s); dfree(kept, s); dfree(flags_d, s); dfree(lkeys, s);
    dfree(plab, s); dfree(pos, s); dfree(sums, s); dfree(maxdeg_d, s);
    if (rc != FAST_OK) {
        graph_release(g, s);
        return rc;
    }
    *out = g;
    return FAST_OK;
}

// ------------------------------------------------------------- CSR read-back

// degree of each vertex
__global__ void k_export_degree(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ lab_vtx, int64_t n,
                                int64_t* __restrict__ deg) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n) deg[lab_vtx[p]] = row_ptr[p + 1] - row_ptr[p];
}

// The entries in vertex order: col_out[] as ids, or keys[] as (row, id) pairs
// still to be sorted.  Warp tiles of 512 entries.
__global__ void __launch_bounds__(256) k_export_cols(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                                                     const int32_t* __restrict__ lab_vtx, int64_t n, int64_t nadj,
                                                     const int64_t* __restrict__ out_ptr, int32_t* __restrict__ col_out,
                                                     uint64_t* __restrict__ keys) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t * 512 < nadj; t += nw) {
        const int64_t tb = t * 512, te = tb + 512 < nadj ? tb + 512 : nadj;
        int64_t r0, r1;
        warp_rows_of(row_ptr, n, tb, te - 1, &r0, &r1);
        for (int64_t e = tb + lane; e < te; e += 32) {
            int64_t lo = r0, hi = r1 + 1;                     // last row in [r0, r1] that starts at or before e
            while (hi - lo > 1) {
                const int64_t mid = (lo + hi) >> 1;
                if (row_ptr[mid] <= e) lo = mid; else hi = mid;
            }
            const int32_t v = lab_vtx[lo], x = lab_vtx[col[e]];
            const int64_t at = out_ptr[v] + (e - row_ptr[lo]);
            if (keys) keys[at] = ((uint64_t)(uint32_t)v << 32) | (uint32_t)x;
            else col_out[at] = x;
        }
    }
}

__global__ void k_key_cols(const uint64_t* __restrict__ keys, int64_t n, int32_t* __restrict__ col) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) col[i] = (int32_t)(keys[i] & 0xFFFFFFFFu);
}

int copy_csr(const fast_graph* g, int64_t* row_ptr, int32_t* col, cudaStream_t s) {
    const int64_t n = g->n, nadj = g->nadj;
    int64_t* out_ptr = nullptr;
    int32_t* out_col = nullptr;
    uint64_t* keys = nullptr;
    int rc = FAST_OK;
    do {
        rc = dalloc(&out_ptr, n + 1, s); if (rc) break;
        rc = dalloc(&out_col, nadj, s); if (rc) break;
        k_export_degree<<<(unsigned)ceil_div(n, 256), 256, 0, s>>>(g->row_ptr, g->lab_vtx, n, out_ptr);
        note_launch();
        rc = scan_exclusive<int64_t>(out_ptr, out_ptr, n, out_ptr + n, s); if (rc) break;
        if (nadj > 0) {
            if (g->csr_by_id) { rc = dalloc(&keys, nadj, s); if (rc) break; }
            const unsigned blocks = (unsigned)std::min<int64_t>(ceil_div(nadj, 4096), (int64_t)num_sms() * 8);
            k_export_cols<<<blocks, 256, 0, s>>>(g->row_ptr, g->col, g->lab_vtx, n, nadj, out_ptr, out_col, keys);
            note_launch();
            if (keys) {
                const int nb = bits_for(n - 1 > 0 ? n - 1 : 1);
                int shifts[16];
                int np = digit_shifts(0, nb, shifts, 8);
                np += digit_shifts(32, 32 + nb, shifts + np, 8);
                rc = radix_sort_u64(keys, nadj, shifts, np, s); if (rc) break;
                k_key_cols<<<(unsigned)ceil_div(nadj, 256), 256, 0, s>>>(keys, nadj, out_col);
                note_launch();
            }
        }
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(row_ptr, out_ptr, (n + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess && nadj) e = cudaMemcpyAsync(col, out_col, nadj * sizeof(int32_t), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) rc = cuda_status(e, "fast_graph_copy_csr", __FILE__, __LINE__);
    } while (0);
    dfree(out_ptr, s); dfree(out_col, s); dfree(keys, s);
    return rc;
}

}  // namespace

extern "C" int fast_load_graph(int64_t n, int64_t m, const int32_t* edges, const int32_t* labels, int flags,
                               void* stream, fast_graph** out) {
    return load_graph(n, m, edges, labels, flags, (cudaStream_t)stream, out);
}

extern "C" int fast_graph_info(const fast_graph* g, int64_t* n, int64_t* nadj, int32_t* num_labels,
                               int64_t* max_degree) {
    if (!g) return set_error(FAST_ERR_INVALID, "fast_graph_info: NULL graph");
    if (n) *n = g->n;
    if (nadj) *nadj = g->nadj;
    if (num_labels) *num_labels = g->num_labels;
    if (max_degree) *max_degree = g->max_degree;
    return FAST_OK;
}

extern "C" int fast_graph_copy_csr(const fast_graph* g, int64_t* row_ptr, int32_t* col, void* stream) {
    if (!g || !row_ptr || (!col && g->nadj)) return set_error(FAST_ERR_INVALID, "fast_graph_copy_csr: NULL argument");
    cudaStream_t s = (cudaStream_t)stream;
    return copy_csr(g, row_ptr, col, s);
}

extern "C" void fast_free_graph(fast_graph* g) {
    if (!g) return;
    graph_release(g, nullptr);
    cudaStreamSynchronize(nullptr);
    trim_freed_memory();                 // a workload ended: hand its pooled memory back
}
