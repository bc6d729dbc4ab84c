// The per-query entry points of the candidate search tree (Sec. IV-A): its
// build, which is the batched build (cst_batch.cu) of one query, and the
// accessors.
#include <cstring>

#include "internal.cuh"

using namespace fast;

namespace {

void cst_release(fast_cst* c) {
    if (!c) return;
    c->arena.release(c->stream);
    delete c;
}

}  // namespace

// --------------------------------------------------------------- C ABI

extern "C" int fast_build_cst(const fast_graph* g, const fast_query_desc* q, const fast_config* cfg, void* stream,
                              fast_cst** out) {
    if (!out) return set_error(FAST_ERR_INVALID, "fast_build_cst: out is NULL");
    *out = nullptr;
    if (!g) return set_error(FAST_ERR_INVALID, "fast_build_cst: graph is NULL");
    if (!q) return set_error(FAST_ERR_INVALID, "query is NULL");
    if (cfg && cfg->refine_rule != 0)
        return set_error(FAST_ERR_INVALID, "fast_build_cst: refine_rule %d (only fast_build_cst_batch refines further)",
                         cfg->refine_rule);
    PoolScope scratch((cudaStream_t)stream);
    int32_t status = FAST_OK;
    const uint64_t trips = build_round_trips();               // those of the last batched build stay
    int rc = build_cst_batch(g, 1, q, &cfg, (cudaStream_t)stream, out, &status);
    set_build_round_trips(trips);
    return rc != FAST_OK ? rc : status;
}

extern "C" int fast_cst_info(const fast_cst* c, int32_t* k, int32_t* root, int32_t* order, int32_t* parent,
                             int64_t* cand, uint64_t* w_u64, double* w_f64) {
    if (!c) return set_error(FAST_ERR_INVALID, "fast_cst_info: NULL cst");
    if (k) *k = c->k;
    if (root) *root = c->root;
    for (int i = 0; i < c->k; i++) {
        if (order) order[i] = c->order[i];
        if (parent) parent[i] = c->parent[i];
        if (cand) cand[i] = c->ncand[i];
    }
    if (w_u64) *w_u64 = c->W;
    if (w_f64) *w_f64 = c->Wf;
    return FAST_OK;
}

extern "C" int fast_cst_candidates(const fast_cst* c, int32_t u, int32_t* out, void* stream) {
    if (!c || u < 0 || u >= c->k || (!out && c->ncand[u])) return set_error(FAST_ERR_INVALID, "fast_cst_candidates: bad argument");
    cudaStream_t s = (cudaStream_t)stream;
    if (c->ncand[u]) FAST_CUDA(cudaMemcpyAsync(out, c->cand[u], c->ncand[u] * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    FAST_CUDA(cudaStreamSynchronize(s));
    return FAST_OK;
}

extern "C" int fast_cst_tree_size(const fast_cst* c, int32_t u, int64_t* entries) {
    if (!c || u < 0 || u >= c->k || !entries) return set_error(FAST_ERR_INVALID, "fast_cst_tree_size: bad argument");
    *entries = c->parent[u] < 0 ? 0 : c->t_entries[u];
    return FAST_OK;
}

extern "C" int fast_cst_tree_lists(const fast_cst* c, int32_t u, int64_t* off, uint32_t* idx, void* stream) {
    if (!c || u < 0 || u >= c->k || c->parent[u] < 0 || !off || (!idx && c->t_entries[u]))
        return set_error(FAST_ERR_INVALID, "fast_cst_tree_lists: bad argument");
    cudaStream_t s = (cudaStream_t)stream;
    int64_t rows = c->ncand[c->parent[u]];
    FAST_CUDA(cudaMemcpyAsync(off, c->t_off[u], (rows + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    if (c->t_entries[u]) FAST_CUDA(cudaMemcpyAsync(idx, c->t_idx[u], c->t_entries[u] * sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    FAST_CUDA(cudaStreamSynchronize(s));
    return FAST_OK;
}

extern "C" int fast_cst_nontree_count(const fast_cst* c, int32_t* count) {
    if (!c || !count) return set_error(FAST_ERR_INVALID, "fast_cst_nontree_count: bad argument");
    *count = c->nnt;
    return FAST_OK;
}

extern "C" int fast_cst_nontree_edge(const fast_cst* c, int32_t e, int32_t* from_u, int32_t* to_u, int64_t* entries) {
    if (!c || e < 0 || e >= c->nnt) return set_error(FAST_ERR_INVALID, "fast_cst_nontree_edge: bad argument");
    if (from_u) *from_u = c->nt_from[e];
    if (to_u) *to_u = c->nt_to[e];
    if (entries) *entries = c->n_entries[e];
    return FAST_OK;
}

extern "C" int fast_cst_nontree_lists(const fast_cst* c, int32_t e, int64_t* off, uint32_t* idx, void* stream) {
    if (!c || e < 0 || e >= c->nnt || !off || (!idx && c->n_entries[e]))
        return set_error(FAST_ERR_INVALID, "fast_cst_nontree_lists: bad argument");
    cudaStream_t s = (cudaStream_t)stream;
    int64_t rows = c->ncand[c->nt_from[e]];
    FAST_CUDA(cudaMemcpyAsync(off, c->n_off[e], (rows + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    if (c->n_entries[e]) FAST_CUDA(cudaMemcpyAsync(idx, c->n_idx[e], c->n_entries[e] * sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    FAST_CUDA(cudaStreamSynchronize(s));
    return FAST_OK;
}

extern "C" int fast_cst_workload(const fast_cst* c, int32_t u, uint64_t* out, void* stream) {
    if (!c || u < 0 || u >= c->k || (!out && c->ncand[u])) return set_error(FAST_ERR_INVALID, "fast_cst_workload: bad argument");
    cudaStream_t s = (cudaStream_t)stream;
    if (c->ncand[u]) FAST_CUDA(cudaMemcpyAsync(out, c->cval[u], c->ncand[u] * sizeof(uint64_t), cudaMemcpyDeviceToHost, s));
    FAST_CUDA(cudaStreamSynchronize(s));
    return FAST_OK;
}

namespace fast {
void cst_release_nosync(fast_cst* c) { cst_release(c); }
}  // namespace fast

extern "C" void fast_free_cst(fast_cst* c) {
    if (!c) return;
    cudaStream_t s = c->stream;
    cst_release(c);
    cudaStreamSynchronize(s);
}
