"""Sizes at which the loader, the list passes, the matcher's list checks and
its flat search change paths, each against the oracle.  Integer results:
equality.  (The float64 workload estimate: compare_cst's bound.)

The file runs after the other GPU tests (its name sorts last).
"""
import numpy as np
import pytest

import oracle
import paper_2102_10768_gb300 as F
from helpers import compare_cst, csr_by_label, sorted_rows

pytestmark = pytest.mark.gpu

PATH3 = np.array([[0, 1], [1, 2]], np.int32)
TRIANGLE = np.array([[0, 1], [1, 2], [0, 2]], np.int32)


def _floor(o, ql, qe):
    """Count, floor and ceiling of the bytes of the default order and filter."""
    oc = oracle.Cst(o, ql, qe)
    k = len(ql)
    allow = {u: oc.cand(u).tolist() for u in range(k)}
    pos = {int(u): i for i, u in enumerate(oc.order)}
    par = [0] + [pos[int(oc.parent[int(oc.order[i])])] for i in range(1, k)]
    return oracle.match(o, ql, qe, order=oc.order, par=par, allow=allow, want_balg=True)


def _check(g, o, ql, qe, emit=0):
    """Tree, count, floor of the bytes, counts under limits and with few cells
    for donated runs, and the embeddings if there are at most `emit`."""
    ql = np.asarray(ql, np.int32)
    gc = F.Cst(g, ql, qe)
    compare_cst(gc, oracle.Cst(o, ql, qe), len(ql))
    want = _floor(o, ql, qe)
    n = want["count"]
    for cells in (0, 3, 129, 1000):
        assert F.match(gc, cfg=F.default_config(queue_cells=cells))["count"] == n
        assert F.last_match_floor_bytes() == want["balg"], cells
        assert F.last_match_bytes() >= want["balg"]
    chunks = F.Chunks(gc, F.default_config(delta_w=max(1, gc.W // 50)))
    assert F.match(gc, chunks)["count"] == n
    for lim in {1, max(1, n // 2), n + 1}:
        assert F.match(gc, cfg=F.default_config(limit=lim))["count"] == min(n, lim)
    counts, status = F.Batch(g, 2, F.default_config()).run([(ql, qe)] * 2)
    assert status.tolist() == [0, 0] and counts.tolist() == [n, n]
    if n <= emit:
        r = F.match(gc, k=n + 2)
        assert r["written"] == n
        rows = sorted_rows(r["emb"][:n].astype(np.int32))
        assert np.array_equal(rows, oracle.match(o, ql, qe, max_emb=emit + 1)["emb"])


def _bipartite(rng, degs, nb, lab_a=0, lab_b=1):
    """len(degs) vertices of label A with degs[i] distinct neighbours among nb
    vertices of label B."""
    na = len(degs)
    e = [np.stack([np.full(d, i), na + rng.choice(nb, d, replace=False)], 1) for i, d in enumerate(degs)]
    lab = np.concatenate([np.full(na, lab_a), np.full(nb, lab_b)]).astype(np.int32)
    return na + nb, np.concatenate(e).astype(np.int32), lab


# ------------------------------------------------------------------- loader

# few labels: a table of segment starts; many for so few edges: a directory of
# runs; ids and labels beyond one 64-bit key: rows exported by id
@pytest.mark.parametrize("n,m,L,by_id", [(1, 0, 1, False), (900, 4000, 3, False), (4000, 20_000, 5000, False),
                                         (5_000_000, 200_000, 300_001, True)])
def test_loader_label_lookup(n, m, L, by_id):
    rng = np.random.default_rng(n)
    e = rng.integers(0, n, size=(m, 2)).astype(np.int32)
    lab = rng.integers(0, min(L, 40), size=n).astype(np.int32)
    lab[-1] = L - 1
    g, o = F.Graph(n, e, lab), oracle.Graph(n, e, lab)
    off, col = g.csr()
    ooff, ocol = o.csr() if by_id else csr_by_label(*o.csr(), lab)
    assert np.array_equal(off, ooff) and np.array_equal(col, ocol)
    if m:
        a = e[e[:, 0] != e[:, 1]][:3]
        for x, y in a:
            ql = np.array([lab[x], lab[y], lab[x]], np.int32)
            compare_cst(F.Cst(g, ql, PATH3), oracle.Cst(o, ql, PATH3), 3)


# both sorts of the loader at the edges of a 2048-key tile and of a warp's 256
# (vertices: one key each; edges: two), few distinct keys and many
@pytest.mark.parametrize("n", [2, 255, 256, 257, 2047, 2048, 2049, 6145])
@pytest.mark.parametrize("m", [1, 127, 128, 129, 1023, 1024, 1025, 5000])
def test_loader_sort_tiles(n, m):
    rng = np.random.default_rng(n * 10_000 + m)
    e = rng.integers(0, n, size=(m, 2)).astype(np.int32)
    lab = rng.integers(0, 300, size=n).astype(np.int32)
    g = F.Graph(n, e, lab)
    off, col = g.csr()
    ooff, ocol = csr_by_label(*oracle.Graph(n, e, lab).csr(), lab)
    assert np.array_equal(off, ooff) and np.array_equal(col, ocol)


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_loader_takes_device_edges_at_any_word(shift):
    import torch
    rng = np.random.default_rng(shift)
    n, m = 700, 3001
    e = rng.integers(0, n, size=(m, 2)).astype(np.int32)
    lab = rng.integers(0, 5, size=n).astype(np.int32)
    buf = torch.zeros(2 * m + shift, dtype=torch.int32, device="cuda")
    buf[shift:] = torch.from_numpy(e.reshape(-1)).cuda()
    lbuf = torch.zeros(n + shift, dtype=torch.int32, device="cuda")
    lbuf[shift:] = torch.from_numpy(lab).cuda()
    g = F.Graph(n, buf[shift:].view(m, 2), lbuf[shift:], device=True)
    off, col = g.csr()
    ooff, ocol = csr_by_label(*oracle.Graph(n, e, lab).csr(), lab)
    assert np.array_equal(off, ooff) and np.array_equal(col, ocol)


# -------------------------------------------------------------------- lists

# rows at the edges of a 512-entry tile, of a 32-row window and of a long row
EDGE_ROWS = [1, 2, 31, 32, 33, 127, 128, 129, 511, 512, 513, 1023, 1024, 1025, 2047, 2048, 2049, 5000]


# label-B vertices: a small set, and 32-bit words around the two sizes at which
# the set's copy in shared memory costs a block per SM and no longer fits
@pytest.mark.parametrize("nb", [5000, 8192 * 32, 8192 * 32 + 1, 12800 * 32, 12800 * 32 + 1, 500_000])
def test_list_rows_and_set_sizes(nb):
    rng = np.random.default_rng(nb)
    n, e, lab = _bipartite(rng, EDGE_ROWS + [1] * 40 + EDGE_ROWS[::-1], nb)
    g, o = F.Graph(n, e, lab), oracle.Graph(n, e, lab)
    for ql, qe in (([0, 1], [[0, 1]]), ([1, 0, 1], PATH3), ([0, 1, 0], PATH3)):
        ql, qe = np.array(ql, np.int32), np.array(qe, np.int32)
        gc = F.Cst(g, ql, qe)
        compare_cst(gc, oracle.Cst(o, ql, qe), len(ql))
        (c,), _ = F.build_csts(g, [(ql, qe)])
        compare_cst(c, oracle.Cst(o, ql, qe), len(ql))


@pytest.mark.parametrize("hits", ["none", "first", "last"])
def test_long_rows_of_the_support_test(hits):
    """A-vertices with many B-neighbours of which none, the first or the last
    has the C-neighbour that the query asks for."""
    rng = np.random.default_rng(5)
    nb = 6000
    degs = [2046, 2047, 2048, 2049, 4096, 5999]
    n, e, lab = _bipartite(rng, degs, nb)
    na = len(degs)
    with_c = []
    for i in range(na):
        row = np.sort(e[e[:, 0] == i, 1])
        if hits != "none" and i % 2 == 0:
            with_c.append(row[0] if hits == "first" else row[-1])
    with_c += [na + nb - 1]                                   # one more, so that C(B) is not empty
    c = np.arange(n, n + len(with_c))
    e = np.concatenate([e, np.stack([with_c, c], 1)]).astype(np.int32)
    lab = np.concatenate([lab, np.full(len(c), 2, np.int32)])
    n += len(c)
    g, o = F.Graph(n, e, lab), oracle.Graph(n, e, lab)
    _check(g, o, [0, 1, 2], PATH3, emit=10_000)


# ------------------------------------------------------------------ matcher

@pytest.mark.parametrize("seed", range(6))
def test_merges_at_the_edges_of_a_tile(seed):
    """Non-tree checks against lists of about a tile (128 entries), far
    shorter and far longer, that start at every offset within 16 bytes."""
    rng = np.random.default_rng(100 + seed)
    sizes = [1, 3, 4, 5, 31, 33, 100, 126, 127, 128, 129, 130, 255, 257, 600, 2900]
    na, nb, nc = 5, 24, 3000
    a, b, c = np.arange(na), na + np.arange(nb), na + nb + np.arange(nc)
    e = [(x, y) for x in a for y in b]
    for x in np.concatenate([a, b]):
        e += [(x, y) for y in rng.choice(c, sizes[int(rng.integers(0, len(sizes)))], replace=False)]
    n = na + nb + nc
    lab = np.concatenate([np.zeros(na), np.ones(nb), np.full(nc, 2)]).astype(np.int32)
    e = np.array(e, np.int32)
    g, o = F.Graph(n, e, lab), oracle.Graph(n, e, lab)
    _check(g, o, [0, 1, 2], TRIANGLE, emit=5000)
    _check(g, o, [0, 1, 2, 1], np.array([[0, 1], [1, 2], [0, 2], [0, 3], [2, 3]], np.int32))


# the last position's ranges: around 32 entries (the short form's line), a
# group of 32 quads, and several; B shares A's label or not
@pytest.mark.parametrize("same", [False, True])
@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 31, 32, 33, 34, 63, 65, 127, 128, 129, 130, 515, 2100])
def test_flat_last_position(d, same):
    rng = np.random.default_rng(d)
    degs = [d, max(1, d - 1), d + 1, 1, d, 2, d + 3]
    n, e, lab = _bipartite(rng, degs, 2200)
    if same:
        lab[:] = 0
    g, o = F.Graph(n, e, lab), oracle.Graph(n, e, lab)
    _check(g, o, [0, 0 if same else 1, 0], PATH3, emit=3000)
    _check(g, o, [0 if same else 1, 0, 0 if same else 1], PATH3, emit=3000)


@pytest.mark.parametrize("k,labels", [(2, 1), (3, 1), (5, 1), (6, 1), (15, 4), (16, 4), (17, 4), (16, 1), (17, 1)])
def test_flat_and_general_search_by_query_size(k, labels):
    """Paths and cycles in a ring with chords: up to 16 vertices are searched
    flat, with up to four earlier images compared in the short form."""
    n = 240
    e = np.array([(i, (i + 1) % n) for i in range(n)] + [(i, (i + 7) % n) for i in range(0, n, 40)], np.int32)
    lab = (np.arange(n) % labels).astype(np.int32)
    g, o = F.Graph(n, e, lab), oracle.Graph(n, e, lab)
    ql = np.arange(k) % labels
    _check(g, o, ql, np.array([(i, i + 1) for i in range(k - 1)], np.int32), emit=20_000)
    if k > 2:
        ring = np.array([(i, (i + 1) % k) for i in range(k)], np.int32)
        _check(g, o, ql, ring, emit=20_000)


@pytest.mark.parametrize("nq", [31, 32, 33, 64, 65, 131])
def test_batches_around_the_window_of_queries(nq):
    """Warps go from a query to the 32nd after it: every query is finished,
    whatever the number, with some that are invalid or have no embedding."""
    rng = np.random.default_rng(nq)
    n, m = 500, 3000
    e = rng.integers(0, n, size=(m, 2)).astype(np.int32)
    lab = rng.integers(0, 4, size=n).astype(np.int32)
    g, o = F.Graph(n, e, lab), oracle.Graph(n, e, lab)
    qs = []
    for i in range(nq):
        k = int(rng.integers(1, 6))
        ql = rng.integers(0, 5 if i % 7 == 0 else 4, size=k).astype(np.int32)      # label 4: in no vertex
        qe = [(int(rng.integers(0, v)), v) for v in range(1, k)] + ([(0, 2)] if k > 2 else [])
        qs.append((ql, np.array(sorted(set(qe)), np.int32).reshape(-1, 2)))
    qs[nq // 2] = (np.zeros(3, np.int32), np.array([[0, 1]], np.int32))            # disconnected
    lim = 5000
    counts, status = F.Batch(g, nq, F.default_config(limit=lim, build_rule=2)).run(qs)
    for i, (ql, qe) in enumerate(qs):
        if i == nq // 2:
            assert status[i] == F.FAST_ERR_INVALID
            continue
        assert status[i] == 0 and counts[i] == oracle.match(o, ql, qe, limit=lim)["count"], i


# ---------------------------------------------------------------- partition

@pytest.mark.parametrize("div", [1, 30, 3000])
def test_chunk_fields_one_by_one(div):
    rng = np.random.default_rng(div)
    n, m = 3000, 40_000
    e = rng.integers(0, n, size=(m, 2)).astype(np.int32)
    lab = rng.integers(0, 3, size=n).astype(np.int32)
    g, o = F.Graph(n, e, lab), oracle.Graph(n, e, lab)
    ql, qe = np.array([0, 1, 2, 0], np.int32), np.array([[0, 1], [1, 2], [2, 3]], np.int32)
    gc, oc = F.Cst(g, ql, qe), oracle.Cst(o, ql, qe)
    delta = max(1, gc.W // div)
    ch = F.Chunks(gc, F.default_config(delta_w=delta, max_chunks=1 << 16))
    want = oc.partition(delta)
    assert ch.n == len(want)
    assert [(j, a, b, w, i) for j, _, a, b, w, i in ch.copy()] == [(j, a, b, w, i) for j, _, a, b, w, i in want]
    assert ch.weights().tolist() == [x[4] for x in want]
    assert ch.w_sum == sum(x[4] for x in want)
    assert F.match(gc, ch)["count"] == oracle.count(o, ql, qe)
