"""Performance cases: the work a user of this library has it do, through the
package's public entry points (``Graph``, ``Cst``, ``Chunks``, ``match``,
``build_csts``, ``partition_many``, ``Batch``).

Graphs and queries follow the repository's own workloads: Erdos-Renyi graphs,
Chung-Lu graphs of exponent 2.1 with Zipf(1.0) labels, R-MAT graphs
(a=.57, b=c=.19), and random-walk queries of 4 to 32 vertices, dense and
sparse alternating.  They are drawn here with torch, on the GPU, from the
seed alone.

A case's ``kind`` says which entry points a pass calls:

* ``load``   an edge list in host memory becomes a resident graph, and its CSR
             is read back;
* ``query``  queries one at a time: candidate search tree, partition, match;
* ``build``  the trees and partitions of many queries together, no matching;
* ``batch``  many queries in one reusable batch (builds, partitions, one
             matcher launch);
* ``count``  one matcher call over a tree and partition already at hand;
* ``emit``   the same with every embedding written to a device buffer.
"""
import math
import random

import numpy as np
import torch

import paper_2102_10768_gb300 as F

DEV = "cuda"


def listed():
    return [
        # The smallest call there is: one 4-vertex query on a 10,000-vertex
        # graph with the library's default rules, embeddings written out.
        dict(name="er10k_one_query", kind="query", graph="er", n=10_000, m=40_000, labels=8, sizes="4", nq=1,
             order=0, filter=0, limit=0, max_chunks=1 << 16, rows=1 << 14),
        # Interactive use on a mid-size graph with the default (path-based)
        # order and label-and-degree filter: two small queries in turn.
        dict(name="powerlaw100k_default_rules", kind="query", graph="powerlaw", n=100_000, m=1_600_000, labels=16,
             sizes="6,8", nq=2, order=0, filter=0, limit=1 << 16, max_chunks=1 << 16, rows=0),
        # The per-query path of the benchmark: one query of each size, one
        # after the other, on the 1M/16M power-law graph.
        dict(name="powerlaw1m_per_query", kind="query", graph="powerlaw", n=1_000_000, m=16_000_000, labels=16,
             sizes="4,8,16,24,32", nq=5, order=1, filter=1, limit=1 << 22, max_chunks=4096, rows=0),
        # What a group worker of the request loop runs at low load: a group
        # of one request, the largest query size.
        dict(name="rmat20_one_request", kind="batch", graph="rmat", n=1 << 20, m=16 << 20, labels=32, sizes="32",
             nq=1, order=1, filter=1, limit=1 << 16, full=0),
        # The request loop under load: a group of eight requests of all sizes.
        dict(name="rmat20_group_of_8", kind="batch", graph="rmat", n=1 << 20, m=16 << 20, labels=32,
             sizes="4,8,12,16,20,24,28,32", nq=8, order=1, filter=1, limit=1 << 16, full=0),
        # A small batch of the benchmark's mix.
        dict(name="powerlaw1m_batch_40", kind="batch", graph="powerlaw", n=1_000_000, m=16_000_000, labels=16,
             sizes="4,8,16,24,32", nq=40, order=1, filter=1, limit=1 << 22, full=0),
        # The benchmark's step at a quarter of its 1,000 queries: throughput.
        dict(name="powerlaw1m_batch_250", kind="batch", graph="powerlaw", n=1_000_000, m=16_000_000, labels=16,
             sizes="4,8,16,24,32", nq=250, order=1, filter=1, limit=1 << 22, full=0),
        # Building trees and partitions for later use, with the weaker
        # default filter, whose candidate sets are the larger ones.
        dict(name="powerlaw1m_build_30", kind="build", graph="powerlaw", n=1_000_000, m=16_000_000, labels=16,
             sizes="7,15,23", nq=30, order=0, filter=0, max_chunks=4096),
        # The paper's own task on the power-law graph: every embedding of
        # small queries counted, no limit, in one batch (of a pool of 200
        # queries, the 12 with the smallest workload estimates).
        dict(name="powerlaw1m_full_count", kind="batch", graph="powerlaw", n=1_000_000, m=16_000_000, labels=16,
             sizes="4", nq=200, order=1, filter=1, limit=0, full=12),
        # Complete enumeration where every list is short (two entries on
        # average) and the search is deep: the matcher alone.
        dict(name="er1m_deep_count", kind="count", graph="er", n=1_000_000, m=16_000_000, labels=16, sizes="10",
             nq=1, order=1, filter=1, max_chunks=4096),
        # Every embedding written out, millions of rows.
        dict(name="er64k_emit", kind="emit", graph="er", n=65_536, m=1_048_576, labels=4, sizes="4", nq=1,
             order=1, filter=0, max_chunks=4096, rows=1 << 24),
        # A graph comes in: edge list in host memory to a resident graph.
        dict(name="powerlaw1m_load", kind="load", graph="powerlaw", n=1_000_000, m=16_000_000, labels=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "batch", "batch", "build", "count", "emit", "load"])
    c = dict(kind=kind)
    if kind in ("count", "emit"):
        c["graph"] = "er"
    else:
        c["graph"] = rng.choice(["powerlaw", "powerlaw", "rmat", "er"])
    if kind == "emit":
        # embeddings expected: n * (degree / labels)^3 / labels, up to some millions
        c["n"] = _log(rng, 8_000, 65_536)
        c["labels"] = rng.randint(4, 8)
        c["m"] = int(c["n"] * c["labels"] * rng.uniform(2.0, 4.0) / 2)
        return c | dict(sizes="4", nq=1, order=rng.choice([0, 1]), filter=rng.choice([0, 1]), max_chunks=4096,
                        rows=1 << 22)
    if kind == "count":
        # a tree query of k vertices has about n * (degree / labels)^(k-1) / labels embeddings
        c["n"] = _log(rng, 50_000, 1_000_000)
        c["labels"] = rng.randint(8, 24)
        k = rng.randint(5, 10)
        c["m"] = int(c["n"] * c["labels"] * rng.uniform(1.2, 2.0) / 2)
        return c | dict(sizes=str(k), nq=1, order=rng.choice([0, 1, 2, 3]), filter=rng.choice([0, 1]), max_chunks=4096)
    if c["graph"] == "rmat":
        c["n"] = 1 << rng.randint(16, 20)
        c["m"] = c["n"] * rng.randint(8, 16)
        c["labels"] = rng.randint(12, 40)
    elif c["graph"] == "er":
        c["n"] = _log(rng, 10_000, 1_000_000)
        c["m"] = c["n"] * rng.randint(4, 12)
        c["labels"] = rng.randint(8, 32)
    else:
        c["n"] = _log(rng, 60_000, 1_000_000)
        c["m"] = c["n"] * rng.randint(8, 16)
        c["labels"] = rng.randint(10, 24)
    if kind == "load":
        return c
    sizes = ",".join(str(s) for s in sorted(rng.sample(range(4, 33), rng.randint(1, 5))))
    order = rng.choice([0, 1, 1, 2, 3])
    if kind == "query":
        limit = 1 << 16 if order != 1 else _log(rng, 1 << 14, 1 << 20)
        return c | dict(sizes=sizes, nq=rng.randint(1, 5), order=order, filter=rng.choice([0, 1]), limit=limit,
                        max_chunks=rng.choice([1024, 4096, 1 << 16]), rows=0)
    if kind == "build":
        return c | dict(sizes=sizes, nq=_log(rng, 1, 30), order=order, filter=rng.choice([0, 1]), max_chunks=4096)
    return c | dict(sizes=sizes, nq=_log(rng, 1, 120), order=1, filter=1, limit=_log(rng, 1 << 14, 1 << 22), full=0)


# ------------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _distinct(n, m, g, pairs):
    """m distinct undirected edges (a < b) out of what pairs(count) draws."""
    keys = torch.empty(0, dtype=torch.int64, device=DEV)
    want = m + m // 4
    for _ in range(64):
        a, b = pairs(want)
        ok = a != b
        k = (torch.minimum(a, b) * n + torch.maximum(a, b))[ok]
        keys = torch.unique(torch.cat([keys, k]))
        if keys.numel() >= m:
            break
        want = 2 * (m - keys.numel()) + 1024
    keys = keys[torch.randperm(keys.numel(), generator=g, device=DEV)[:m]]
    flip = torch.rand(keys.numel(), generator=g, device=DEV) < 0.5
    a, b = keys // n, keys % n
    return torch.stack([torch.where(flip, b, a), torch.where(flip, a, b)], 1).to(torch.int32).contiguous()


def _graph(case, seed):
    """(edges int32 [m, 2], labels int32 [n]) on the GPU."""
    n, m, kind = case["n"], case["m"], case["graph"]
    g = _gen(seed)
    if kind == "er":
        def pairs(c):
            return (torch.randint(0, n, (c,), generator=g, device=DEV),
                    torch.randint(0, n, (c,), generator=g, device=DEV))
    elif kind == "powerlaw":
        w = torch.arange(1, n + 1, device=DEV, dtype=torch.float64) ** (-1.0 / 1.1)     # exponent 2.1
        cum = torch.cumsum(w, 0)

        def pairs(c):
            u = torch.rand((2, c), generator=g, device=DEV, dtype=torch.float64) * cum[-1]
            x = torch.searchsorted(cum, u).clamp_(max=n - 1)
            return x[0], x[1]
    else:
        scale = n.bit_length() - 1
        perm = torch.randperm(n, generator=g, device=DEV)

        def pairs(c):
            a = torch.zeros(c, dtype=torch.int64, device=DEV)
            b = torch.zeros(c, dtype=torch.int64, device=DEV)
            for _ in range(scale):
                r = torch.rand(c, generator=g, device=DEV)
                a = 2 * a + (r >= 0.76)
                b = 2 * b + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
            return perm[a], perm[b]
    edges = _distinct(n, m, g, pairs)
    if kind == "er":
        lab = torch.randint(0, case["labels"], (n,), generator=g, device=DEV)
    else:
        z = torch.cumsum(1.0 / torch.arange(1, case["labels"] + 1, device=DEV, dtype=torch.float64), 0)
        lab = torch.searchsorted(z, torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * z[-1])
        lab = lab.clamp_(max=case["labels"] - 1)
    return edges, lab.to(torch.int32)


def _both_ways(edges, n):
    """Sorted keys row * n + col of the adjacency."""
    a, b = edges[:, 0].long(), edges[:, 1].long()
    return torch.sort(torch.cat([a * n + b, b * n + a]))[0]


def _walks(edges, lab, n, sizes, nq, seed):
    """nq random-walk queries, sizes in turn; dense (every edge among the
    walk's vertices, average degree above 3 where the graph allows it) and
    sparse (the walk's tree and extra edges up to 1.5 k) alternating."""
    keys = _both_ways(edges, n)
    ptr = torch.searchsorted(keys, torch.arange(n + 1, device=DEV) * n).cpu().numpy()
    col = (keys % n).to(torch.int32).cpu().numpy()
    del keys
    labels = lab.cpu().numpy()
    rng = random.Random(seed)
    out = []
    for i in range(nq):
        k = sizes[i % len(sizes)]
        dense = (i // len(sizes) + i) % 2 == 0
        for attempt in range(2000):
            cur = rng.randrange(n)
            verts, tree, steps = [cur], [], 0
            while len(verts) < k and steps < 200 * k + 1000:
                lo, hi = int(ptr[cur]), int(ptr[cur + 1])
                if lo == hi:
                    break
                nx = int(col[lo + rng.randrange(hi - lo)])
                if nx not in verts:
                    tree.append((verts.index(cur), len(verts)))
                    verts.append(nx)
                cur = nx
                steps += 1
            if len(verts) < k:
                continue
            pairs = []
            va = np.array(verts, dtype=np.int32)
            for x in range(k):
                row = col[ptr[verts[x]]:ptr[verts[x] + 1]]
                at = np.searchsorted(row, va[x + 1:])
                hit = (at < row.size) & (row[np.minimum(at, row.size - 1)] == va[x + 1:])
                pairs += [(x, x + 1 + int(y)) for y in np.nonzero(hit)[0]]
            if dense and k > 4 and 2 * len(pairs) <= 3 * k and attempt < 40:
                continue
            if not dense:
                extra = [p for p in pairs if p not in set(tree)]
                rng.shuffle(extra)
                pairs = tree + extra[:max(0, 3 * k // 2 - len(tree))]
            out.append((labels[va].astype(np.int32), np.array(pairs, dtype=np.int32)))
            break
        else:
            raise RuntimeError("no random walk of %d vertices found" % k)
    return out


def _inputs(case, seed):
    edges, lab = _graph(case, seed)
    qs = []
    if case["kind"] != "load":
        sizes = [int(s) for s in case["sizes"].split(",")]
        qs = _walks(edges, lab, case["n"], sizes, case["nq"], seed)
    return edges, lab, qs


def _config(case):
    kw = dict(delta_w=1 << 20, max_chunks=case.get("max_chunks", 4096), order_rule=case["order"],
              filter_rule=case["filter"], limit=case.get("limit", 0))
    if case["kind"] == "batch":
        kw["build_rule"] = 2
    return F.default_config(**kw)


def prepare(case, seed):
    edges, lab, qs = _inputs(case, seed)
    s = dict(case=case, queries=qs)
    if case["kind"] == "load":
        s["edges"], s["labels"] = edges.cpu().numpy(), lab.cpu().numpy()
        return s
    s["graph"] = F.Graph(case["n"], edges, lab, device=True)
    s["cfg"] = _config(case)
    if case["kind"] == "batch":
        if case["full"]:
            # the queries of the smallest workload estimates, an upper bound of their counts
            csts, _ = F.build_csts(s["graph"], qs, s["cfg"])
            by_w = sorted((c.W, i) for i, c in enumerate(csts))
            s["queries"] = [qs[i] for _, i in by_w[:case["full"]]]
            del csts
        s["batch"] = F.Batch(s["graph"], len(s["queries"]), s["cfg"])
    elif case["kind"] in ("count", "emit"):
        s["cst"] = F.Cst(s["graph"], *qs[0], s["cfg"])
        s["chunks"] = F.Chunks(s["cst"], s["cfg"])
    if case.get("rows"):
        s["rows"] = torch.empty((case["rows"], len(qs[0][0])), dtype=torch.int32, device=DEV)
    return s


# --------------------------------------------------------------------- a pass

def _keys(rows, n, size):
    """The embeddings as sorted 64-bit keys (the matcher writes them in no
    order), and zeros up to `size`."""
    bits = max(1, (n - 1).bit_length())
    key = rows[:, 0].long()
    for p in range(1, rows.shape[1]):
        key = (key << bits) | rows[:, p].long()
    out = torch.zeros(size, dtype=torch.int64, device=DEV)
    out[:key.numel()] = torch.sort(key)[0]
    return out


def _weights(chunks, size):
    """The chunks' workload estimates, and zeros up to `size`."""
    out = np.zeros(size, np.int64)
    w = chunks.weights().view(np.int64)
    out[:w.size] = w
    return out


def _tree(c):
    return dict(order=c.order, parent=c.parent, ncand=c.ncand, W=np.array([c.W], np.uint64).view(np.int64), Wf=c.Wf)


def _joined(parts):
    """{name: one array} of a list of dicts of arrays and numbers."""
    return {k: np.concatenate([np.atleast_1d(p[k]) for p in parts]) for k in parts[0]}


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "load":
        g = F.Graph(case["n"], state["edges"], state["labels"])
        off, col = g.csr()
        info = g.info()
        g.close()
        return dict(off=off, col=col, info=np.array([info[k] for k in sorted(info)], np.int64))
    cfg = state["cfg"]
    if kind == "batch":
        counts, status = state["batch"].run(state["queries"])
        return dict(counts=counts, status=status, chunks=state["batch"].timing()["chunks"])
    if kind == "count":
        r = F.match(state["cst"], state["chunks"], cfg=cfg)
        return dict(count=r["count"])
    if kind == "emit":
        r = F.match(state["cst"], state["chunks"], k=state["rows"].shape[0], emb_out=state["rows"], cfg=cfg)
        return dict(count=r["count"], rows=_keys(state["rows"][:r["written"]], case["n"], case["rows"]))
    if kind == "build":
        csts, _ = F.build_csts(state["graph"], state["queries"], cfg)
        chunks, _ = F.partition_many(csts, cfg)
        out = _joined([_tree(c) | dict(chunks=ch.n, weights=_weights(ch, case["max_chunks"]))
                       for c, ch in zip(csts, chunks)])
        for h in chunks + csts:
            h.close()
        return out
    parts, rows = [], None
    for ql, qe in state["queries"]:
        c = F.Cst(state["graph"], ql, qe, cfg)
        ch = F.Chunks(c, cfg)
        buf = state.get("rows")
        r = F.match(c, ch, k=0 if buf is None else buf.shape[0], emb_out=buf, cfg=cfg)
        if buf is not None:
            rows = _keys(buf[:r["written"]], case["n"], case["rows"])
        parts.append(_tree(c) | dict(chunks=ch.n, wsum=np.array([ch.w_sum], np.uint64).view(np.int64),
                                     count=r["count"]))
        ch.close()
        c.close()
    return _joined(parts) | dict(rows=rows)


# ---------------------------------------------------------------- what it needs

def work(case):
    """Bytes: per query vertex the ids of its label's vertices, per query edge
    the adjacency between the two labels (uniform labels assumed), each read
    once; the last vertex of every embedding counted or each row written."""
    n, m, L = case["n"], case["m"], case["labels"]
    if case["kind"] == "load":
        return {"bytes": 8 * m + 4 * n + 8 * (n + 1) + 8 * m, "flops": 0}
    ks = [int(s) for s in case["sizes"].split(",")]
    nq = case["nq"]
    k = sum(ks[i % len(ks)] for i in range(nq)) / nq
    tree = k * 4 * n / L + 1.5 * k * 4 * 2 * m / (L * L)
    if case["kind"] == "build":
        return {"bytes": int(nq * tree), "flops": 0}
    if case["kind"] in ("count", "emit"):
        found = n / L * (2 * m / n / L) ** (k - 1)
        return {"bytes": int(tree + found * 4 * (k if case["kind"] == "emit" else 1)), "flops": 0}
    if case["kind"] == "batch" and case["full"]:
        return {"bytes": int(case["full"] * (tree + 4 * 2.0 ** 27)), "flops": 0}
    found = case["limit"] or n / L * (2 * m / n / L) ** (k - 1)
    return {"bytes": int(nq * (tree + 4 * found)), "flops": 0}


# ---------------------------------------------------------------- in 64 bits

class _Adj:
    """Adjacency sorted by (label of the row, label of the neighbour, row, neighbour)."""

    def __init__(self, edges, lab, n, L):
        self.n, self.L, self.lab = n, L, lab.long()
        keys = _both_ways(edges, n)
        src, dst = keys // n, keys % n
        pair = self.lab[src] * L + self.lab[dst]
        pair, at = torch.sort(pair, stable=True)
        self.src, self.dst = src[at], dst[at]
        self.beg = torch.searchsorted(pair, torch.arange(L * L + 1, device=DEV)).tolist()
        self.keys = keys
        self.deg = torch.bincount(src, minlength=n)
        self.near = torch.bincount(src * L + self.lab[dst], minlength=n * L).view(n, L)

    def between(self, a, b):
        s = slice(self.beg[a * self.L + b], self.beg[a * self.L + b + 1])
        return self.src[s], self.dst[s]


def _tree_of(A, ql, qe, nlf):
    """Root, parents, refined candidate masks and the float64 workload estimate
    of a query: filter, top-down, one bottom-up pass, sums over the lists."""
    k, nb = len(ql), [set() for _ in ql]
    for a, b in qe.tolist():
        nb[a].add(b)
        nb[b].add(a)
    C = []
    for u in range(k):
        ok = (A.lab == int(ql[u])) & (A.deg >= len(nb[u]))
        if nlf:
            need = {}
            for w in nb[u]:
                need[int(ql[w])] = need.get(int(ql[w]), 0) + 1
            for l, c in need.items():
                ok &= A.near[:, l] >= c
        C.append(ok)
    size = [int(c.sum()) for c in C]
    root = 0
    for u in range(1, k):
        if size[u] * len(nb[root]) < size[root] * len(nb[u]):
            root = u
    parent, bfs = [-2] * k, [root]
    parent[root] = -1
    for u in bfs:
        for w in sorted(nb[u]):
            if parent[w] == -2:
                parent[w] = u
                bfs.append(w)
    for u in bfs[1:]:
        s, d = A.between(int(ql[parent[u]]), int(ql[u]))
        hit = torch.zeros(A.n, dtype=torch.bool, device=DEV)
        hit[d[C[parent[u]][s]]] = True
        C[u] &= hit
    value = [None] * k
    for u in reversed(bfs):
        kids = [w for w in range(k) if parent[w] == u]
        for w in kids:
            s, d = A.between(int(ql[u]), int(ql[w]))
            hit = torch.zeros(A.n, dtype=torch.bool, device=DEV)
            hit[s[C[w][d]]] = True
            C[u] &= hit
        v = C[u].double()
        for w in kids:
            s, d = A.between(int(ql[u]), int(ql[w]))
            v *= torch.zeros(A.n, dtype=torch.float64, device=DEV).index_add_(0, s, value[w][d])
            value[w] = None
        value[u] = v
    return parent, [int(c.sum()) for c in C], float(value[root].sum())


def _embeddings(A, ql, qe, want_rows):
    """Every embedding of a small query by joins along a breadth-first order:
    their number, or their rows."""
    k, nb = len(ql), [set() for _ in ql]
    for a, b in qe.tolist():
        nb[a].add(b)
        nb[b].add(a)
    order = [0]
    for u in order:
        order += [w for w in sorted(nb[u]) if w not in order]
    count, rows = 0, []
    first = torch.nonzero(A.lab == int(ql[order[0]])).squeeze(1)
    todo = [p[:, None] for p in torch.split(first, 1 << 16)][::-1]
    while todo:
        part = todo.pop()
        i = part.shape[1]
        if i == k or part.shape[0] == 0:
            count += part.shape[0]
            if want_rows and part.shape[0]:
                at = [order.index(u) for u in range(k)]
                rows.append(part[:, at])
            continue
        u = order[i]
        placed = [order.index(w) for w in nb[u] if w in order[:i]]
        p = min(placed)
        src, dst = A.between(int(ql[order[p]]), int(ql[u]))
        x = part[:, p].contiguous()
        lo, hi = torch.searchsorted(src, x), torch.searchsorted(src, x, right=True)
        num = hi - lo
        row = torch.repeat_interleave(torch.arange(part.shape[0], device=DEV), num)
        off = torch.arange(row.numel(), device=DEV) - (torch.cumsum(num, 0) - num)[row]
        v = dst[lo[row] + off]
        ok = torch.ones_like(v, dtype=torch.bool)
        for q in range(i):
            if ql[order[q]] == ql[u]:
                ok &= part[row, q] != v
        for q in placed:
            if q != p:
                key = part[row, q] * A.n + v
                at = torch.searchsorted(A.keys, key).clamp_(max=A.keys.numel() - 1)
                ok &= A.keys[at] == key
        new = torch.cat([part[row[ok]], v[ok][:, None]], 1)
        todo += list(torch.split(new, 1 << 20))[::-1]
    return count, torch.cat(rows) if rows else torch.empty((0, k), dtype=torch.int64, device=DEV)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None                      # counts up to a limit, or of billions of embeddings
    edges, lab, qs = _inputs(case, seed)
    n, L = case["n"], int(lab.max()) + 1
    if kind == "load":
        a, b = edges[:, 0].long(), edges[:, 1].long()
        src, dst = torch.cat([a, b]), torch.cat([b, a])
        key = torch.sort((src * L + lab.long()[dst]) * n + dst)[0]
        deg = torch.bincount(src, minlength=n)
        off = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(deg, 0)])
        return dict(off=off, col=(key % n).to(torch.int32),
                    info=np.array([int(deg.max()), n, 2 * case["m"], L], np.int64))
    A = _Adj(edges, lab, n, L)
    if kind in ("count", "emit"):
        c, rows = _embeddings(A, *qs[0], kind == "emit")
        return dict(count=c) if kind == "count" else dict(count=c, rows=_keys(rows, n, case["rows"]))
    parts = []
    for ql, qe in qs:
        parent, ncand, w = _tree_of(A, ql, qe, case["filter"] == 1)
        parts.append(dict(parent=np.array(parent, np.int32), ncand=np.array(ncand, np.int64), Wf=w))
    out = _joined(parts) | dict(order=None, W=None, chunks=None)
    if kind == "build":
        return out | dict(weights=None)
    out |= dict(wsum=None, count=None, rows=None)
    if case["rows"]:
        c, rows = _embeddings(A, *qs[0], True)
        out |= dict(count=np.array([c]), rows=_keys(rows, n, case["rows"]))
    return out
