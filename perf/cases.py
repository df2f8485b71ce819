"""Measured workloads: index builds and queries through the public binding.

A case names a graph, what is built from it and, for queries, what is asked.
Graphs are seeded and made on the GPU: R-MAT (a, b, c, d = .57, .19, .19, .05,
ids relabelled at random, any vertex count), planted partitions (SBM) and
Erdos-Renyi. A build's outputs are the whole index, copied into the caller's
own device tensors; a query's outputs are its labels.
"""
import math

import numpy as np
import torch

import paper_2012_11188_gb300 as gs

DEVICE = "cuda"


def listed():
    return [
        # The first thing a user does: a small planted partition in host
        # memory, int32 offsets. Launches, copies and waits count most here.
        {"name": "build_sbm_10k_host", "op": "build", "graph": "sbm", "n": 10000, "block": 200,
         "p_in": 0.05, "p_out": 0.0004, "host": True, "kind": "cosine"},
        # A social-network-like graph of ordinary size, Jaccard.
        {"name": "build_rmat_s20_jaccard", "op": "build", "graph": "rmat", "n": 1 << 20, "ef": 16,
         "host": False, "kind": "jaccard"},
        # The largest: the graph the benchmark quotes its headline on.
        {"name": "build_rmat_s24_cosine", "op": "build", "graph": "rmat", "n": 1 << 24, "ef": 16,
         "host": False, "kind": "cosine"},
        # The approximate index on a skewed graph, SimHash and MinHash.
        {"name": "lsh_simhash256_rmat_s22", "op": "lsh", "graph": "rmat", "n": 1 << 22, "ef": 16,
         "host": False, "kind": "cosine", "k": 256, "threshold": 128},
        {"name": "lsh_minhash64_rmat_s22", "op": "lsh", "graph": "rmat", "n": 1 << 22, "ef": 16,
         "host": False, "kind": "jaccard", "k": 64, "threshold": 128},
        # Real-valued edge weights (strengths of ties, affinities).
        {"name": "weighted_rmat_s20", "op": "weighted", "graph": "rmat", "n": 1 << 20, "ef": 16,
         "host": False, "kind": "cosine"},
        # A dense similarity graph shaped like the paper's blood vessel graph.
        {"name": "dense_er_25825", "op": "build", "graph": "er", "n": 25825, "degree": 5400,
         "host": False, "kind": "cosine"},
        # Many small graphs of uneven size in one call (one per user, per
        # day, per sample).
        {"name": "batch_512_sbm", "op": "batch", "graph": "batch", "count": 512, "n_lo": 100,
         "n_hi": 20000, "host": False, "kind": "cosine"},
        # One interactive query of a resident index, small and large graph.
        {"name": "query_sbm_10k_hubs", "op": "query", "graph": "sbm", "n": 10000, "block": 200,
         "p_in": 0.05, "p_out": 0.0004, "host": False, "kind": "cosine", "mu": 3, "eps": 0.25,
         "hubs": True},
        {"name": "query_rmat_s22", "op": "query", "graph": "rmat", "n": 1 << 22, "ef": 16,
         "host": False, "kind": "cosine", "mu": 5, "eps": 0.3, "hubs": False},
        # A server's full batch of queries of different parameters.
        {"name": "query_batch64_rmat_s22", "op": "queries", "graph": "rmat", "n": 1 << 22, "ef": 16,
         "host": False, "kind": "cosine", "count": 64, "hubs": False},
        # The parameter sweep that picks (mu, eps) by modularity.
        {"name": "sweep_rmat_s20", "op": "sweep", "graph": "rmat", "n": 1 << 20, "ef": 16,
         "host": False, "kind": "cosine", "pairs": 594},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, most):
    """A graph of at most about `most` sampled edges."""
    if rng.random() < 0.7:
        ef = rng.choice([6, 8, 12, 16, 16, 24, 32])
        return {"graph": "rmat", "n": _log(rng, 2000, max(4000, most // ef)), "ef": ef}
    n = _log(rng, 1000, min(200000, max(2000, most // 8)))
    return {"graph": "sbm", "n": n, "block": rng.choice([50, 120, 200, 333]),
            "p_in": round(rng.uniform(0.03, 0.2), 3), "p_out": round(4.0 / n, 8)}


def draw(rng):
    op = rng.choice(["build", "build", "build", "lsh", "lsh", "weighted", "dense", "batch", "query",
                     "query", "queries", "sweep"])
    kind = rng.choice(["cosine", "jaccard"])
    if op == "build":
        g = _draw_graph(rng, 1 << 27)
        return {"op": op, **g, "host": g["n"] < 50000 and rng.random() < 0.5, "kind": kind}
    if op == "lsh":
        k = rng.choice([64, 128, 256] if kind == "cosine" else [32, 64, 128])
        return {"op": op, "graph": "rmat", "n": _log(rng, 50000, 1 << 22), "ef": 16, "host": False,
                "kind": kind, "k": k, "threshold": rng.choice([64, 96, 128, 200])}
    if op == "weighted":
        return {"op": op, **_draw_graph(rng, 1 << 25), "host": False, "kind": "cosine"}
    if op == "dense":
        n = _log(rng, 4100, 26000)
        return {"op": "build", "graph": "er", "n": n, "degree": int(n * rng.uniform(0.08, 0.5)),
                "host": False, "kind": kind}
    if op == "batch":
        lo = _log(rng, 60, 1000)
        return {"op": op, "graph": "batch", "count": _log(rng, 4, 512), "n_lo": lo,
                "n_hi": lo * rng.randint(2, 16), "host": False, "kind": kind}
    g = _draw_graph(rng, 1 << 25)
    if op == "query":
        return {"op": op, **g, "host": False, "kind": kind, "mu": rng.randint(2, 16),
                "eps": rng.randint(2, 14) / 20.0, "hubs": rng.random() < 0.5}
    if op == "queries":
        return {"op": op, **g, "host": False, "kind": kind, "count": _log(rng, 2, 64),
                "hubs": rng.random() < 0.3}
    return {"op": "sweep", **_draw_graph(rng, 1 << 22), "host": False, "kind": kind,
            "pairs": _log(rng, 20, 400)}


# ---------------------------------------------------------------- graphs
# A case fixes every graph's vertex and edge counts; the seed decides the rest.
def _gen(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _csr(key, n):
    """CSR (int64 offsets, int32 ids) from one key lo * n + hi per edge."""
    key = torch.sort(torch.cat([key, key % n * n + key // n]))[0]
    rows = torch.arange(n + 1, device=DEVICE, dtype=torch.int64) * n
    off = torch.searchsorted(key, rows)
    return off, (key % n).to(torch.int32)


def _rmat_edges(n, ef):
    return min(int(0.9 * ef * n), n * (n - 1) // 8)


def _rmat(n, ef, seed):
    """R-MAT samples, cleaned, until 0.9 * ef * n edges are there."""
    g = _gen(seed)
    levels = max(1, (n - 1).bit_length())
    perm = torch.randperm(n, generator=g, device=DEVICE)
    want = _rmat_edges(n, ef)
    key = torch.empty(0, dtype=torch.int64, device=DEVICE)
    while len(key) < want:
        parts = [key]
        left = int(1.15 * (want - len(key))) + 1024
        while left > 0:
            m = min(left, 1 << 26)
            left -= m
            src = torch.zeros(m, dtype=torch.int32, device=DEVICE)
            dst = torch.zeros(m, dtype=torch.int32, device=DEVICE)
            for _ in range(levels):
                r = torch.rand(m, generator=g, device=DEVICE)
                down = r >= 0.76
                right = ((r >= 0.57) & ~down) | (r >= 0.95)
                src.mul_(2).add_(down)
                dst.mul_(2).add_(right)
            keep = (src < n) & (dst < n) & (src != dst)
            u, v = perm[src[keep].long()], perm[dst[keep].long()]
            parts.append(torch.minimum(u, v) * n + torch.maximum(u, v))
        key = torch.unique(torch.cat(parts))
    if len(key) > want:
        key = key[torch.randperm(len(key), generator=g, device=DEVICE)[:want]]
    return _csr(key, n)


def _sbm_edges(n, blocks, p_in, p_out):
    """Expected edges of a planted partition (near-equal blocks)."""
    inside = n * (n / blocks - 1) / 2
    return int(p_in * inside + p_out * (n * (n - 1) / 2 - inside))


def _t(x, dtype):
    return torch.tensor(x, device=DEVICE, dtype=dtype)


def _sbm(params, seed):
    """CSR of planted partitions packed in one id range: graph i has ns[i]
    vertices in blocks[i] contiguous near-equal blocks. Pairs are drawn
    somewhat more often than p_in and p_out ask for, cleaned, and thinned to
    the expected number of edges."""
    g = _gen(seed)
    ns, blocks = _t([p[0] for p in params], torch.int64), _t([p[1] for p in params], torch.int64)
    p_in, p_out = _t([p[2] for p in params], torch.float64), _t([p[3] for p in params], torch.float64)
    want = _t([_sbm_edges(*p) for p in params], torch.int64)
    base = torch.cumsum(ns, 0) - ns
    n, nf = int(ns.sum()), ns.double()
    graphs = torch.arange(len(ns), device=DEVICE)
    gid = torch.repeat_interleave(graphs, blocks)  # one entry per block
    b = torch.arange(len(gid), device=DEVICE) - (torch.cumsum(blocks, 0) - blocks)[gid]
    lo, hi = b * ns[gid] // blocks[gid], (b + 1) * ns[gid] // blocks[gid]
    size = (hi - lo).double()
    more = 1.05 + 8 / torch.sqrt(want + 1.0)
    uniform = lambda e: torch.rand(len(e), generator=g, device=DEVICE, dtype=torch.float64)  # noqa: E731
    while True:
        rate = -torch.log1p(-p_in) * more
        cnt = torch.poisson(rate[gid] * size * (size - 1) / 2, generator=g).long()
        e = torch.repeat_interleave(torch.arange(len(gid), device=DEVICE), cnt)
        s = (hi - lo)[e]
        u = (uniform(e) * s).long()
        v = (u + 1 + (uniform(e) * (s - 1)).long()) % s.clamp(min=1)
        first = (base[gid] + lo)[e]
        u, v = first + u, first + v
        # between blocks: drawn over all pairs of a graph, those inside a block dropped
        cnt = torch.poisson(-torch.log1p(-p_out) * more * nf * (nf - 1) / 2, generator=g).long()
        e = torch.repeat_interleave(graphs, cnt)
        x, y = (uniform(e) * nf[e]).long(), (uniform(e) * nf[e]).long()
        keep = ((x + 1) * blocks[e] - 1) // ns[e] != ((y + 1) * blocks[e] - 1) // ns[e]
        u, v = torch.cat([u, (base[e] + x)[keep]]), torch.cat([v, (base[e] + y)[keep]])
        key = torch.unique(torch.minimum(u, v) * n + torch.maximum(u, v))
        of = torch.searchsorted(base, key // n, right=True) - 1  # the edge's graph (ascending)
        have = torch.bincount(of, minlength=len(ns))
        if bool((have >= want).all()):
            break
        more = more * 1.3
    by = torch.argsort(of + uniform(of) * 0.999)  # each graph's edges in a random order
    place = torch.arange(len(by), device=DEVICE) - (torch.cumsum(have, 0) - have)[of]
    return _csr(key[by[place < want[of]]], n)


def _er(n, degree, seed):
    g = _gen(seed)
    want = n * degree // 2
    p = min(1.0, degree / (n - 1) * 1.01)
    a = torch.zeros(n, n, dtype=torch.bool, device=DEVICE)
    for i in range(0, n, 4096):
        j = min(n, i + 4096)
        a[i:j] = torch.rand(j - i, n, generator=g, device=DEVICE) < p
    at = a.triu_(1).view(-1).nonzero()[:, 0]
    drop = torch.randperm(len(at), generator=g, device=DEVICE)[want:]
    a.view(-1)[at[drop]] = False
    a |= a.clone().t()
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEVICE)
    off[1:] = torch.cumsum(a.sum(1), 0)
    return off, a.nonzero()[:, 1].to(torch.int32)


def _batch_params(case):
    """Graphs of a batch: n log-uniform, 2 to 64 blocks, p_in .02 to .2."""
    r = np.random.RandomState(case["count"] + case["n_lo"]).rand(case["count"], 3)
    lo, hi = math.log(case["n_lo"]), math.log(case["n_hi"])
    out = []
    for x, y, z in r.tolist():
        n, p = int(round(math.exp(lo + x * (hi - lo)))), 0.02 + 0.18 * z
        out.append((n, min(n, 2 + int(y * 63)), p, p / 50))
    return out


def _batch(case, seed):
    params = _batch_params(case)
    off, adj = _sbm(params, seed)
    out, v, a0 = [], 0, 0
    for p in params:
        a1 = a0 + 2 * _sbm_edges(*p)
        out.append((off[v:v + p[0] + 1] - a0, adj[a0:a1] - v))
        v, a0 = v + p[0], a1
    return out


def _sbm_params(case):
    n = case["n"]
    return n, max(1, n // case["block"]), case["p_in"], case["p_out"]


def _graph(case, seed):
    if case["graph"] == "rmat":
        return _rmat(case["n"], case["ef"], seed)
    if case["graph"] == "sbm":
        return _sbm([_sbm_params(case)], seed)
    if case["graph"] == "er":
        return _er(case["n"], case["degree"], seed)
    return _batch(case, seed)


def _size(case):
    """Graphs, vertices and arcs of a case's input."""
    g = case["graph"]
    if g == "rmat":
        return 1, case["n"], 2 * _rmat_edges(case["n"], case["ef"])
    if g == "er":
        return 1, case["n"], case["n"] * case["degree"] // 2 * 2
    ps = [_sbm_params(case)] if g == "sbm" else _batch_params(case)
    return len(ps), sum(p[0] for p in ps), 2 * sum(_sbm_edges(*p) for p in ps)


def _rows(off):
    return torch.repeat_interleave(torch.arange(len(off) - 1, device=off.device), off.diff())


def _weights(off, adj, seed):
    """One weight per edge, U[0.05, 3), the same on both arcs."""
    n = len(off) - 1
    src, dst = _rows(off), adj.long()
    w = torch.rand(len(adj), generator=_gen(seed + 1), device=DEVICE, dtype=torch.float64) * 2.95 + 0.05
    twin = torch.searchsorted(src * n + dst, dst * n + src)
    return torch.where(src < dst, w, w[twin])


# ---------------------------------------------------------------- the workloads
def _kind(case):
    return gs.COSINE if case["kind"] == "cosine" else gs.JACCARD


def _queries(case, seed):
    r = np.random.RandomState(seed % (1 << 31))
    c = case["count"]
    return r.randint(2, 33, c).astype(np.int32), r.randint(2, 19, c) / 20.0


def prepare(case, seed):
    st = {"case": case}
    g = _graph(case, seed)
    if case["host"]:
        g = (g[0].to(torch.int32).cpu().numpy(), g[1].cpu().numpy())
    op = case["op"]
    if op == "weighted":
        st["weights"] = _weights(*g, seed)
    if op == "lsh":
        st["lsh"] = gs.make_lsh(_kind(case), case["k"], case["threshold"])
    if op in ("build", "batch", "weighted", "lsh"):
        st["graph"] = g
        # the caller's buffers for the index arrays; co_off takes up to n + 1
        # entries (maximum degree + 1) a graph
        graphs, n, arcs = _size(case)
        st["out"] = {"no_id": torch.empty(arcs, dtype=torch.int32, device=DEVICE),
                     "no_sim": torch.empty(arcs, dtype=torch.float64, device=DEVICE),
                     "co_off": torch.zeros(n + graphs, dtype=torch.int64, device=DEVICE),
                     "co_id": torch.empty(arcs, dtype=torch.int32, device=DEVICE),
                     "co_thr": torch.empty(arcs, dtype=torch.float64, device=DEVICE)}
        return st
    # queries: a resident index, and device rows for the labels
    st["index"] = gs.ScanIndex.build(g, _kind(case))
    n = st["index"].n
    if op == "query":
        st["labels"] = torch.empty(n, dtype=torch.int32, device=DEVICE)
    elif op == "queries":
        st["mus"], st["epss"] = _queries(case, seed)
        st["labels"] = torch.empty(case["count"], n, dtype=torch.int32, device=DEVICE)
    else:
        mus, epss = gs.paper_sigma()
        at = np.linspace(0, len(mus) - 1, case["pairs"]).astype(int)
        st["mus"], st["epss"] = mus[at], epss[at]
    return st


def _export(ixs, out):
    """The arrays of one or more indexes, end to end in the caller's tensors."""
    p = {k: t.data_ptr() for k, t in out.items()}
    export = gs.load().scan_index_export
    a = c = 0
    for ix in ixs:
        rc = export(ix._h, None, p["no_id"] + 4 * a, p["no_sim"] + 8 * a, p["co_off"] + 8 * c,
                    p["co_id"] + 4 * a, p["co_thr"] + 8 * a)
        if rc != 0:
            raise gs.ScanError(rc, "scan_index_export")
        a += ix.arcs
        c += ix.n + 1
    return out


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "query":
        return state["index"].query(case["mu"], case["eps"], hubs=case["hubs"], out=state["labels"])
    if op == "queries":
        return state["index"].query_batch(state["mus"], state["epss"], hubs=case["hubs"],
                                          out=state["labels"])
    if op == "sweep":
        return state["index"].sweep(state["mus"], state["epss"])
    if op == "batch":
        ixs = gs.ScanIndex.build_batch(state["graph"], _kind(case))
        out = _export(ixs, state["out"])
        for ix in ixs:
            ix.free()
        return out
    with gs.ScanIndex.build(state["graph"], _kind(case), lsh=state.get("lsh"),
                            weights=state.get("weights")) as ix:
        return _export([ix], state["out"])


def work(case):
    _, n, arcs = _size(case)
    op = case["op"]
    if op == "query":
        return {"bytes": 4 * n, "flops": 0}  # the labels
    if op == "queries":
        return {"bytes": 4 * n * case["count"], "flops": 0}
    if op == "sweep":
        # the labels of a pair are used, not kept: the index once
        return {"bytes": 28 * arcs + 12 * n + 8 * case["pairs"], "flops": 0}
    # CSR in; neighbour order and core order out (ids and values)
    byte = 8 * n + 4 * arcs + 24 * arcs + (8 * arcs if op == "weighted" else 0)
    # a dense graph's counts are half of a symmetric matrix product
    return {"bytes": byte, "flops": float(n) ** 3 if case["graph"] == "er" else 0}


# ---------------------------------------------------------------- 64-bit values
def _counts(off, adj, w=None):
    """Per arc: common neighbours, or with weights the sum over them of
    w(u,x) w(v,x); by wedges of the degree-oriented graph."""
    n = len(off) - 1
    src, dst = _rows(off), adj.long()
    deg = off.diff()
    rank = torch.empty(n, dtype=torch.int64, device=DEVICE)
    rank[torch.argsort(deg, stable=True)] = torch.arange(n, device=DEVICE)
    rs, rd = rank[src], rank[dst]
    up = (rs < rd).nonzero()[:, 0]
    key, order = torch.sort(rs[up] * n + rd[up])
    arc = up[order]  # out-arcs by (rank of tail, rank of head)
    a, b = key // n, key % n
    start = torch.searchsorted(a, torch.arange(n + 1, device=DEVICE))
    after = start[a + 1] - torch.arange(len(key), device=DEVICE) - 1  # heads after this one
    acc = torch.zeros(len(key), dtype=torch.float64, device=DEVICE)
    wk = w[arc] if w is not None else None
    pre = torch.cumsum(after, 0)
    i = 0
    while i < len(key):
        base = int(pre[i - 1]) if i else 0
        j = max(i + 1, int(torch.searchsorted(pre, torch.tensor(base + (1 << 26), device=DEVICE))))
        j = min(j, len(key))
        e = torch.repeat_interleave(torch.arange(i, j, device=DEVICE), after[i:j])
        f = torch.arange(len(e), device=DEVICE) - (pre[e] - after[e] - base) + e + 1
        want = b[e] * n + b[f]
        at = torch.searchsorted(key, want).clamp_(max=len(key) - 1)
        hit = key[at] == want
        e, f, at = e[hit], f[hit], at[hit]
        for x, y, z in ((e, f, at), (f, e, at), (at, e, f)):
            one = torch.ones(len(x), dtype=torch.float64, device=DEVICE)
            acc.index_add_(0, x, one if w is None else wk[y] * wk[z])
        i = j
    out = torch.zeros(len(adj), dtype=torch.float64, device=DEVICE)
    out[arc] = acc
    twin = torch.searchsorted(src * n + dst, dst * n + src)
    return torch.where(rs < rd, out, out[twin])


def _counts_dense(off, adj):
    """Common neighbours by a matrix product: whole numbers below 2^24."""
    n = len(off) - 1
    src, dst = _rows(off), adj.long()
    a = torch.zeros(n, n, dtype=torch.float32, device=DEVICE)
    a[src, dst] = 1
    c = a @ a
    return c[src, dst].double()


def _orders(off, adj, sim):
    """no_sim and co_thr from the similarity of every arc."""
    src = _rows(off)
    val, at = torch.sort(sim, descending=True, stable=True)
    row, by = torch.sort(src[at], stable=True)
    no = val[by]
    r = torch.arange(len(no), device=DEVICE) - off[row]
    val, at = torch.sort(no, descending=True, stable=True)
    return no, val[torch.sort(r[at], stable=True)[1]]


def exact(case, seed):
    if case["op"] == "lsh" or case["op"] in ("query", "queries", "sweep"):
        return None  # estimates by hashing, or labels
    _, _, arcs = _size(case)
    if case["graph"] == "rmat" and arcs > 4.2e7:
        return None  # too long
    g = _graph(case, seed)
    no, co = [], []
    for off, adj in (g if case["op"] == "batch" else [g]):
        if len(adj) == 0:
            continue
        src, dst = _rows(off), adj.long()
        d = off.diff().double()
        if case["op"] == "weighted":
            w = _weights(off, adj, seed)
            t = _counts(off, adj, w)
            sq = torch.ones(len(d), dtype=torch.float64, device=DEVICE).index_add_(0, src, w * w)
            sim = (2 * w + t) / (sq[src].sqrt() * sq[dst].sqrt())
        else:
            small = case["graph"] != "rmat" and len(off) <= 30000
            t = _counts_dense(off, adj) if small else _counts(off, adj)
            if case["kind"] == "cosine":
                sim = (t + 2) / ((d[src] + 1) * (d[dst] + 1)).sqrt()
            else:
                sim = (t + 2) / (d[src] + d[dst] - t)
        x, y = _orders(off, adj, sim)
        no.append(x)
        co.append(y)
    return {"no_id": None, "no_sim": torch.cat(no), "co_off": None, "co_id": None,
            "co_thr": torch.cat(co)}
