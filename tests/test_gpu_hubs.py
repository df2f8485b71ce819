"""Counting with a hub (one of the at most 65535 vertices of highest degree)
in the middle: graphs whose hubs end inside and at the ends of the degree
order, a degree class too large to be taken, equal degrees (numbered by id),
out-lists that start at even and odd positions, suffixes around the lane and
round lengths, weights, LSH and 64-bit indices. Against the oracle."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2012_11188_gb300 as gs

pytestmark = pytest.mark.gpu

KEYS = ("sim", "no_id", "no_sim", "co_off", "co_id", "co_thr")


def circulant(n, half, first=0):
    """n vertices, each joined to the `half` next ones around a ring."""
    v = np.repeat(np.arange(n), half)
    return np.stack([first + v, first + (v + np.tile(np.arange(1, half + 1), n)) % n], 1)


def lattice(n, half, hubs, seed):
    """A ring lattice plus hubs joined to one another and to random vertices."""
    rng = np.random.default_rng(seed)
    e = [circulant(n, half)]
    for i, d in enumerate(hubs):
        e.append(np.stack([np.full(d, n + i), rng.choice(n, d, replace=False)], 1))
        e.append(np.array([(n + i, n + j) for j in range(i)], dtype=np.int64).reshape(-1, 2))
    return graphgen.from_edges(n + len(hubs), np.concatenate(e))


GRAPHS = {
    # every vertex a hub
    "rmat": lambda: graphgen.rmat(12, 48, seed=2),
    # 66000 vertices of about one degree, more than may be hubs: some classes
    "classes": lambda: lattice(66000, 32, [700, 701, 701, 1500, 3000], 3),
    # one class of 66000 equal degrees is left out, a few vertices are hubs
    "one_class": lambda: graphgen.from_edges(
        67600, np.concatenate([circulant(66000, 40),
                               circulant(1600, 380, 66000)])),
    # complete bipartite-like core: long out-lists of every parity
    "core": lambda: lattice(3000, 150, [513, 600, 777, 1024, 2047, 2999], 5),
}


@pytest.fixture(scope="module", params=list(GRAPHS))
def graph(request):
    return GRAPHS[request.param]()


def equal(ix, ox, keys=KEYS):
    ex = ix.export()
    for k in keys:
        assert np.array_equal(ex[k], getattr(ox, k)), k


def test_exact_and_wide(graph):
    ox = oracle.Index(graph)
    with gs.ScanIndex.build(graph, counts=gs.COUNTS_SPARSE) as ix:
        equal(ix, ox)
    gs.set_wide_index(True)
    try:
        with gs.ScanIndex.build(graph, counts=gs.COUNTS_SPARSE) as ix:
            equal(ix, ox)
    finally:
        gs.set_wide_index(False)


@pytest.mark.parametrize("cfg", [{"long_list": 1}, {"long_list": 1 << 20, "rounds": 8},
                                 {"cta_chunk": 256, "warp_deg": 64}])
def test_strategies(graph, cfg):
    ox = oracle.Index(graph, oracle.JACCARD)
    gs.set_count_config(cfg)
    try:
        with gs.ScanIndex.build(graph, gs.JACCARD, counts=gs.COUNTS_SPARSE) as ix:
            equal(ix, ox)
    finally:
        gs.set_count_config(None)


def test_integer_weights(graph):
    w = graphgen.edge_weights(graph, 3, "int")  # every sum is exact
    ox = oracle.Index(graph, oracle.COSINE, sim=oracle.weighted_similarities(graph, w))
    with gs.ScanIndex.build(graph, weights=w) as ix:
        equal(ix, ox)


def test_lsh(graph):
    ox = oracle.LSHIndex(graph, oracle.COSINE, 64, T=600, seed=2)
    with gs.ScanIndex.build(graph, lsh=gs.make_lsh(gs.COSINE, 64, 600, seed=2)) as ix:
        equal(ix, ox)


def test_range_counts(graph):
    ox = oracle.Index(graph)
    src = np.repeat(np.arange(graph.n), np.diff(graph.off))
    d = np.diff(graph.off)
    cut = [0, graph.n // 3, graph.n - 2, graph.n]
    t = sum(gs.closed_counts_range(graph, a, b).astype(np.int64) for a, b in zip(cut, cut[1:]))
    want = (t + 2) / np.sqrt(((d[src] + 1) * (d[graph.adj] + 1)).astype(np.float64))
    assert np.array_equal(want, ox.sim)
