"""The passes that walk 32 rows per warp (CSR checks, orientation, out-arc
walks): empty rows at every place of a group, rows that start and end on chunk
boundaries, rows of several chunks, rows beyond 4096 left to their own kernel
in the middle of a group, vertex counts that are no multiple of 32, and bad
rows of every kind at each place. Against the oracle."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2012_11188_gb300 as gs

pytestmark = pytest.mark.gpu


def pattern(degrees, seed):
    """A graph whose first vertices have about the listed degrees, their
    neighbours drawn from a tail of further vertices."""
    rng = np.random.default_rng(seed)
    n0, tail = len(degrees), max(degrees) + 37
    e = [np.stack([np.full(d, i), n0 + rng.choice(tail, d, replace=False)], 1)
         for i, d in enumerate(degrees) if d]
    return graphgen.from_edges(n0 + tail, np.concatenate(e))


PATTERNS = {
    "chunks": [32, 0, 32, 31, 1, 0, 0, 64, 33, 31, 96, 0, 1, 1, 1, 29, 32] * 4 + [5],
    "empties": [0] * 31 + [40] + [3] + [0] * 31 + [0] * 64 + [7, 0, 0, 100, 0],
    "long": [10, 4096, 0, 4097, 33, 5000, 1, 0, 4095, 9000, 2] * 5,
    "one": [1],
}


@pytest.mark.parametrize("name", list(PATTERNS))
def test_patterns(name):
    g = pattern(PATTERNS[name], 4)
    ox = oracle.Index(g)
    with gs.ScanIndex.build(g, counts=gs.COUNTS_SPARSE) as ix:
        ex = ix.export()
    for k in ("sim", "no_id", "no_sim", "co_off", "co_id", "co_thr"):
        assert np.array_equal(ex[k], getattr(ox, k)), k


@pytest.mark.parametrize("what", ["order", "duplicate", "loop", "range", "negative", "missing"])
@pytest.mark.parametrize("where", [0, 1, 6, 17, 40, 63])
def test_bad_rows(what, where):
    g = pattern(PATTERNS["chunks"], 9)
    off, adj = g.off.copy(), g.adj.copy()
    v = next(x for x in range(where, g.n) if off[x + 1] - off[x] >= 29)
    b, e = off[v], off[v + 1]
    i = b + (where % (e - b - 1))
    if what == "order":
        adj[i], adj[i + 1] = adj[i + 1], adj[i]
    elif what == "duplicate":
        adj[i + 1] = adj[i]
    elif what == "loop":
        adj[b] = v
    elif what == "range":
        adj[e - 1] = g.n
    elif what == "negative":
        adj[b] = -1
    else:  # an arc without its reverse
        adj[e - 1] = v + 1 if adj[e - 1] != v + 1 else v + 2
        adj[b:e] = np.sort(adj[b:e])
    with pytest.raises(gs.ScanError) as err:
        gs.ScanIndex.build(graphgen.CSR(off, adj), counts=gs.COUNTS_SPARSE)
    assert err.value.status == -3
