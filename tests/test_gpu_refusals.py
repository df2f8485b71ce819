"""Builds refused for what the counting finds (a CSR that is not symmetric, a
weight that is negative, not finite or unequal on its two arcs): the status, and
that neither the neighbour order nor the core order is built first."""
import numpy as np
import pytest

import graphgen
import paper_2012_11188_gb300 as gs

pytestmark = pytest.mark.gpu

EINVAL, EBADGRAPH = -1, -3
# the core order of a graph with arcs: a histogram, segment sizes, tiles, their
# places and five prefix sums, the transpose (each at least one launch)
CORE_ORDER = 10


def launches(call):
    before = gs.kernel_launches()
    call()
    return gs.kernel_launches() - before


def refused(status, call):
    with pytest.raises(gs.ScanError) as e:
        call()
    assert e.value.status == status


@pytest.mark.parametrize("lsh", [None, 30])
@pytest.mark.parametrize("fault", ["negative", "nan", "inf", "unequal"])
def test_bad_weights(fault, lsh):
    g = graphgen.rmat(12, 16, seed=1)
    w = graphgen.edge_weights(g, 1)
    lsh = gs.make_lsh(gs.COSINE, 64, lsh) if lsh else None
    good = launches(lambda: gs.ScanIndex.build(g, weights=w, lsh=lsh).free())
    at = int(g.off[int(np.argmax(np.diff(g.off)))])  # an arc of the largest row
    w = w.copy()
    w[at] = {"negative": -1.0, "nan": np.nan, "inf": np.inf, "unequal": w[at] + 1}[fault]
    if fault == "nan":  # on both arcs of the edge: no inequality to find
        row = int(np.searchsorted(g.off, at, side="right") - 1)
        x = int(g.adj[at])
        w[int(g.off[x]) + int(np.searchsorted(g.adj[g.off[x]:g.off[x + 1]], row))] = np.nan
    bad = launches(lambda: refused(EINVAL, lambda: gs.ScanIndex.build(g, weights=w, lsh=lsh)))
    assert bad <= good - CORE_ORDER


def circulant(n, steps):
    rows = np.sort((np.arange(n)[:, None] + np.array(steps)[None, :]) % n, axis=1)
    return np.arange(n + 1, dtype=np.int64) * len(steps), rows.astype(np.int32).reshape(-1)


@pytest.mark.parametrize("kind", [gs.COSINE, gs.JACCARD])
@pytest.mark.parametrize("counts", [gs.COUNTS_SPARSE, gs.COUNTS_DENSE])
def test_not_symmetric(kind, counts):
    """Every vertex v lists v + s for steps s of one sign each, of which as many
    arcs ascend as descend (what a symmetric graph has, and what is checked
    before the counting)."""
    n = 4096
    # the arcs of step s > 0 ascend from n - s vertices, of s < 0 from |s|:
    # n - s1 + n - s2 + s3 + s4 = 2 n with s3 + s4 = s1 + s2
    odd = circulant(n, [3, 50, -20, -33])
    even = circulant(n, [3, 50, -3, -50])
    up = (odd[1] > np.repeat(np.arange(n), 4)).sum()
    assert up == len(odd[1]) // 2
    good = launches(lambda: gs.ScanIndex.build(even, kind, counts=counts).free())
    bad = launches(lambda: refused(EBADGRAPH, lambda: gs.ScanIndex.build(odd, kind, counts=counts)))
    assert bad <= good - CORE_ORDER
    refused(EBADGRAPH, lambda: gs.ScanIndex.build_batch([even, odd, even], kind))
