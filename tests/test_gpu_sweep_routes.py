"""Sweeps of eight pairs and more on either side of their routes: from 131,072
vertices on, labels turned where the cores reach many neighbours and single passes
where they reach few, rows at the lengths from which a CTA (2048) and all CTAs (65,536) take them. Every sum is a
whole number, so the modularity is the same double as that of each clustering
by itself (scan_modularity)."""
import numpy as np
import pytest

import graphgen
import paper_2012_11188_gb300 as gs

pytestmark = pytest.mark.gpu


def stars(sizes, extra):
    """Stars of the given numbers of leaves, each centre joined to the next, and
    `extra` vertices without edges."""
    edges, base, centres = [], 0, []
    for s in sizes:
        edges += [(base, base + 1 + i) for i in range(s)]
        centres.append(base)
        base += s + 1
    edges += list(zip(centres[:-1], centres[1:]))
    return graphgen.from_edges(base + extra, edges)


GRAPHS = {
    "around a CTA's row": lambda: stars([2046, 2047, 2048, 2049, 700], 140000),
    "around all CTAs' row": lambda: stars([65535, 65536, 30], 100000),
    "short rows only": lambda: stars([500, 40, 1], 131072 - 544),
    "one vertex less": lambda: stars([500, 40, 1], 131072 - 545),
    "rmat": lambda: graphgen.rmat(17, 16, seed=6),
    "sbm": lambda: graphgen.sbm(150000, 1500, 0.2, 0.00001, seed=7),
    "small": lambda: graphgen.rmat(11, 16, seed=6),
}
# (mu, eps) without cores, with a few, with most vertices
NONE = [(100000, 0.1), (3, 1.0), (60000, 0.5)]
FEW = [(700, 0.0), (1000, 0.0), (2000, 0.02), (500, 0.02), (40, 0.15)]
MOST = [(2, 0.0), (2, 0.01), (3, 0.05)]


@pytest.mark.parametrize("name", GRAPHS)
@pytest.mark.parametrize("pairs", [NONE * 3, FEW * 2, NONE * 6 + FEW * 4, MOST * 3 + NONE * 9,
                                   FEW * 9 + MOST])
def test_sweep_equals_single_clusterings(name, pairs):
    g = GRAPHS[name]()
    with gs.ScanIndex.build(g) as ix:
        got = ix.sweep([m for m, _ in pairs], [e for _, e in pairs])
        want = {p: ix.modularity(ix.query(*p)) for p in set(pairs)}
    assert np.array_equal(got, [want[p] for p in pairs])
