"""Borders by where their first core stands in their own prefix, and by how many
borders of 32 neighbours are still looking: a lane looks alone at 8 entries, or
at up to 64 while more than 4 lanes look, the warp goes through the rest.
Against the oracle."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2012_11188_gb300 as gs

pytestmark = pytest.mark.gpu


def first_core_at(ix, mu, eps, labels):
    """Position in its own neighbour order of every border's first core."""
    ex = ix.export()
    cores = ex["co_id"][ex["co_off"][mu - 2]:ex["co_off"][mu - 1]]
    thr = ex["co_thr"][ex["co_off"][mu - 2]:ex["co_off"][mu - 1]]
    core = np.zeros(ix.n, bool)
    core[cores[thr >= eps]] = True
    return core, ex


GRAPHS = {
    "rmat": (lambda: graphgen.rmat(11, 24, seed=2), [(100, 0.02), (300, 0.0), (600, 0.02)]),
    "dense": (lambda: graphgen.sbm(900, 3, 0.5, 0.05, seed=3),
              [(194, 0.0), (202, 0.05), (206, 0.0), (212, 0.05)]),
    "blocks": (lambda: graphgen.sbm(3000, 30, 0.3, 0.01, seed=4), [(69, 0.0), (74, 0.0), (82, 0.0)]),
}


@pytest.mark.parametrize("name", GRAPHS)
def test_borders(name):
    make, pairs = GRAPHS[name]
    g = make()
    ox = oracle.Index(g)
    seen = set()
    with gs.ScanIndex.build(g) as ix:
        rows = ix.query_batch([m for m, _ in pairs] * 2, [e for _, e in pairs] * 2, hubs=True)
        for i, (mu, eps) in enumerate(pairs):
            want = ox.query(mu, eps, hubs=True)
            assert np.array_equal(rows[i], want) and np.array_equal(rows[len(pairs) + i], want)
            assert np.array_equal(ix.query(mu, eps, hubs=True), want), (mu, eps)
            core, ex = first_core_at(ix, mu, eps, want)
            for v in np.flatnonzero(~core & (want >= 0)):
                at = np.flatnonzero(core[ex["no_id"][g.off[v]:g.off[v + 1]]])[0]
                seen.add("8" if at < 8 else "64" if at < 64 else "more")
    assert seen == {"8", "64", "more"}
