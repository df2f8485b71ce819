"""LSH index mode at the sizes where its kernels change: closed neighbourhoods
around one warp pass of the SimHash counters (960 elements) and around the
arc pieces of the estimate pass (1024), rows of many pieces, and sketch
lengths of every way of reading them (one to 32 lanes a sketch, several reads
per lane, lengths that are no multiple of 16 bytes). Bit for bit against the
oracle."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2012_11188_gb300 as gs

pytestmark = pytest.mark.gpu

HUBS = [129, 958, 959, 960, 961, 1023, 1024, 1025, 1920, 2047, 2049, 5000, 7680, 9000]  # leaves per hub


def hub_graph():
    """Hubs of the listed leaf counts, joined to one another, over leaves that
    share neighbours."""
    h = len(HUBS)
    edges = [(i, j) for i in range(h) for j in range(i)]
    edges += [(i, h + x) for i, d in enumerate(HUBS) for x in range(d)]
    edges += [(h + x, h + x + 1) for x in range(max(HUBS) - 1)]
    return graphgen.from_edges(h + max(HUBS), edges)


def check(kind, okind, k, T, seed, **kw):
    g = hub_graph()
    ox = oracle.LSHIndex(g, okind, k, T=T, seed=seed, **kw)
    with gs.ScanIndex.build(g, kind, lsh=gs.make_lsh(kind, k, T, seed=seed, **kw)) as ix:
        ex = ix.export()
    for key in ("sim", "no_id", "no_sim", "co_off", "co_id", "co_thr"):
        assert np.array_equal(ex[key], getattr(ox, key)), key


@pytest.mark.parametrize("T", [0, 128])
@pytest.mark.parametrize("k", [64, 128, 192, 256, 320, 512, 1024, 4096])
def test_simhash_lengths(k, T):
    check(gs.COSINE, oracle.COSINE, k, T, 9)


@pytest.mark.parametrize("k", [1, 2, 4, 8, 16, 32, 64, 128, 256, 1024])
def test_minhash_kpartition_lengths(k):
    check(gs.JACCARD, oracle.JACCARD, k, 0, 4, kpartition=True)


@pytest.mark.parametrize("k", [3, 12, 20, 50, 100])
def test_minhash_standard_lengths(k):
    check(gs.JACCARD, oracle.JACCARD, k, 0, 4, kpartition=False)
