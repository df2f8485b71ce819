"""Queries where their phases change: eps-prefixes around one queued piece
(1024 entries) and of several pieces, borders whose first core lies within
the entries a lane looks at alone (8), within the warp's steps (128) or far
behind them, core searches of every length class, batches of more queries
than one scan step, and single queries from several threads and streams at
once. Against the oracle, bit for bit."""
import threading

import numpy as np
import pytest

import graphgen
import oracle
import paper_2012_11188_gb300 as gs

pytestmark = pytest.mark.gpu

DEGREES = [7, 8, 9, 31, 33, 127, 136, 137, 264, 1023, 1024, 1025, 1056, 2048, 2049, 3500]


@pytest.fixture(scope="module")
def graph():
    """Hubs of the listed degrees over shared leaves, a clique of the hubs:
    with a large mu few hubs are cores and the others are borders whose own
    prefixes are long; plus a denser random part."""
    h, leaves = len(DEGREES), max(DEGREES)
    edges = [(i, j) for i in range(h) for j in range(i)]
    edges += [(i, h + x) for i, d in enumerate(DEGREES) for x in range(d)]
    r = graphgen.rmat(11, 12, seed=3)
    src = np.repeat(np.arange(r.n), np.diff(r.off))
    edges += [(h + leaves + int(a), h + leaves + int(b)) for a, b in zip(src, r.adj)]
    edges += [(h + 5, h + leaves + 1)]
    g = graphgen.from_edges(h + leaves + r.n, edges)
    return g, oracle.Index(g)


MUS = [2, 3, 10, 30, 100, 200, 1030, 1200, 2100, 3000, 3516, 3517, 5000]
EPSS = [0.0, 0.01, 0.03, 0.1, 0.35, 1.0]


@pytest.mark.parametrize("hubs", [False, True])
def test_single_and_batched_queries(graph, hubs):
    g, ox = graph
    pairs = [(m, e) for m in MUS for e in EPSS]
    with gs.ScanIndex.build(g) as ix:
        want = [ox.query(m, e, hubs=hubs) for m, e in pairs]
        for (m, e), w in zip(pairs, want):
            assert np.array_equal(ix.query(m, e, hubs=hubs), w), (m, e)
        # a batch of more than 256 queries, in another order
        k = [(7 * i) % len(pairs) for i in range(300)]
        got = ix.query_batch([pairs[i][0] for i in k], [pairs[i][1] for i in k], hubs=hubs)
        for i, row in zip(k, got):
            assert np.array_equal(row, want[i]), pairs[i]


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_unaligned_device_labels(graph, shift):
    import torch
    g, ox = graph
    with gs.ScanIndex.build(g) as ix:
        buf = torch.full((g.n + 8,), 77, dtype=torch.int32, device="cuda")
        ix.query(30, 0.03, hubs=True, out=buf[shift:shift + g.n])
        got = buf.cpu().numpy()
    assert np.array_equal(got[shift:shift + g.n], ox.query(30, 0.03, hubs=True))
    assert (got[:shift] == 77).all() and (got[shift + g.n:] == 77).all()


@pytest.mark.parametrize("count", [1, 7, 8, 31, 32, 33, 70])
def test_sweep_lengths(graph, count):
    """One clustering at a time, a full batch, a batch and a remainder; rows
    longer than one arc piece of the modularity pass (512)."""
    g, ox = graph
    pairs = [(m, e) for m in MUS for e in EPSS]
    pairs = [pairs[(11 * i) % len(pairs)] for i in range(count)]
    with gs.ScanIndex.build(g) as ix:
        got = ix.sweep([m for m, _ in pairs], [e for _, e in pairs])
    want = [oracle.modularity(g, ox.query(m, e)) for m, e in pairs]
    # whole numbers below 2^53 on both sides up to the last two divisions
    assert np.abs(got - np.array(want)).max() <= 1e-12


def test_threads_and_streams(graph):
    import torch
    g, ox = graph
    pairs = [(3, 0.1), (30, 0.03), (1200, 0.0), (10, 0.35)]
    want = [ox.query(m, e, hubs=True) for m, e in pairs]
    bad = []
    with gs.ScanIndex.build(g) as ix:
        def work(t):
            st = torch.cuda.Stream()
            out = torch.empty(g.n, dtype=torch.int32, device="cuda")
            for i in range(40):
                j = (i + t) % len(pairs)
                ix.query(*pairs[j], hubs=True, out=out, stream=st)
                with torch.cuda.stream(st):
                    if not np.array_equal(out.cpu().numpy(), want[j]):
                        bad.append((t, i))
        ts = [threading.Thread(target=work, args=(t,)) for t in range(4)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
    assert not bad
