"""Offsets that descend: many rows look longer than 4096 entries although the
arcs have room for few of them. The degree pass lists long rows in arcs / 4096
+ 1 places; such offsets are refused by every entry point that takes a CSR,
whatever their number, and the builds after them are not affected."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2012_11188_gb300 as gs

pytestmark = pytest.mark.gpu

EBADGRAPH = -3


def zigzag(n, arcs, low=0):
    """n rows (even): arcs, -arcs, arcs, ... entries; first offset 0, last arcs."""
    off = np.full(n + 1, arcs, np.int64)
    off[::2] = low
    off[0], off[-1] = 0, arcs
    return off, (np.arange(arcs) % n).astype(np.int32)


def refused(call):
    with pytest.raises(gs.ScanError) as e:
        call()
    assert e.value.status == EBADGRAPH


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("n,arcs,low", [(64, 4098, 0), (5000, 8192, 0), (300001, 12290, 4),
                                        (1000000, 1 << 20, 17)])
def test_descending_offsets_are_refused(n, arcs, low, device):
    off, adj = zigzag(n, arcs, low)
    g = (off, adj)
    if device:
        import torch
        g = (torch.from_numpy(off).cuda(), torch.from_numpy(adj).cuda())
    refused(lambda: gs.ScanIndex.build(g))
    refused(lambda: gs.ScanIndex.build(g, weights=np.ones(arcs)))
    refused(lambda: gs.closed_counts_range(g, 0, n))
    if n <= 65536:
        refused(lambda: gs.ScanIndex.build(g, counts=gs.COUNTS_DENSE))
    good = graphgen.rmat(9, 8, seed=1)
    pair = (good.off, good.adj)
    if device:
        pair = (torch.from_numpy(good.off).cuda(), torch.from_numpy(good.adj).cuda())
    refused(lambda: gs.ScanIndex.build_batch([pair, g, pair]))
    ox = oracle.Index(good)
    with gs.ScanIndex.build(pair) as ix:
        ex = ix.export()
    for key in ("no_id", "no_sim", "co_off", "co_id", "co_thr"):
        assert np.array_equal(ex[key], getattr(ox, key)), key


def test_as_many_long_rows_as_fit():
    """Rows of 4097 entries each, as many as the list has places, and a star:
    accepted."""
    n = 4098  # a complete graph: every row has 4097 entries, (n - 1) / 4096 of the list taken
    full = np.arange(n, dtype=np.int32)
    adj = np.concatenate([np.delete(full, v) for v in range(n)])
    off = np.arange(n + 1, dtype=np.int64) * (n - 1)
    with gs.ScanIndex.build((off, adj), counts=gs.COUNTS_SPARSE) as ix:
        ex = ix.export()
    assert (ex["no_sim"] == 1.0).all()
    assert np.array_equal(ex["no_id"], adj)
    leaves = 200000
    star = graphgen.from_edges(leaves + 1, [(0, i) for i in range(1, leaves + 1)])
    with gs.ScanIndex.build(star) as ix:
        assert ix.maxdeg == leaves
