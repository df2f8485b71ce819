"""Packing and export of a batch: graphs of host and device arrays, int32 and
int64 offsets, views at odd element offsets, graphs without vertices or arcs
between others, sizes around the 4096-element chunks; every index equals the
one built alone, copied to host or device, whole or in part. Bad members are
refused."""
import numpy as np
import pytest

import graphgen
import paper_2012_11188_gb300 as gs

pytestmark = pytest.mark.gpu

KEYS = ("no_id", "no_sim", "co_off", "co_id", "co_thr")


def graphs():
    e = np.zeros(0, np.int64)
    return [graphgen.rmat(6, 6, seed=1), graphgen.CSR(np.zeros(1, np.int64), e.astype(np.int32)),
            graphgen.CSR(np.zeros(6, np.int64), e.astype(np.int32)),
            graphgen.sbm(4096, 16, 0.05, 0.001, seed=2), graphgen.from_edges(2, [(0, 1)]),
            graphgen.rmat(9, 12, seed=3), graphgen.from_edges(4095, [(0, 4094)]),
            graphgen.sbm(300, 3, 0.3, 0.01, seed=4)]


def member(g, how, shift):
    import torch
    off = g.off.astype(np.int32) if "32" in how else g.off
    if "host" in how:
        return off, g.adj
    pad = torch.zeros(shift, dtype=torch.int32)
    adj = torch.cat([pad, torch.from_numpy(g.adj)]).cuda()[shift:]
    o = torch.from_numpy(off)
    return torch.cat([torch.zeros(shift, dtype=o.dtype), o]).cuda()[shift:], adj


@pytest.mark.parametrize("how", ["host", "host32", "device", "device32", "mixed"])
def test_batch_equals_singles(how):
    import torch
    gl = graphs()
    ways = ["host", "device32", "device", "host32"] if how == "mixed" else [how]
    batch = [member(g, ways[i % len(ways)], i % 3) for i, g in enumerate(gl)]
    for g, ix in zip(gl, gs.ScanIndex.build_batch(batch)):
        with gs.ScanIndex.build(g, counts=gs.COUNTS_SPARSE) as one:
            want, got = one.export(), ix.export()
            for k in want:
                assert np.array_equal(want[k], got[k]), k
            # into device tensors, all five arrays and two of them
            t = {k: torch.full((want[k].size,), 7, dtype=torch.from_numpy(want[k]).dtype,
                               device="cuda") for k in KEYS}
            for skip in ((), ("no_sim", "co_off", "co_id")):
                p = [0 if k in skip or t[k].numel() == 0 else t[k].data_ptr() for k in KEYS]
                assert gs.load().scan_index_export(ix._h, None, *p) == 0
                for k in KEYS:
                    if k not in skip:
                        assert np.array_equal(t[k].cpu().numpy(), want[k]), k
                    t[k].fill_(7)
        ix.free()


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("what", ["first", "last", "inner", "id", "negative"])
def test_bad_member(what, device):
    import torch
    gl = graphs()
    off, adj = gl[5].off.copy(), gl[5].adj.copy()
    if what == "first":
        off[0] = 1
    elif what == "last":
        off[-1] -= 1
    elif what == "inner":
        off[7] = len(adj) + 5
    elif what == "id":
        adj[3] = gl[5].n
    else:
        adj[3] = -2
    batch = [(g.off, g.adj) for g in gl]
    batch[5] = (off, adj)
    if device:
        batch = [(torch.from_numpy(o).cuda(), torch.from_numpy(a).cuda()) for o, a in batch]
    with pytest.raises(gs.ScanError) as err:
        gs.ScanIndex.build_batch(batch)
    assert err.value.status == -3
