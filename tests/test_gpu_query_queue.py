"""Batches that ask for more row pieces than the queue holds (131,072 pieces
past the first 1024 entries of a core's prefix): every warp then walks its
whole prefixes. Against queries that have no queue (scan_query_noalloc) and
against single queries, whose own queue is not full."""
import numpy as np
import pytest

import paper_2012_11188_gb300 as gs

pytestmark = pytest.mark.gpu

CAP = 1 << 17
PIECE = 1024


def groups(sizes, links):
    """Complete graphs of the given sizes, a path of `links` extra vertices
    hanging off each, and every complete graph joined to the next by one edge."""
    rows, base, heads = [], 0, []
    extra = []
    for s in sizes:
        ids = np.arange(base, base + s)
        rows += [np.delete(ids, i) for i in range(s)]
        rows += [np.zeros(0, np.int64)] * links
        heads.append(base)
        for k in range(links):
            extra.append((base + (s - 1 if k == 0 else s + k - 1), base + s + k))
        base += s + links
    extra += list(zip(heads[:-1], heads[1:]))
    more = [[] for _ in range(base)]
    for a, b in extra:
        more[a].append(b)
        more[b].append(a)
    rows = [np.sort(np.concatenate([r, np.array(m, np.int64)])) for r, m in zip(rows, more)]
    off = np.zeros(base + 1, np.int64)
    off[1:] = np.cumsum([len(r) for r in rows])
    return off, np.concatenate(rows).astype(np.int32)


@pytest.mark.parametrize("count", [16, 40])
def test_batch_that_fills_the_queue(count):
    import ctypes

    import torch
    sizes, links = [3100, 2049, 1500, 4200], 3
    g = groups(sizes, links)
    n = len(g[0]) - 1
    # similarities within a group are 1 or next to it, at its ends lower
    mus = [2 + (i * 389) % 4400 for i in range(count)]
    epss = [[0.0, 0.3, 0.9, 0.97][i % 4] for i in range(count)]
    asked = sum((s - 2) // PIECE * s for s in sizes) * count  # where every group is cores
    assert asked > CAP  # (some of the queries with a large mu ask for less)
    lib = gs.load()
    with gs.ScanIndex.build(g) as ix:
        out = torch.full((count, n), 77, dtype=torch.int32, device="cuda")
        ix.query_batch(mus, epss, hubs=True, out=out)
        got = out.cpu().numpy()
        pieces = 0
        one = torch.empty(n, dtype=torch.int32, device="cuda")
        for i in range(count):
            assert np.array_equal(got[i], ix.query(mus[i], epss[i], hubs=True)), i
            rc = lib.scan_query_noalloc(ix._h, mus[i], ctypes.c_double(epss[i]),
                                        ctypes.c_void_p(one.data_ptr()), 1, ctypes.c_size_t(0))
            torch.cuda.synchronize()
            assert rc == 0 and np.array_equal(got[i], one.cpu().numpy()), i
            lab = got[i]
            for s, b in zip(sizes, np.cumsum([0] + [x + links for x in sizes[:-1]])):
                if mus[i] <= s and (lab[b:b + s] >= 0).all():
                    pieces += (s - 2) // PIECE * s
        assert pieces > CAP
