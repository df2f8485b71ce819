"""Calls at the limit of device memory: an allocator that refuses requests
beyond a number of bytes. What is only there for speed (slabs, hub numbers,
the queue of row pieces, the labels turned for the sweep) is left out where
there is no room for it, and the results are the same."""
import contextlib
import ctypes

import numpy as np
import pytest

import graphgen
import paper_2012_11188_gb300 as gs
from paper_2012_11188_gb300 import scan

pytestmark = pytest.mark.gpu

MB = 1 << 20


class Limited:
    """Allocator hooks over torch's allocator: bytes held, their peak, a limit."""

    def __init__(self):
        self.held = self.peak = 0
        self.limit = None
        self.sizes = {}

    def alloc(self, nbytes, stream, ctx):
        import torch
        if self.limit is not None and self.held + nbytes > self.limit:
            return None
        p = torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0))
        self.held += nbytes
        self.peak = max(self.peak, self.held)
        self.sizes[p] = nbytes
        return p

    def free(self, p, nbytes, stream, ctx):
        import torch
        assert self.sizes.pop(p) == nbytes
        self.held -= nbytes
        torch.cuda.caching_allocator_delete(p)

    @contextlib.contextmanager
    def at_most(self, more):
        """`more` bytes beyond what is held now."""
        self.limit, self.peak = self.held + more, self.held
        yield
        self.limit = None


@pytest.fixture()
def memory():
    m = Limited()
    hooks = scan.ALLOC_FN(m.alloc), scan.FREE_FN(m.free)
    cast = [ctypes.cast(h, ctypes.c_void_p) for h in hooks]
    assert gs.load().scan_set_allocator(cast[0], cast[1], None) == 0
    yield m
    assert gs.load().scan_set_allocator(None, None, None) == 0
    assert m.held == 0 and not m.sizes


def hub_rows():
    """Rows of several pieces (1024 entries) and many short ones."""
    edges = [(i, j) for i in range(6) for j in range(i)]
    edges += [(i, 6 + x) for i in range(6) for x in range(1500 + 700 * i)]
    edges += [(6 + x, 6 + x + 1) for x in range(0, 6000, 2)]
    return graphgen.from_edges(6 + 6001, edges)


@pytest.mark.parametrize("count", [1, 5])
def test_queries_without_room_for_the_queue(memory, count):
    import torch
    g = hub_rows()
    with gs.ScanIndex.build(g) as ix:
        mus, epss = [3, 2, 900, 4, 2500][:count], [0.0, 0.02, 0.01, 0.3, 0.0][:count]
        want = np.stack([ix.query(m, e, hubs=True) for m, e in zip(mus, epss)])
        out = torch.full((count, g.n), 77, dtype=torch.int32, device="cuda")
        # parents, parameters, core counts and a status word
        with memory.at_most(4 * count * g.n + 4 * count + 8 * count + 8 * (2 * count + 1) + 4):
            if count == 1:
                ix.query(mus[0], epss[0], hubs=True, out=out)
            else:
                ix.query_batch(mus, epss, hubs=True, out=out)
    assert np.array_equal(out.cpu().numpy(), want)


def test_server_without_room_for_the_queue(memory):
    import torch
    g = hub_rows()
    with gs.ScanIndex.build(g) as ix:
        want = ix.query(3, 0.0, hubs=True)
        out = torch.full((g.n,), 77, dtype=torch.int32, device="cuda")
        # parents of four queries, destinations, parameters, core counts, two
        # status words
        with memory.at_most(4 * 4 * g.n + 4 * 8 + 4 * 4 + 4 * 8 + 8 * 9 + 8):
            with gs.Server(max_batch=4) as srv:
                srv.wait(srv.submit_query(ix, 3, 0.0, out, hubs=True), timeout_ms=60000)
    assert np.array_equal(out.cpu().numpy(), want)


@pytest.mark.parametrize("count,room", [(40, "one"), (40, "labels"), (40, "queries"), (40, "all"),
                                        (8, "one"), (8, "queries")])
def test_sweep_without_room_for_all_clusterings(memory, count, room):
    """Room for the passes of one clustering at a time, for the turned labels
    but not the sums of all clusterings, for both but not the queries' own
    scratch, and for everything."""
    g = hub_rows()
    mus = [2 + 3 * (i % 13) for i in range(count)]
    epss = [(i % 9) / 20.0 for i in range(count)]
    batch = min(count, 32)
    need = 4 * batch * g.n  # label rows
    need += 4 * batch * g.n + 12 * batch + 8 * (2 * batch + 1)  # the queries
    need += 8 * g.n  # sums of one clustering
    need += 8 * (4 * count + 1) + 4
    turned, sums = 4 * 32 * g.n, 8 * batch * g.n
    more = {"one": 0, "labels": turned, "queries": turned + sums - 4 * batch * g.n + 8 * g.n,
            "all": turned + sums + 4 * MB}[room]
    with gs.ScanIndex.build(g) as ix:
        want = ix.sweep(mus, epss)
        with memory.at_most(need + more):
            got = ix.sweep(mus, epss)
    assert np.array_equal(got, want)


def graphs():
    return {"sbm": graphgen.sbm(10000, 50, 0.05, 0.0004, seed=1),
            "rmat": graphgen.rmat(13, 16, seed=2),
            "sparse": graphgen.sbm(60000, 3000, 0.05, 0.00001, seed=3),
            "tiny": graphgen.sbm(500, 5, 0.1, 0.01, seed=4)}


def figure(g):
    """Device bytes of a build, without what is only there for speed."""
    return 51 * g.arcs + 36 * g.n + MB


def same(a, b):
    for key in a:
        assert np.array_equal(a[key], b[key]), key


@pytest.mark.parametrize("name", ["sbm", "rmat", "sparse", "tiny"])
@pytest.mark.parametrize("kind", [gs.COSINE, gs.JACCARD])
def test_builds_in_little_room(memory, name, kind):
    g = graphs()[name]
    with gs.ScanIndex.build(g, kind, counts=gs.COUNTS_SPARSE) as ix:
        want = ix.export()
    with memory.at_most(figure(g)):
        ix = gs.ScanIndex.build(g, kind, counts=gs.COUNTS_SPARSE)
    got = ix.export()
    ix.free()
    same(got, want)


def test_batch_and_counts_in_little_room(memory):
    gl = [graphgen.sbm(3000 + 500 * i, 20, 0.05, 0.001, seed=i) for i in range(6)]
    n, arcs = sum(g.n for g in gl), sum(g.arcs for g in gl)
    want = []
    for ix in gs.ScanIndex.build_batch(gl):
        want.append(ix.export())
        ix.free()
    # a build of the union, and offsets relative to each graph
    with memory.at_most(51 * arcs + 36 * n + MB + 16 * (n + len(gl))):
        ixs = gs.ScanIndex.build_batch(gl)
    for ix, w in zip(ixs, want):
        same(ix.export(), w)
        ix.free()
    g = graphs()["rmat"]
    counts = gs.closed_counts_range(g, 0, g.n)
    # the graph and the counts (8 bytes an arc), the counting's own (28)
    with memory.at_most(36 * g.arcs + 36 * g.n + MB):
        assert np.array_equal(gs.closed_counts_range(g, 0, g.n), counts)


@pytest.mark.parametrize("name", ["sbm", "rmat", "sparse", "tiny"])
@pytest.mark.parametrize("more", [0, 2 * MB, 8 * MB])
def test_server_builds_stay_within_their_budget(memory, name, more):
    g = graphs()[name]
    with gs.ScanIndex.build(g) as ix:
        want = ix.export()
    budget = figure(g) + more
    with gs.Server(memory_budget=budget) as srv:
        memory.peak = memory.held
        ix = srv.wait(srv.submit_build(g, gs.COSINE), timeout_ms=60000)
        assert memory.peak - memory.held + ix.device_bytes <= budget
    same(ix.export(), want)
    ix.free()


def test_out_of_memory_is_reported(memory):
    g = graphs()["sbm"]
    with memory.at_most(28 * g.arcs):
        for call in (lambda: gs.ScanIndex.build(g), lambda: gs.ScanIndex.build_batch([g, g]),
                     lambda: gs.closed_counts_range(g, 0, g.n)):
            with pytest.raises(gs.ScanError) as e:
                call()
            assert e.value.status == -2


@pytest.mark.parametrize("nseg,length", [(1, 400000), (40000, 10), (60, 9000)])
def test_sort_in_little_room(memory, nseg, length):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(5)
    keys = torch.randint(0, 5000, (nseg * length,), device="cuda", generator=gen).double()
    ids = torch.arange(nseg * length, device="cuda", dtype=torch.int32) % length
    off = torch.arange(nseg + 1, device="cuda", dtype=torch.int64) * length
    sorted_in = []
    for less in (0, 3 * MB):  # with the slab of 4 MB, then less than that needs
        k, v = keys.clone(), ids.clone()
        with memory.at_most((memory.peak - less) if less else 1 << 40):
            gs.sort_segments_desc(k, v, off, max_len=length)
        sorted_in.append((k.cpu().numpy(), v.cpu().numpy()))
    for a, b in zip(*sorted_in):
        assert np.array_equal(a, b)
    order = np.lexsort((ids.cpu().numpy(), -keys.cpu().numpy(),
                        np.repeat(np.arange(nseg), length)))
    assert np.array_equal(sorted_in[0][1], ids.cpu().numpy()[order])
