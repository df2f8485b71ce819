"""Host code of the library where the outcome depends on the machine: memory of
another device, refused launches, arrays shorter than the call says. On a CUDA runtime of host
memory."""
import ctypes

import numpy as np
import pytest

import fake_cuda


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fake_cuda.Fake(str(tmp_path_factory.mktemp("fake_cuda")))


@pytest.fixture()
def clean(fake):
    yield fake
    fake.lib.fake_set_device(0)
    fake.lib.fake_refuse_cooperative(0)


def edgeless(fake, n=5):
    off, adj = np.zeros(n + 1, np.int64), np.zeros(0, np.int32)
    return fake.build(fake.csr(off, adj, 0)), (off, adj)


# device of the index, of the destination, and the current one; what copies
@pytest.mark.parametrize("index,dst,now,kernel", [(0, 0, 0, True), (1, 1, 1, True),
                                                  (0, 1, 1, False), (0, 1, 0, False),
                                                  (0, 0, 1, False)])
def test_export_across_devices(clean, index, dst, now, kernel):
    """A kernel of the current device copies only where both sides are its
    own memory; everything else is a copy of the runtime's."""
    fake = clean
    fake.lib.fake_set_device(index)
    h, _ = edgeless(fake)
    co_off = np.full(1, 77, np.int64)
    fake.region(co_off, device=dst)
    fake.lib.fake_set_device(now)
    fake.lib.fake_clear_log()
    assert fake.lib.scan_index_export(h, None, None, None, co_off.ctypes.data, None, None) == 0
    log = fake.log()
    assert any("k_export" in x for x in log) == kernel
    if not kernel:
        assert co_off[0] == 0 and "copy 8" in log
    fake.lib.fake_set_device(index)
    fake.lib.scan_index_free(h)


EBADGRAPH, ECUDA = -3, -4


@pytest.mark.parametrize("short", [None, "offsets", "adj"])
@pytest.mark.parametrize("off_type", [np.int64, np.int32])
def test_batch_of_short_arrays(clean, short, off_type):
    """Kernels pack a batch from the callers' arrays only where those are as
    long as the call says: a copy refuses the others, a kernel would read past
    their ends."""
    fake = clean
    off, adj = np.array([0, 2, 4, 6], off_type), np.array([1, 2, 0, 2, 0, 1], np.int32)
    fake.region(off, nbytes=off.nbytes - off.itemsize if short == "offsets" else None)
    fake.region(adj, nbytes=adj.nbytes - 8 if short == "adj" else None)
    graphs = (fake_cuda.scan_csr * 2)(*[fake.csr(off, adj, 1)] * 2)
    out = (ctypes.c_void_p * 2)()
    fake.lib.fake_clear_log()
    rc = fake.lib.scan_index_build_batch(graphs, 2, 0, None, 0, out)
    log = fake.log()
    # (the kernels do nothing here, so the checks of a whole graph find no edge)
    assert rc == (ECUDA if short else EBADGRAPH)
    assert any("k_pack" in x for x in log) == (short is None)
    assert ("copy refused" in log) == (short is not None)


@pytest.mark.parametrize("short", [False, True])
def test_export_to_a_short_array(clean, short):
    fake = clean
    h, _ = edgeless(fake)
    co_off = np.full(1, 77, np.int64)
    fake.region(co_off, nbytes=4 if short else 8)
    fake.lib.fake_clear_log()
    rc = fake.lib.scan_index_export(h, None, None, None, co_off.ctypes.data, None, None)
    assert rc == (ECUDA if short else 0)
    assert any("k_export" in x for x in fake.log()) != short
    fake.lib.scan_index_free(h)


@pytest.mark.parametrize("refuse", [False, True])
@pytest.mark.parametrize("device", [False, True])
def test_query_where_a_cooperative_launch_is_refused(clean, refuse, device):
    """A single query is one cooperative launch; a stream or a process with
    fewer multiprocessors than the device refuses it, and the launches of a
    batch answer."""
    fake = clean
    h, _ = edgeless(fake)
    labels = np.full(5, 77, np.int32)
    if device:
        fake.region(labels)
    fake.lib.fake_refuse_cooperative(int(refuse))
    fake.lib.fake_clear_log()
    assert fake.lib.scan_query(h, 2, 0.5, labels.ctypes.data, 1, 0) == 0
    log = fake.log()
    assert any("k_query_one" in x for x in log)
    for name in ("k_get_cores", "k_core_prefix", "k_mark_cores", "k_union", "k_labels", "k_hubs"):
        assert any(name in x for x in log) == refuse, name
    if refuse:  # cleared by the batch's own memset
        assert (labels == -1).all()
    fake.lib.scan_index_free(h)
