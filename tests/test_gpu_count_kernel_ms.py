"""scan_last_count_kernel_ms: the CTA counting kernels of the last build, a
batch's in all its builds, 0 where none ran."""
import numpy as np
import pytest

import graphgen
import paper_2012_11188_gb300 as gs

pytestmark = pytest.mark.gpu


def dense_graph(n=4200, degree=800):
    """Ring of n vertices, each next to the `degree` nearest: the dense path's."""
    steps = np.concatenate([np.arange(1, degree // 2 + 1), -np.arange(1, degree // 2 + 1)])
    rows = np.sort((np.arange(n)[:, None] + steps[None, :]) % n, axis=1)
    return np.arange(n + 1, dtype=np.int64) * degree, rows.astype(np.int32).reshape(-1)


def after(call):
    for ix in call():
        ix.free()
    return gs.last_count_kernel_ms()


def test_last_count_kernel_ms():
    sparse = graphgen.rmat(14, 16, seed=1)
    dense = dense_graph()
    empty = (np.zeros(11, np.int64), np.zeros(0, np.int32))
    assert after(lambda: [gs.ScanIndex.build(sparse)]) > 0
    assert after(lambda: [gs.ScanIndex.build(dense)]) == 0
    assert after(lambda: [gs.ScanIndex.build(sparse)]) > 0
    assert after(lambda: [gs.ScanIndex.build(empty)]) == 0
    # some members by the matrix product, the others together
    assert after(lambda: gs.ScanIndex.build_batch([sparse, dense])) > 0
    assert after(lambda: gs.ScanIndex.build_batch([dense, sparse, dense])) > 0
    assert after(lambda: gs.ScanIndex.build_batch([dense, dense])) == 0
    assert after(lambda: gs.ScanIndex.build_batch([empty, empty])) == 0
