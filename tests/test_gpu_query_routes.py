"""Single queries on either side of their routes: few cores (one cooperative
launch) and many (the launches of a batch), hubs in the launch and after it,
labels copied at once and after the wait, no cores at all. Against the batch
and, where it is quick, the oracle."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2012_11188_gb300 as gs

pytestmark = pytest.mark.gpu


def ring(n, k):
    """Every vertex next to the k nearest on both sides; two long chords."""
    steps = np.concatenate([np.arange(1, k + 1), -np.arange(1, k + 1)])
    rows = np.sort((np.arange(n)[:, None] + steps[None, :]) % n, axis=1)
    return np.arange(n + 1, dtype=np.int64) * (2 * k), rows.astype(np.int32).reshape(-1)


def launches(call):
    before = gs.kernel_launches()
    call()
    return gs.kernel_launches() - before


# vertices, both sides' neighbours, whether all vertices as cores are many
@pytest.mark.parametrize("n,k,many", [(500, 4, False), (38000, 4, False), (40000, 4, False),
                                      (66000, 3, False), (600000, 4, True), (60000, 150, True)])
@pytest.mark.parametrize("hubs", [False, True])
def test_all_or_none_are_cores(n, k, many, hubs):
    import torch
    with gs.ScanIndex.build(ring(n, k)) as ix:
        out = torch.empty(n, dtype=torch.int32, device="cuda")
        for mu, eps, cores in ((2, 0.1, True), (k, 0.0, True), (2 * k + 1, 0.05, True),
                               (2 * k + 2, 0.0, False), (2, 1.0, False)):
            out.fill_(77)
            took = launches(lambda: ix.query(mu, eps, hubs=hubs, out=out))
            assert (out.cpu().numpy() == (0 if cores else -1)).all(), (mu, eps)
            # one launch, hubs perhaps another; a batch is at least five
            assert (took > 3) == (many and cores), (mu, eps, took)
            host = np.full(n, 77, np.int32)
            ix.query(mu, eps, hubs=hubs, out=host)
            assert (host == (0 if cores else -1)).all(), (mu, eps)


@pytest.mark.parametrize("scale", [10, 15, 17])
@pytest.mark.parametrize("hubs", [False, True])
def test_single_equals_batch(scale, hubs):
    g = graphgen.rmat(scale, 16, seed=scale)
    pairs = [(m, e) for m in (2, 3, 5, 20, 100) for e in (0.0, 0.05, 0.2, 0.4)]
    with gs.ScanIndex.build(g) as ix:
        rows = ix.query_batch([m for m, _ in pairs], [e for _, e in pairs], hubs=hubs)
        for (mu, eps), row in zip(pairs, rows):
            assert np.array_equal(ix.query(mu, eps, hubs=hubs), row), (mu, eps)
    if scale == 10:
        ox = oracle.Index(g)
        for (mu, eps), row in zip(pairs, rows):
            assert np.array_equal(row, ox.query(mu, eps, hubs=hubs)), (mu, eps)
