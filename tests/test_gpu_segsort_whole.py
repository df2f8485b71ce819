"""Segments of 4097 to 16384 elements when no segment is longer and there are
no more of them than multiprocessors: sorted whole by one CTA. Lengths around
the thread's 16 elements, the class bounds and the largest, tie patterns, and
one segment or one element more, which take the sample-sort split again.
Against numpy."""
import numpy as np
import pytest

import paper_2012_11188_gb300 as gs

pytestmark = pytest.mark.gpu


def check(keys, ids, lens):
    import torch
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    k, v = torch.from_numpy(keys).cuda(), torch.from_numpy(ids).cuda()
    gs.sort_segments_desc(k, v, torch.from_numpy(off).cuda())
    k, v = k.cpu().numpy(), v.cpu().numpy()
    for a, b in zip(off[:-1], off[1:]):
        o = np.lexsort((ids[a:b], -keys[a:b]))
        assert np.array_equal(k[a:b], keys[a:b][o]) and np.array_equal(v[a:b], ids[a:b][o]), b - a


@pytest.mark.parametrize("pattern", ["random", "equal", "two_values", "ascending", "descending",
                                     "rounded"])
@pytest.mark.parametrize("longest", [16384, 16385])
def test_whole_segments(pattern, longest):
    rng = np.random.default_rng(5)
    lens = np.array([longest, 4096, 4097, 4098, 5000, 0, 1, 33, 8191, 8192, 8193, 12000, 16383,
                     16369, 16368])
    total = int(lens.sum())
    ids = rng.permutation(total).astype(np.int32)
    keys = {"random": lambda: rng.random(total), "equal": lambda: np.full(total, 0.5),
            "two_values": lambda: rng.choice([0.0, 0.75], total),
            "ascending": lambda: np.sort(rng.random(total)),
            "descending": lambda: -np.sort(-rng.random(total)),
            "rounded": lambda: np.round(rng.random(total), 2)}[pattern]()
    check(keys, ids, lens)


@pytest.mark.parametrize("count", [1, 100, 400, 3000])
def test_counts_of_long_segments(count):
    """Few enough for a CTA each, split into buckets, and so many that those
    of up to 8192 are sorted by one CTA each again."""
    rng = np.random.default_rng(6)
    lens = rng.integers(4097, 8194, count)
    lens[:3] = [8192, 8193, 4097][:count]
    total = int(lens.sum())
    check(rng.random(total), rng.permutation(total).astype(np.int32), lens)
