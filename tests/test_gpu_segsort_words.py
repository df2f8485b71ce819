"""Segments of 33 to 4096 elements, sorted as packed 64-bit words where the
ranges of their keys and ids leave room and as pairs elsewhere: zeros,
denormals, 1e-300 to 1e300, infinity, keys a few units in the last place
apart, ids of every width up to all 32 bits, ranges that fill the 64 bits to
the last one or are one bit too wide, and the lengths around the thread's 8
words, a warp's 256 and the classes. Against numpy. (Ascending ids, which take
the position instead, are those of every index build.)"""
import numpy as np
import pytest

import paper_2012_11188_gb300 as gs

pytestmark = pytest.mark.gpu

LENS = np.array([33, 34, 39, 40, 41, 64, 100, 255, 256, 257, 264, 500, 511, 512, 513, 700, 1023,
                 1024, 1025, 1500, 2047, 2048, 2049, 3000, 4088, 4089, 4095, 4096] * 3)


def ulps(rng, n, spread):
    """0.5 plus a few units in the last place."""
    return np.frombuffer((np.float64(0.5).view(np.int64) +
                          rng.integers(0, spread, n)).astype(np.int64).tobytes(), np.float64)


KEYS = {
    "similarities": lambda r, n: r.integers(2, 30, n) / np.sqrt(r.integers(4, 4000, n) * 1.0),
    "uniform": lambda r, n: r.random(n),
    "narrow": lambda r, n: 0.75 + r.random(n) * 2.0 ** -20,
    "zeros": lambda r, n: np.where(r.random(n) < 0.3, 0.0, 0.25 + r.random(n) / 64),
    "all_zero": lambda r, n: np.zeros(n),
    "wide": lambda r, n: 10.0 ** r.uniform(-300, 300, n),
    "denormal": lambda r, n: np.where(r.random(n) < 0.5, 5e-324 * r.integers(0, 9, n), r.random(n)),
    "infinity": lambda r, n: np.where(r.random(n) < 0.01, np.inf, r.random(n)),
    "ulps_few": lambda r, n: np.where(r.random(n) < 0.002, 1e-200, ulps(r, n, 1 << 40)),
    "ulps_runs": lambda r, n: np.where(r.random(n) < 0.01, 1e-200, ulps(r, n, 50)),
}
IDS = {
    "small": lambda r, n: r.permutation(n).astype(np.int32),
    "wide": lambda r, n: r.choice(2 ** 31 - 1, n, replace=False).astype(np.int32),
    "signed": lambda r, n: np.unique(r.integers(-2 ** 31, 2 ** 31, 2 * n))[
        r.permutation(n)].astype(np.int32),
    "ascending": lambda r, n: np.arange(n, dtype=np.int32),
}


@pytest.mark.parametrize("ids", list(IDS))
@pytest.mark.parametrize("keys", list(KEYS))
def test_words(keys, ids):
    import torch
    rng = np.random.default_rng(17)
    n = int(LENS.sum())
    k, v = KEYS[keys](rng, n), IDS[ids](rng, n)
    off = np.concatenate([[0], np.cumsum(LENS)]).astype(np.int64)
    dk, dv = torch.from_numpy(k.copy()).cuda(), torch.from_numpy(v.copy()).cuda()
    gs.sort_segments_desc(dk, dv, torch.from_numpy(off).cuda())
    dk, dv = dk.cpu().numpy(), dv.cpu().numpy()
    for a, b in zip(off[:-1], off[1:]):
        o = np.lexsort((v[a:b], -k[a:b]))
        assert np.array_equal(dk[a:b], k[a:b][o]), (b - a)
        assert np.array_equal(dv[a:b], v[a:b][o]), (b - a)


@pytest.mark.parametrize("over", [-1, 0, 1])
@pytest.mark.parametrize("vbits", [6, 12, 24, 31, 32])
def test_words_filled_to_the_last_bit(vbits, over):
    """Key and id ranges of exactly 64 - vbits + over and vbits bits."""
    import torch
    rng = np.random.default_rng(vbits)
    lens = [60, 64]
    kbits = min(62, 64 - vbits + over)
    k, v = [], []
    for n in lens:
        d = rng.integers(0, 1 << kbits, n, dtype=np.uint64)
        d[0], d[1] = 0, (1 << kbits) - 1
        k.append((d + np.uint64(1)).view(np.float64))
        x = rng.choice(1 << min(vbits, 20), n, replace=False).astype(np.int64) << max(0, vbits - 20)
        x[x == x.max()] = (1 << vbits) - 1
        x[x == x.min()] = 0
        v.append((x - (1 << 31) if vbits == 32 else x).astype(np.int32))
    k, v = np.concatenate(k), np.concatenate(v)
    off = np.array([0, lens[0], sum(lens)], dtype=np.int64)
    dk, dv = torch.from_numpy(k.copy()).cuda(), torch.from_numpy(v.copy()).cuda()
    gs.sort_segments_desc(dk, dv, torch.from_numpy(off).cuda())
    dk, dv = dk.cpu().numpy(), dv.cpu().numpy()
    bits = k.view(np.uint64)
    for a, b in zip(off[:-1], off[1:]):
        o = np.lexsort((v[a:b], ~bits[a:b]))
        assert np.array_equal(dk[a:b].view(np.uint64), bits[a:b][o])
        assert np.array_equal(dv[a:b], v[a:b][o])
