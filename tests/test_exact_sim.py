"""The integer forms of the cosine and the Jaccard similarity (csrc/exact_sim.cuh)
against IEEE double arithmetic, bit for bit: c / sqrt(P) and c / D for operands
of every size, at the ends of their ranges, for squares, products of neighbours
and equal operands, with the hardware approximation they start from exact, at
its documented error, and twice as far off. Host code, compiled here."""
import subprocess
import textwrap

import numpy as np
import pytest

import paper_2012_11188_gb300._build as build

SOURCE = """
static float es_error = 0;
#define GS_ES_ERROR es_error
#include "exact_sim.cuh"
extern "C" void run(long n, float error, const unsigned* c, const unsigned long long* p,
                    const unsigned* d, double* cosine, double* ratio) {
  es_error = error;
  for (long i = 0; i < n; ++i) {
    cosine[i] = gscan::exact_cosine(c[i], p[i]);
    ratio[i] = gscan::exact_ratio(c[i], d[i]);
  }
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import ctypes
    tmp = tmp_path_factory.mktemp("exact_sim")
    src, so = tmp / "t.cpp", tmp / "t.so"
    src.write_text(textwrap.dedent(SOURCE))
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off",
                    "-I", build.CSRC, str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    lib.run.argtypes = [ctypes.c_long, ctypes.c_float] + [ctypes.c_void_p] * 5

    def call(error, c, p, d):
        out = np.empty(len(c)), np.empty(len(c))
        lib.run(len(c), error, c.ctypes.data, p.ctypes.data, d.ctypes.data, out[0].ctypes.data,
                out[1].ctypes.data)
        return out
    return call


def operands(n, seed):
    r = np.random.default_rng(seed)
    size = lambda bits: np.maximum(1, r.integers(0, 2 ** 62, n) >> (62 - r.integers(1, bits + 1, n)))  # noqa: E731
    u, v = size(26), size(26)
    k = np.arange(n) % 5
    v = np.where(k == 1, u + r.integers(0, 3, n), np.where(k == 2, u, v))
    p = u.astype(np.uint64) * v.astype(np.uint64)
    c = np.where(k == 3, np.minimum(u, v), size(31))
    d = np.where(k == 4, c, size(32))
    edge = np.array([1, 2, 3, 4, 2 ** 31 - 1, 2 ** 31, 2 ** 32 - 1], dtype=np.uint64)
    ce, de = (x.ravel() for x in np.meshgrid(edge, edge))
    pe = de * np.uint64(2 ** 20 + 1)
    return (np.concatenate([c, ce]).astype(np.uint32), np.concatenate([p, pe]).astype(np.uint64),
            np.concatenate([d, de]).astype(np.uint32))


@pytest.mark.parametrize("error", [0.0, 2.0 ** -22, -2.0 ** -22, 2.0 ** -21, -2.0 ** -21])
def test_bits(run, error):
    c, p, d = operands(1_000_000, 3)
    assert int(p.max()) < 2 ** 53
    cosine, ratio = run(error, c, p, d)
    cd = c.astype(np.float64)
    assert np.array_equal(cosine, cd / np.sqrt(p.astype(np.float64)))
    assert np.array_equal(ratio, cd / d.astype(np.float64))
