"""The graph of every element of packed graphs (csrc/graph_walk.cuh), host code
compiled here: against numpy's search, and how many bases an element reads,
whatever number of empty graphs lies between two elements."""
import ctypes
import subprocess

import numpy as np
import pytest

import paper_2012_11188_gb300._build as build

SOURCE = """
#include "graph_walk.cuh"
static long loads;
struct Counted {
  const int64_t* p;
  int64_t operator[](int64_t i) const { ++loads; return p[i]; }
};
// graphs of first, first + step, ... below end, and the loads of each
extern "C" void walk(const int64_t* base, int64_t G, int64_t first, int64_t step, int64_t end,
                     int64_t* g, int64_t* cost) {
  loads = 0;
  gscan::GraphWalk<Counted> w(Counted{base}, G, first);
  for (int64_t i = first; i < end; i += step) {
    *g++ = w.at(i);
    *cost++ = loads;
    loads = 0;
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    tmp = tmp_path_factory.mktemp("graph_walk")
    src, so = tmp / "t.cpp", tmp / "t.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, str(src),
                    "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    P, L = ctypes.c_void_p, ctypes.c_int64
    lib.walk.argtypes = [P, L, L, L, L, P, P]
    return lib


SIZES = {
    "one": [7],
    "even": [10] * 500,
    "triangles": [6] * 20000,
    "empty between": [3000] + [0] * 20000 + [3000],
    "empty at the ends": [0] * 300 + [5, 0, 0, 1, 900] + [0] * 300,
    "single elements": [1, 0] * 3000,
    "random": list(np.random.default_rng(1).integers(0, 40, 3000)),
}


@pytest.mark.parametrize("name", SIZES)
@pytest.mark.parametrize("step", [1, 256])
def test_walk(lib, name, step):
    sizes = np.array(SIZES[name], np.int64)
    base = np.concatenate([[0], np.cumsum(sizes)])
    G = len(sizes)
    search = int(np.ceil(np.log2(max(G, 2)))) + 1
    for c0 in range(0, int(base[-1]), 4096):
        for first in sorted({c0, min(c0 + 1, int(base[-1]) - 1), min(c0 + 255, int(base[-1]) - 1)}):
            end = min(int(base[-1]), c0 + 4096)
            at = np.arange(first, end, step)
            if len(at) == 0:
                continue
            g, cost = np.empty_like(at), np.empty_like(at)
            lib.walk(base.ctypes.data, G, first, step, end, g.ctypes.data, cost.ctypes.data)
            assert np.array_equal(g, np.searchsorted(base, at, side="right") - 1)
            assert cost[0] <= search + 1 + 4 + search
            assert cost[1:].max(initial=0) <= 4 + search
