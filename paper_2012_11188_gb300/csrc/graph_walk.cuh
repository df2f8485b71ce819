// The graph of an element of packed graphs: graph g owns the elements base[g]
// .. base[g + 1) of the union (G + 1 ascending bases; a graph may be empty).
#pragma once

#include <stdint.h>

namespace gscan {

#ifdef __CUDACC__
#define GS_WALK_HD __host__ __device__ __forceinline__
#else
#define GS_WALK_HD inline
#endif

// largest i in [lo, hi) with a[i] <= x (a[lo] <= x)
template <class A>
GS_WALK_HD int64_t last_le(const A& a, int64_t lo, int64_t hi, int64_t x) {
  while (hi - lo > 1) {
    const int64_t mid = (lo + hi) >> 1;
    if (a[mid] <= x) lo = mid; else hi = mid;
  }
  return lo;
}

// Graphs of ascending elements: a few steps on from the last one's, and a
// search of the rest where that is not enough, so that an element never costs
// more than STEPS loads and a search whatever lies between (without the
// search a chunk with 20,000 empty graphs in it was 20,000 dependent loads
// for each of its threads: the batched build of two graphs with 20,000 empty
// ones between them took 16.5 ms in all, now 10.9).
template <class A>
struct GraphWalk {
  static constexpr int STEPS = 4;
  A base;
  int64_t G, g;
  GS_WALK_HD GraphWalk(A a, int64_t graphs, int64_t first)
      : base(a), G(graphs), g(last_le(a, 0, graphs, first)) {}
  GS_WALK_HD int64_t at(int64_t i) {  // i below base[G], not below the last one
    for (int k = 0; k < STEPS; ++k) {
      if (base[g + 1] > i) return g;
      ++g;
    }
    return g = last_le(base, g, G, i);
  }
};

}  // namespace gscan
