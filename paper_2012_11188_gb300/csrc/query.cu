// (mu, eps) queries on the index (Algorithms 3-5, Section 6.2, Section 4.3).
//
// Phases, each over all (query, core) items of a batch:
//  1. GetCores (Algorithm 3): the cores are the prefix of CO[mu] whose
//     threshold is >= eps; its length comes from one search (CO[mu] is
//     sorted by non-increasing threshold). The prefix marks parent[v] = v.
//  2. Cluster (Algorithm 5, union-find of Section 6.2): every core u takes the
//     eps-prefix of NO[u] and unions with each core neighbour of larger id.
//     The union-find is lock-free: find() halves paths, unite() CASes the
//     larger root under the smaller one, so every root is the smallest id of
//     its component and labels are canonical.
//  3. AssignNonCores (Algorithm 4) with the deterministic rule of Section
//     7.3.4: a non-core takes the label of the first core in its own
//     eps-prefix of NO -- the most similar eps-similar core, smallest id among
//     equal similarities (NO breaks ties by id). Only the non-cores found in
//     the cores' eps-prefixes are visited (each claimed once by a CAS on its
//     label), so the query's work follows the eps-edges of its clusters
//     (Theorem 4.3's O(Z)) plus two clears of n words; every other label
//     stays -1.
//  4. With SCAN_Q_HUBS (Section 4.3): an unclustered vertex whose neighbours
//     carry two distinct labels becomes -2.
//
// What bounds them is latency, not bytes: dependent loads (a search, a
// neighbour, its parent), the longest row a single warp walks, and the
// launches. So searches are 32-way (a warp probes 32 places at once: five
// steps for 4M entries instead of 22); prefixes longer than PIECE entries go
// to a queue in pieces that any warp may take (R-MAT s22 has rows of 1.5e5
// entries: a batch of 64 queries spent 2.2 ms in phase 2 on the warps that
// walked them, and one thread scanning a border's long prefix alone made
// phase 3 83% of a parameter sweep); and a single query with little work is one
// cooperative launch whose phases are separated by grid barriers, instead of
// eight launches, two clears and three small copies.
// Measured against one launch per phase, binary searches and whole rows: one
// query with hubs on an SBM graph of 10k vertices 80 -> 49 us, (5, 0.3) on R-MAT
// s22 76 -> 29 us, 594 pairs of a sweep on R-MAT s20 420 -> 48 ms. A batch of 64
// queries gains by which queries it holds: sets of the same ranges take 0.6 to
// 1.4 ms.
#include <cooperative_groups.h>

#include "scan_internal.cuh"

namespace gscan {

namespace {

constexpr int UNITE_LIMIT = 1 << 22;

__device__ __forceinline__ int32_t ld_volatile(const int32_t* p) {
  return *(const volatile int32_t*)p;
}

__device__ __forceinline__ int32_t uf_find(int32_t* parent, int32_t x) {
  for (int it = 0; it < UNITE_LIMIT; ++it) {
    const int32_t p = ld_volatile(parent + x);
    if (p == x) return x;
    const int32_t gp = ld_volatile(parent + p);
    if (gp != p) atomicCAS(parent + x, p, gp);  // path halving; only moves towards the root
    x = gp;
  }
  return x;
}

__device__ __forceinline__ bool uf_unite(int32_t* parent, int32_t a, int32_t b) {
  for (int it = 0; it < UNITE_LIMIT; ++it) {
    a = uf_find(parent, a);
    b = uf_find(parent, b);
    if (a == b) return true;
    if (a > b) { const int32_t t = a; a = b; b = t; }
    if (atomicCAS(parent + b, b, a) == b) {  // hook larger root under smaller
      // Roots hooked at the same time form a chain as long as there are warps (a
      // ring whose vertices know only their neighbours: one find along it was 2 of
      // a query's 3 ms). Halving it here is everyone's work side by side, and at
      // most one more find per vertex.
      uf_find(parent, b);
      return true;
    }
  }
  return false;
}

// Warp-wide: number of leading entries of the non-increasing array
// x[0..len) that are >= eps, 32 probes a step.
__device__ __forceinline__ int64_t prefix_ge(const double* __restrict__ x, int64_t len, double eps) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, hi = len;  // the answer is in [lo, hi]
  while (hi - lo > 32) {
    const int64_t step = (hi - lo + 32) / 33;
    const int64_t at = lo + step * (lane + 1) - 1;
    const unsigned m = __ballot_sync(0xffffffffu, at < hi && x[at] >= eps);
    const int c = __popc(m);  // the first c probes hold
    const int64_t nlo = lo + step * c;
    if (c < 32) hi = min(hi, nlo + step - 1);  // probe c does not
    lo = nlo;
  }
  const int64_t at = lo + lane;
  return lo + __popc(__ballot_sync(0xffffffffu, at < hi && x[at] >= eps));
}

// A piece of a core's eps-prefix, for any warp to take.
constexpr int PIECE = 1024;
struct QPiece {
  int32_t q, u;
  int32_t begin, end;  // entries of NO[u]; begin = end: none
};

struct QArgs {
  const int64_t* off;
  const int32_t* deg;
  const int32_t* adj;
  const int32_t* no_id;
  const double* no_sim;
  const int64_t* co_off;
  const int32_t* co_id;
  const double* co_thr;
  int64_t n;
  int32_t maxdeg;
  const int* mu;       // Q
  const double* eps;   // Q
  int64_t* ncp;        // Q+1: exclusive prefix of the core counts (flattened (query, core) items)
  int Q;
  int32_t* parent;     // Q * n (-1 = not a core)
  int32_t* labels;     // Q * n, used when lab_ptrs is null
  int32_t* const* lab_ptrs;  // Q destinations (device), or null
  unsigned* status;
  QPiece* queue;       // null: every warp walks its whole prefixes
  unsigned long long* queued;  // pieces asked for; more than queue_cap: the queue was full
  unsigned queue_cap;
  unsigned long long* reached;  // null, or receives the entries of all cores' prefixes
};

__device__ __forceinline__ int32_t* labels_of(const QArgs& a, int q) {
  return a.lab_ptrs ? a.lab_ptrs[q] : a.labels + (int64_t)q * a.n;
}

__global__ void k_init_labels(QArgs a) {
  int32_t* lab = labels_of(a, blockIdx.y);
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < a.n;
       v += (int64_t)gridDim.x * blockDim.x)
    lab[v] = -1;
}

// item i of the flattened (query, core) list -> query q, core index i - ncp[q]
__device__ __forceinline__ int item_query(const QArgs& a, int64_t i) {
  int lo = 0, hi = a.Q;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (a.ncp[mid] <= i) lo = mid; else hi = mid;
  }
  return lo;
}

// Warp-wide: number of cores of (mu, eps).
__device__ __forceinline__ int64_t count_cores(const QArgs& a, int mu, double eps) {
  if (mu < 2 || mu > a.maxdeg + 1) return 0;
  const int64_t b = a.co_off[mu - 2], e = a.co_off[mu - 1];
  return prefix_ge(a.co_thr + b, e - b, eps);
}

// Core counts of all queries, a warp each, into ncp[0..Q); then their
// exclusive prefix sums in place (one CTA).
__global__ void k_get_cores(QArgs a) {
  const int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (q >= a.Q) return;
  const int64_t c = count_cores(a, a.mu[q], a.eps[q]);
  if ((threadIdx.x & 31) == 0) a.ncp[q] = c;
}

constexpr int PREFIX_T = 256;
__global__ void __launch_bounds__(PREFIX_T) k_core_prefix(QArgs a) {
  __shared__ int64_t ws[PREFIX_T / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int64_t carry = 0;
  for (int q0 = 0; q0 < a.Q; q0 += PREFIX_T) {
    const int q = q0 + threadIdx.x;
    const int64_t own = q < a.Q ? a.ncp[q] : 0;
    int64_t inc = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) ws[wid] = inc;
    __syncthreads();
    int64_t before = carry;
    for (int w = 0; w < PREFIX_T / 32; ++w) {
      if (w < wid) before += ws[w];
      carry += ws[w];
    }
    if (q < a.Q) a.ncp[q] = before + inc - own;
    __syncthreads();
  }
  if (threadIdx.x == 0) a.ncp[a.Q] = carry;
}

// One query's arguments, or the batch's by item: what a phase needs of item it.
struct Item {
  int q;
  int32_t u;
  double eps;
  int32_t* parent;
  int32_t* lab;
};
template <bool ONE>
__device__ __forceinline__ Item item_at(const QArgs& a, int64_t it, int mu, double eps) {
  if (ONE) return {0, a.co_id[a.co_off[mu - 2] + it], eps, a.parent, a.labels};
  const int q = item_query(a, it);
  return {q, a.co_id[a.co_off[a.mu[q] - 2] + (it - a.ncp[q])], a.eps[q],
          a.parent + (int64_t)q * a.n, labels_of(a, q)};
}

template <bool ONE>
__device__ __forceinline__ void phase_mark(const QArgs& a, int64_t total, int mu, double eps,
                                           int64_t t0, int64_t nt) {
  for (int64_t it = t0; it < total; it += nt) {
    const Item x = item_at<ONE>(a, it, mu, eps);
    x.parent[x.u] = x.u;
  }
}

// unions of core u with the cores of larger id in entries [b, e) of NO[u]
__device__ __forceinline__ bool union_range(const QArgs& a, int32_t* parent, int32_t u, int64_t b,
                                            int64_t e) {
  const int lane = threadIdx.x & 31;
  const int32_t* ids = a.no_id + a.off[u];
  bool ok = true;
  for (int64_t j = b + lane; j < e; j += 32) {
    const int32_t x = ids[j];
    if (x > u && ld_volatile(parent + x) >= 0) ok &= uf_unite(parent, u, x);
  }
  return ok;
}

// A warp per (query, core) item; what is past the first PIECE entries of a
// prefix is queued if there is room for all of it, else walked here.
template <bool ONE>
__device__ __forceinline__ void phase_union(const QArgs& a, int64_t total, int mu, double eps,
                                            int64_t w0, int64_t nw) {
  const int lane = threadIdx.x & 31;
  bool fail = false;
  unsigned reached = 0;  // (rows of more than 2^16 entries count as that many)
  for (int64_t it = w0; it < total; it += nw) {
    const Item x = item_at<ONE>(a, it, mu, eps);
    int64_t pu = prefix_ge(a.no_sim + a.off[x.u], a.deg[x.u], x.eps);
    if (!ONE) reached += (unsigned)min(pu, (int64_t)1 << 16);
    if (pu > PIECE && a.queue) {
      const unsigned np = (unsigned)((pu - 1) / PIECE);  // pieces past the first
      unsigned long long at = 0;
      if (lane == 0) at = atomicAdd(a.queued, (unsigned long long)np);
      at = __shfl_sync(0xffffffffu, at, 0);
      const bool fits = at + np <= a.queue_cap;
      for (unsigned i = lane; i < np && at + i < a.queue_cap; i += 32) {
        const int32_t b = (int32_t)(i + 1) * PIECE;
        const int32_t e = (int32_t)min(pu, (int64_t)b + PIECE);
        a.queue[at + i] = QPiece{x.q, x.u, b, fits ? e : b};
      }
      if (fits) pu = PIECE;
    }
    fail |= !union_range(a, x.parent, x.u, 0, pu);
  }
  if (!ONE && a.reached && reached && lane == 0) atomicAdd(a.reached, (unsigned long long)reached);
  if (__any_sync(0xffffffffu, fail) && lane == 0) atomicOr(a.status, (unsigned)DEV_LIMIT);
}

__device__ __forceinline__ void phase_union_queue(const QArgs& a, int64_t w0, int64_t nw) {
  const int lane = threadIdx.x & 31;
  const int64_t cnt = (int64_t)min(*a.queued, (unsigned long long)a.queue_cap);
  bool fail = false;
  for (int64_t i = w0; i < cnt; i += nw) {
    const QPiece p = a.queue[i];
    fail |= !union_range(a, a.parent + (int64_t)p.q * a.n, p.u, p.begin, p.end);
  }
  if (__any_sync(0xffffffffu, fail) && lane == 0) atomicOr(a.status, (unsigned)DEV_LIMIT);
}

// labels of the cores: their union-find root (the smallest id of the cluster)
template <bool ONE>
__device__ __forceinline__ void phase_core_labels(const QArgs& a, int64_t total, int mu, double eps,
                                                  int64_t t0, int64_t nt) {
  for (int64_t it = t0; it < total; it += nt) {
    const Item x = item_at<ONE>(a, it, mu, eps);
    x.lab[x.u] = uf_find(x.parent, x.u);
  }
}

constexpr int32_t CLAIMED = -3;
constexpr int OWN_STEP = 4;    // entries of its own prefix a border's lane looks at per step
constexpr int OWN_LEAST = 8;   // entries looked at before the warp may take over
constexpr int OWN_MOST = 64;   // and at which it takes over in any case
constexpr int OWN_LANES = 4;   // borders left over of which the warp takes over before

// 32 neighbours of core c, x in the lane's (-1: none, or a core). The lane that
// claims x first looks for the first core in x's own eps-prefix of NO (most
// similar, smallest id on ties; sigma is symmetric, so that prefix holds at
// least the core that found it). The lanes go through their prefixes side by
// side, OWN_STEP entries in flight each; once few are left, or the prefixes are
// long, the whole warp takes one border after another, 128 entries at a time.
// (One after another from the ninth entry on: 594 pairs of a sweep on R-MAT s20
// 51.8 ms, now 47.2.)
__device__ __forceinline__ void border_chunk(const QArgs& a, const Item& c, int32_t x) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int32_t* parent = c.parent;
  bool mine = x >= 0 && atomicCAS(c.lab + x, -1, CLAIMED) == -1;
  unsigned todo = __ballot_sync(FULL, mine);
  if (!todo) return;
  int64_t xb = 0;
  int32_t xd = 0;
  if (mine) {
    xb = a.off[x];
    xd = a.deg[x];
  }
  int t0 = 0;  // entries looked at
  do {
    if (mine) {
      double sv[OWN_STEP];
      int32_t y[OWN_STEP], py[OWN_STEP];
#pragma unroll
      for (int t = 0; t < OWN_STEP; ++t) {
        const bool in = t0 + t < xd;
        sv[t] = in ? a.no_sim[xb + t0 + t] : -1.0;
        y[t] = in ? a.no_id[xb + t0 + t] : x;
      }
#pragma unroll
      for (int t = 0; t < OWN_STEP; ++t) py[t] = ld_volatile(parent + y[t]);
      int32_t first = -1;
      bool over = false;  // the end of the prefix
#pragma unroll
      for (int t = 0; t < OWN_STEP; ++t) {
        over |= first < 0 && !(sv[t] >= c.eps);
        if (first < 0 && !over && py[t] >= 0) first = y[t];
      }
      // (over without a core cannot be with symmetric similarities)
      if (first >= 0 || over) {
        c.lab[x] = first >= 0 ? uf_find(parent, first) : -1;
        mine = false;
      }
    }
    t0 += OWN_STEP;
    todo = __ballot_sync(FULL, mine);
    if (!todo) return;
  } while (t0 < OWN_LEAST || (t0 < OWN_MOST && __popc(todo) > OWN_LANES));
  do {
    const int src = __ffs(todo) - 1;
    todo &= todo - 1;
    const int64_t rb = __shfl_sync(FULL, xb, src);
    const int32_t rd = __shfl_sync(FULL, xd, src);
    const int32_t xs = __shfl_sync(FULL, x, src);
    int32_t first = -1;
    bool end = false;
    for (int32_t t1 = t0; t1 < rd && first < 0 && !end; t1 += 128) {
      double sv[4];
      int32_t y[4], py[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int32_t t = t1 + 32 * k + lane;
        sv[k] = t < rd ? a.no_sim[rb + t] : -1.0;
        y[k] = t < rd ? a.no_id[rb + t] : xs;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) py[k] = ld_volatile(parent + y[k]);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const bool in = sv[k] >= c.eps;
        const unsigned m = __ballot_sync(FULL, in && py[k] >= 0);
        if (first < 0 && m) first = __shfl_sync(FULL, y[k], __ffs(m) - 1);
        end |= !__all_sync(FULL, in);
      }
    }
    if (lane == 0) c.lab[xs] = first >= 0 ? uf_find(parent, first) : -1;
  } while (todo);
}

// Every non-core in entries [b, e) of NO[u] is a border. Most entries are cores:
// 128 at a time are tested, and what is left goes on by chunks of 32.
__device__ __forceinline__ void border_range(const QArgs& a, const Item& c, uint32_t b, uint32_t e) {
  constexpr int W = 4;
  const int lane = threadIdx.x & 31;
  const int32_t* ids = a.no_id + a.off[c.u];
  for (uint32_t j0 = b; j0 < e; j0 += 32 * W) {
    int32_t x[W];
    unsigned some = 0;  // bit k: a non-core in chunk k
#pragma unroll
    for (int k = 0; k < W; ++k) {
      const uint32_t j = j0 + 32 * k + lane;
      x[k] = j < e ? ids[j] : -1;
    }
#pragma unroll
    for (int k = 0; k < W; ++k)
      if (x[k] >= 0 && ld_volatile(c.parent + x[k]) < 0) some |= 1u << k;
    unsigned any = __reduce_or_sync(0xffffffffu, some);
    while (any) {
      const int k = __ffs(any) - 1;
      any &= any - 1;
      border_chunk(a, c, some >> k & 1u ? ids[j0 + 32 * k + lane] : -1);
    }
  }
}

template <bool ONE>
__device__ __forceinline__ void phase_borders(const QArgs& a, int64_t total, int mu, double eps,
                                              int64_t w0, int64_t nw) {
  // the pieces queued for the unions are the ones of this phase too, unless
  // the queue was full: then every warp walks its whole prefixes
  const int64_t asked = a.queue ? (int64_t)*a.queued : 0;
  const bool queued = asked <= (int64_t)a.queue_cap;
  for (int64_t it = w0; it < total; it += nw) {
    const Item x = item_at<ONE>(a, it, mu, eps);
    int64_t pu = prefix_ge(a.no_sim + a.off[x.u], a.deg[x.u], x.eps);
    if (a.queue && queued) pu = min(pu, (int64_t)PIECE);
    border_range(a, x, 0, (uint32_t)pu);
  }
  if (a.queue && queued)
    for (int64_t i = w0; i < asked; i += nw) {
      const QPiece p = a.queue[i];
      const Item x{p.q, p.u, ONE ? eps : a.eps[p.q], a.parent + (int64_t)p.q * a.n,
                   ONE ? a.labels : labels_of(a, p.q)};
      border_range(a, x, p.begin, p.end);
    }
}

// warp per unclustered vertex
__device__ __forceinline__ void phase_hubs(const QArgs& a, int32_t* lab, int64_t w0, int64_t nw) {
  const int lane = threadIdx.x & 31;
  for (int64_t v = w0; v < a.n; v += nw) {
    if (ld_volatile(lab + v) != -1) continue;
    const int64_t rb = a.off[v], re = rb + a.deg[v];
    int32_t first = -1;
    bool hub = false;
    for (int64_t j0 = rb; j0 < re && !hub; j0 += 32) {
      const int64_t j = j0 + lane;
      int32_t l = -1;
      if (j < re) l = lab[a.adj[j]];
      if (l == -2) l = -1;  // hub marks are written in this pass; they are not clusters
      // first clustered label in this chunk
      const unsigned m = __ballot_sync(0xffffffffu, l >= 0);
      if (!m) continue;
      if (first < 0) first = __shfl_sync(0xffffffffu, l, __ffs(m) - 1);
      hub = __any_sync(0xffffffffu, l >= 0 && l != first);
    }
    if (hub && lane == 0) lab[v] = -2;
  }
}

__device__ __forceinline__ int64_t grid_thread() {
  return (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
}
__device__ __forceinline__ int64_t grid_threads() { return (int64_t)gridDim.x * blockDim.x; }

// The batch's phases, one launch each.
__global__ void k_mark_cores(QArgs a) {
  phase_mark<false>(a, a.ncp[a.Q], 0, 0.0, grid_thread(), grid_threads());
}
__global__ void __launch_bounds__(256, 8) k_union(QArgs a) {
  phase_union<false>(a, a.ncp[a.Q], 0, 0.0, grid_thread() >> 5, grid_threads() >> 5);
}
__global__ void k_union_queue(QArgs a) {
  phase_union_queue(a, grid_thread() >> 5, grid_threads() >> 5);
}
// Borders do not read core labels, only parents. Six CTAs a multiprocessor: the
// walks wait for dependent loads, and the registers spilled for it are those of
// the few borders (a ring of 1M vertices, all of them cores: four CTAs 1.12 ms,
// five 1.15, six 1.07).
__global__ void __launch_bounds__(256, 6) k_labels(QArgs a) {
  const int64_t total = a.ncp[a.Q];
  phase_core_labels<false>(a, total, 0, 0.0, grid_thread(), grid_threads());
  phase_borders<false>(a, total, 0, 0.0, grid_thread() >> 5, grid_threads() >> 5);
}
__global__ void k_hubs(QArgs a) {
  if (a.ncp[blockIdx.y + 1] == a.ncp[blockIdx.y]) return;  // no clusters, no hubs
  const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  phase_hubs(a, labels_of(a, blockIdx.y), w0, ((int64_t)gridDim.x * blockDim.x) >> 5);
}

// -1 in p[0..n), as 16-byte stores between the first and last 16-byte boundary
__device__ __forceinline__ void fill_minus1(int32_t* p, int64_t n, int64_t t0, int64_t nt) {
  const int64_t head = min(n, (int64_t)(((16 - ((uintptr_t)p & 15)) & 15) / 4));
  const int64_t vec = (n - head) / 4;
  int4* p4 = reinterpret_cast<int4*>(p + head);
  for (int64_t i = t0; i < vec; i += nt) p4[i] = make_int4(-1, -1, -1, -1);
  for (int64_t i = t0; i < head; i += nt) p[i] = -1;
  for (int64_t i = head + 4 * vec + t0; i < n; i += nt) p[i] = -1;
}

// One query as one cooperative launch: the same phases between grid barriers,
// (mu, eps) as arguments, the status in a word that the host reads directly.
// Every CTA searches the core count for itself (it is one cached path). A query
// of more than `most` cores is left to the batch's launches, and hubs of a large
// graph to k_hubs: one kernel for all phases has the registers of the largest, so
// half as many warps walk the rows (ring of 1M vertices, each a core: 1.95 ms
// here, 1.07 as a batch of one).
constexpr int ONE_T = 256;
constexpr unsigned ONE_HEAVY = 1u << 31;  // in the status word: nothing was labelled
__global__ void __launch_bounds__(ONE_T, 4)
k_query_one(QArgs a, int mu, double eps, int hubs, int64_t most) {
  cooperative_groups::grid_group grid = cooperative_groups::this_grid();
  __shared__ int64_t s_nc;
  const int64_t t0 = grid_thread(), nt = grid_threads();
  if (t0 == 0) *a.queued = 0;
  fill_minus1(a.parent, a.n, t0, nt);
  fill_minus1(a.labels, a.n, t0, nt);
  if (threadIdx.x < 32) {
    const int64_t c = count_cores(a, mu, eps);
    if (threadIdx.x == 0) s_nc = c;
  }
  __syncthreads();
  const int64_t nc = s_nc;  // the same in every CTA
  if (t0 == 0) {
    a.ncp[0] = 0;
    a.ncp[1] = nc > most ? 0 : nc;
    if (nc > most) *a.status = ONE_HEAVY;
  }
  if (nc == 0 || nc > most) return;
  grid.sync();
  phase_mark<true>(a, nc, mu, eps, t0, nt);
  grid.sync();
  phase_union<true>(a, nc, mu, eps, t0 >> 5, nt >> 5);
  grid.sync();
  if (a.queue && *a.queued) {  // the same in every CTA: nothing adds to it any more
    phase_union_queue(a, t0 >> 5, nt >> 5);
    grid.sync();
  }
  phase_core_labels<true>(a, nc, mu, eps, t0, nt);
  phase_borders<true>(a, nc, mu, eps, t0 >> 5, nt >> 5);
  if (!hubs) return;
  grid.sync();
  phase_hubs(a, a.labels, t0 >> 5, nt >> 5);
}

// Resident CTAs of k_query_one per multiprocessor (0: no cooperative launch).
int query_one_per_sm() {
  static std::atomic<int> cached[64];  // 1 + the value, zero until looked up
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int c = cached[dev].load(std::memory_order_relaxed);
  if (c == 0) {
    int coop = 0, per = 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_query_one, ONE_T, 0) != cudaSuccess) {
      cudaGetLastError();
      per = 0;
    }
    c = 1 + (per < 4 ? per : 4);
    cached[dev].store(c, std::memory_order_relaxed);
  }
  return c - 1;
}

// Where a single query leaves the cooperative launch: where it is expected to
// take ONE_LOSS us longer than the launches of a batch, which cost 45 us more,
// and 20 us for the attempt. Measured, always one launch, always a batch, and by
// this rule, us: ring of 1M vertices 1900, 1067, 1090, of 300k 555, 367, 385, of
// 100k 230, 213, 228; 100 cliques of 600 547, 456, 490; SBM of 100k vertices (2, 0)
// 500, 690, 500.
constexpr double ONE_LOSS = 150.0;
constexpr int64_t ONE_HUBS = 8;         // vertices per resident warp: hubs in a launch of their own
                                        // beyond (R-MAT s22 (3, 0.3) 1686 -> 1092 us)
constexpr int64_t ONE_COPY = 1 << 16;   // labels

dim3 hubs_grid(int64_t n, int Q) {
  return dim3((unsigned)std::max<int64_t>(
                  1, std::min<int64_t>((n + 7) / 8, sm_count() * 16 / std::min(Q, 16) + 1)), Q);
}

unsigned queue_capacity(const IndexData& ix, int Q) {
  // pieces past the first of a row: none when no row is longer than one
  if (ix.maxdeg <= PIECE) return 0;
  const int64_t all = (int64_t)Q * (ix.arcs / PIECE + 1);
  return (unsigned)std::min<int64_t>(all, QUERY_QUEUE_MAX);
}

}  // namespace

// Launch sequence of a batch of Q queries; every pointer is device memory.
int launch_query_batch(const IndexData& ix, int Q, const int* mu, const double* eps, int64_t* nc,
                       int32_t* parent, int32_t* labels, int32_t* const* lab_ptrs, int flags,
                       cudaStream_t s, unsigned* status_dev, void* queue, size_t queue_bytes,
                       unsigned long long* reached) {
  const int64_t n = ix.n;
  GS_CUDA(cudaMemsetAsync(parent, 0xff, sizeof(int32_t) * (size_t)Q * n, s));
  // queue: a 16-byte head with the count, then the pieces
  const unsigned cap = queue && queue_bytes > 16 && ix.maxdeg > PIECE
      ? (unsigned)std::min<size_t>((queue_bytes - 16) / sizeof(QPiece), QUERY_QUEUE_MAX) : 0;
  QArgs a{ix.off, ix.deg, ix.adj, ix.no_id, ix.no_sim, ix.co_off, ix.co_id, ix.co_thr,
          n, ix.maxdeg, mu, eps, nc, Q, parent, labels, lab_ptrs, status_dev,
          cap ? reinterpret_cast<QPiece*>((char*)queue + 16) : nullptr,
          reinterpret_cast<unsigned long long*>(queue), cap, reached};
  if (cap) GS_CUDA(cudaMemsetAsync(queue, 0, 16, s));
  const unsigned gx = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, sm_count() * 8 / std::min(Q, 8) + 1));
  if (lab_ptrs) {
    k_init_labels<<<dim3(gx, Q), 256, 0, s>>>(a);
    GS_LAUNCH();
  } else {
    GS_CUDA(cudaMemsetAsync(labels, 0xff, sizeof(int32_t) * (size_t)Q * n, s));
  }
  k_get_cores<<<(Q + 3) / 4, 128, 0, s>>>(a);
  GS_LAUNCH();
  k_core_prefix<<<1, PREFIX_T, 0, s>>>(a);
  GS_LAUNCH();
  // the (query, core) items of the whole batch share one grid
  k_mark_cores<<<sm_count() * 8, 256, 0, s>>>(a);
  GS_LAUNCH();
  k_union<<<sm_count() * 16, 256, 0, s>>>(a);
  GS_LAUNCH();
  if (cap) {
    k_union_queue<<<sm_count() * 16, 256, 0, s>>>(a);
    GS_LAUNCH();
  }
  k_labels<<<sm_count() * 16, 256, 0, s>>>(a);
  GS_LAUNCH();
  if (flags & SCAN_Q_HUBS) {
    k_hubs<<<hubs_grid(n, Q), 256, 0, s>>>(a);
    GS_LAUNCH();
  }
  return SCAN_OK;
}

size_t query_queue_bytes(const IndexData& ix, int Q) {
  const unsigned cap = queue_capacity(ix, Q);
  return cap ? 16 + (size_t)cap * sizeof(QPiece) : 0;
}

int run_query_one(const IndexData& ix, int mu, double eps, int32_t* labels, int32_t* host_labels,
                  int flags, Pool& pool, cudaStream_t s, bool* done) {
  *done = false;
  const int64_t n = ix.n;
  const int per_sm = query_one_per_sm();
  PinnedSlot slot;  // the kernel's status word
  unsigned* status = static_cast<unsigned*>(slot.p);
  if (per_sm == 0 || !status) return SCAN_OK;
  *status = 0;
  // parents, the counts of queued pieces and of cores, pieces; without pieces
  // where there is no room for them
  const size_t count_at = ((size_t)n * sizeof(int32_t) + 7) & ~(size_t)7;
  const size_t head = count_at + 3 * sizeof(int64_t);
  unsigned cap = queue_capacity(ix, 1);
  char* scratch = cap ? pool.get<char>(head + (size_t)cap * sizeof(QPiece)) : nullptr;
  if (!scratch) {
    cap = 0;
    scratch = pool.get<char>(head);
  }
  if (!scratch) return SCAN_ENOMEM;
  int32_t* parent = reinterpret_cast<int32_t*>(scratch);
  unsigned long long* queued = reinterpret_cast<unsigned long long*>(scratch + count_at);
  int64_t* nc = reinterpret_cast<int64_t*>(scratch + count_at) + 1;
  QArgs a{ix.off, ix.deg, ix.adj, ix.no_id, ix.no_sim, ix.co_off, ix.co_id, ix.co_thr,
          n, ix.maxdeg, nullptr, nullptr, nc, 1, parent, labels, nullptr, status,
          cap ? reinterpret_cast<QPiece*>(scratch + head) : nullptr, queued, cap, nullptr};
  // a warp per core at most, and no more CTAs than are resident at once
  const int64_t want = std::max<int64_t>(1, (n + ONE_T / 32 - 1) / (ONE_T / 32));
  const int64_t resident = (int64_t)sm_count() * per_sm;
  const unsigned g = (unsigned)std::min<int64_t>(want, resident);
  const int64_t warps = resident * (ONE_T / 32);
  // the most cores: an item costs a warp here about 2.5 us and 1.5 us per 32
  // entries of its row more than in the batch's launches
  const double steps = (double)ix.arcs / (double)n / 32.0;
  int64_t most = (int64_t)(ONE_LOSS * (double)warps / (2.5 + 1.5 * steps));
  const bool hubs = flags & SCAN_Q_HUBS, hubs_after = hubs && n > ONE_HUBS * warps;
  int hubs_in = hubs && !hubs_after;
  void* args[] = {&a, &mu, &eps, &hubs_in, &most};
  // refused where the stream or the process has fewer multiprocessors than
  // the device: the launches of a batch answer then
  if (cudaLaunchCooperativeKernel((const void*)k_query_one, dim3(g), dim3(ONE_T), args, 0, s) !=
      cudaSuccess) {
    cudaGetLastError();
    pool.put(scratch);
    return SCAN_OK;
  }
  GS_LAUNCH();
  if (hubs_after) {
    k_hubs<<<hubs_grid(n, 1), 256, 0, s>>>(a);
    GS_LAUNCH();
  }
  // labels for the host follow at once where they are few
  const bool copy_now = host_labels && n <= ONE_COPY;
  auto copy = [&] {
    return cudaMemcpyAsync(host_labels, labels, (size_t)n * sizeof(int32_t),
                           cudaMemcpyDeviceToHost, s);
  };
  if (copy_now) GS_CUDA(copy());
  GS_CUDA(cudaStreamSynchronize(s));
  const unsigned st = *(volatile unsigned*)status;
  if (st & ONE_HEAVY) {
    pool.put(scratch);
    return SCAN_OK;
  }
  *done = true;
  if (host_labels && !copy_now) {
    GS_CUDA(copy());
    GS_CUDA(cudaStreamSynchronize(s));
  }
  if (st & DEV_LIMIT) return SCAN_ETIMEOUT;
  return SCAN_OK;
}

int run_queries(const IndexData& ix, int Q, const int* mu_host, const double* eps_host,
                int32_t* labels_dev, int flags, Pool& pool, cudaStream_t s, unsigned* status_dev,
                unsigned long long* reached_dev) {
  if (Q <= 0) return SCAN_OK;
  const int64_t n = ix.n;
  int* mu = pool.get<int>(Q);
  double* eps = pool.get<double>(Q);
  int64_t* nc = pool.get<int64_t>((size_t)Q + 1);
  int32_t* parent = pool.get<int32_t>((size_t)Q * (size_t)(n > 0 ? n : 1));
  if (!mu || !eps || !nc || !parent) {
    pool.put(mu);
    pool.put(eps);
    pool.put(nc);
    pool.put(parent);
    return SCAN_ENOMEM;
  }
  size_t qb = query_queue_bytes(ix, Q);
  char* queue = qb ? pool.get<char>(qb) : nullptr;
  if (!queue) qb = 0;  // no room: a warp walks a long row alone
  GS_CUDA(cudaMemcpyAsync(mu, mu_host, sizeof(int) * Q, cudaMemcpyHostToDevice, s));
  GS_CUDA(cudaMemcpyAsync(eps, eps_host, sizeof(double) * Q, cudaMemcpyHostToDevice, s));
  if (n == 0) return SCAN_OK;
  GS_TRY(launch_query_batch(ix, Q, mu, eps, nc, parent, labels_dev, nullptr, flags, s, status_dev,
                            queue, qb, reached_dev));
  pool.put(mu);
  pool.put(eps);
  pool.put(nc);
  pool.put(parent);
  if (queue) pool.put(queue);
  return SCAN_OK;
}

// The same launches as run_queries with every scratch array supplied by the
// caller (mu, eps, core counts and parents already in device memory); used by
// the entry point that must not allocate.
int run_queries_prealloc(const IndexData& ix, int Q, const int* mu_dev, const double* eps_dev,
                         int64_t* nc_dev, int32_t* parent, int32_t* labels_dev, int flags,
                         cudaStream_t s, unsigned* status_dev) {
  if (Q <= 0 || ix.n == 0) return SCAN_OK;
  return launch_query_batch(ix, Q, mu_dev, eps_dev, nc_dev, parent, labels_dev, nullptr, flags, s,
                            status_dev, nullptr, 0);
}

}  // namespace gscan
