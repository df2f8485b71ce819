// Graph preparation: device-wide scans, degrees with CSR checks, and the
// degree orientation of Section 6.1 (every edge directed towards its endpoint
// of larger (degree, id)).
#include "scan_internal.cuh"

namespace gscan {

namespace {

constexpr int SCAN_T = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_T * SCAN_ITEMS;

template <class T>
__device__ __forceinline__ int64_t load_val(const T* in, int64_t i, int64_t n) {
  return i < n ? (int64_t)in[i] : 0;
}

// Block-wide exclusive scan of one int64 per thread; returns the block total.
__device__ int64_t block_exclusive_scan(int64_t v, int64_t* out_excl) {
  __shared__ int64_t warp_tot[SCAN_T / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int64_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[wid] = x;
  __syncthreads();
  if (wid == 0) {
    int64_t w = lane < SCAN_T / 32 ? warp_tot[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int64_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < SCAN_T / 32) warp_tot[lane] = w;  // inclusive
  }
  __syncthreads();
  const int64_t before_warp = wid ? warp_tot[wid - 1] : 0;
  const int64_t total = warp_tot[SCAN_T / 32 - 1];
  *out_excl = before_warp + x - v;
  __syncthreads();
  return total;
}

template <class T>
__global__ void k_tile_sums(const T* in, int64_t n, int64_t* sums) {
  const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
  int64_t s = 0;
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k) s += load_val(in, base + k, n);
  int64_t ex;
  int64_t tot = block_exclusive_scan(s, &ex);
  if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

// out has n+1 entries; tile_base[b] is the exclusive prefix of tile b.
template <class T>
__global__ void k_tile_scan(const T* in, int64_t n, const int64_t* tile_base, int64_t* out) {
  const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
  int64_t v[SCAN_ITEMS];
  int64_t s = 0;
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k) { v[k] = load_val(in, base + k, n); s += v[k]; }
  int64_t ex;
  block_exclusive_scan(s, &ex);
  int64_t run = ex + (tile_base ? tile_base[blockIdx.x] : 0);
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k) {
    const int64_t i = base + k;
    if (i <= n) out[i] = run;
    run += v[k];
  }
}

template <class T>
int scan_impl(const T* in, int64_t* out, int64_t n, Pool& pool, cudaStream_t s) {
  // tiles cover indices 0..n (n+1 outputs)
  const int64_t tiles = (n + 1 + SCAN_TILE - 1) / SCAN_TILE;
  if (tiles == 1) {
    k_tile_scan<T><<<1, SCAN_T, 0, s>>>(in, n, nullptr, out);
    GS_LAUNCH();
    return SCAN_OK;
  }
  int64_t* sums = pool.tmp<int64_t>(tiles);
  int64_t* base = pool.tmp<int64_t>(tiles + 1);
  if (!sums || !base) return SCAN_ENOMEM;
  k_tile_sums<T><<<(unsigned)tiles, SCAN_T, 0, s>>>(in, n, sums);
  GS_LAUNCH();
  GS_TRY(scan_impl<int64_t>(sums, base, tiles, pool, s));
  k_tile_scan<T><<<(unsigned)tiles, SCAN_T, 0, s>>>(in, n, base, out);
  GS_LAUNCH();
  pool.put(sums);
  pool.put(base);
  return SCAN_OK;
}

// Degrees and CSR checks, 32 rows per warp (RowGroup). Rows longer than
// DEG_LONG are listed for k_degrees_long and left out (one warp would walk
// a hub's row alone, one dependent load at a time). A group with a bad row
// bound is not walked. The list has max_long = arcs / DEG_LONG + 1 places,
// enough for offsets that do not descend; more long rows than that prove the
// offsets bad (0, arcs, 0, arcs, ... makes every other row a long one), and
// what does not fit is not listed.
constexpr int DEG_LONG = 4096;

__global__ void __launch_bounds__(256)
k_degrees(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
          int64_t n, int64_t arcs, int32_t* __restrict__ deg, int32_t* maxdeg,
          unsigned* status, int32_t* __restrict__ long_rows,
          unsigned* __restrict__ n_long, unsigned max_long) {
  constexpr unsigned FULL = 0xffffffffu;
  __shared__ int scratch[8][64];
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int32_t local_max = 0;
  unsigned bad = warp == 0 && (off[0] != 0 || off[n] != arcs) ? 1 : 0;
  for (int64_t v0 = warp * 32; v0 < n; v0 += nwarps * 32) {
    const int64_t v = v0 + lane;
    int64_t b = 0, e = 0;
    if (v < n) { b = off[v]; e = off[v + 1]; }
    // rows must lie inside [0, arcs] before adj is touched
    const bool row_bad = b < 0 || e > arcs || e - b < 0 || e - b > 0x7fffffff;
    const bool is_long = !row_bad && e - b > DEG_LONG;
    if (v < n) {
      deg[v] = row_bad ? 0 : (int32_t)(e - b);
      if (!row_bad) local_max = max(local_max, (int32_t)(e - b));
      if (is_long) {
        const unsigned at = atomicAdd(n_long, 1u);
        if (at < max_long) long_rows[at] = (int32_t)v; else bad = 1;
      }
    }
    if (__any_sync(FULL, row_bad)) {
      bad = 1;
      continue;
    }
    RowGroup g;
    g.init(is_long ? 0 : (int)(e - b), scratch[threadIdx.x >> 5]);
    // element of a virtual position: adj[base of its row + position]
    const int64_t base = __shfl_sync(FULL, b, g.row) - g.vs;
    int32_t carry = 0;  // the element before the chunk
    for (int i0 = 0; i0 < g.total; i0 += 32) {
      const int k = g.chunk(i0);
      const int i = i0 + lane;
      const int64_t bk = __shfl_sync(FULL, base, k);
      const int32_t own = (int32_t)v0 + __shfl_sync(FULL, g.row, k);
      const bool act = i < g.total;
      const int32_t x = act ? adj[bk + i] : 0;
      int32_t prev = __shfl_up_sync(FULL, x, 1);
      if (lane == 0) prev = carry;
      carry = __shfl_sync(FULL, x, 31);
      if (act) {
        if (x < 0 || x >= n || x == own) bad = 1;
        // strictly ascending inside a row: sorted, no duplicates
        if (!(g.starts >> lane & 1u) && prev >= x) bad = 1;
      }
    }
  }
  for (int o = 16; o; o >>= 1) local_max = max(local_max, __shfl_xor_sync(FULL, local_max, o));
  bad = __any_sync(FULL, bad);
  if (lane == 0) {
    if (local_max) atomicMax(maxdeg, local_max);
    if (bad) atomicOr(status, (unsigned)DEV_BADGRAPH);
  }
}

// The CSR checks of the listed long rows, one CTA per row.
__global__ void __launch_bounds__(1024)
k_degrees_long(const int64_t* __restrict__ off, const int32_t* __restrict__ adj, int64_t n,
               const int32_t* __restrict__ long_rows, const unsigned* __restrict__ n_long,
               unsigned max_long, unsigned* status) {
  const unsigned cnt = min(*n_long, max_long);
  unsigned bad = 0;
  for (unsigned r = blockIdx.x; r < cnt; r += gridDim.x) {
    const int32_t v = long_rows[r];
    const int64_t b = off[v], e = off[v + 1];
    for (int64_t i = b + threadIdx.x; i < e; i += blockDim.x) {
      const int32_t x = adj[i];
      if (x < 0 || x >= n || x == v) bad = 1;
      if (i > b && adj[i - 1] >= x) bad = 1;
    }
  }
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(status, (unsigned)DEV_BADGRAPH);
}

__device__ __forceinline__ bool lower(int32_t du, int32_t u, int32_t dv, int32_t v) {
  return du < dv || (du == dv && u < v);
}

// Orientation in place: the out-arcs of v (neighbours of larger (degree, id))
// are compacted, in id order, to the front of v's own CSR slot range, so
// out(v) = oadj[off[v] .. off[v] + od[v]) needs no separate offsets; the
// in-arcs fill the row from its end; opos holds each arc's position in the
// row. 32 rows per warp (RowGroup): lane k keeps the out-arcs placed so far
// of the k-th non-empty row, and a position finds its place by ballots masked
// to its row's lower lanes; the in-arcs before it are the other positions
// before it. Rows longer than LONG_ROW are listed in long_rows for
// k_orient_long and left out.
constexpr int LONG_ROW = 4096;
constexpr int LONG_T = 1024;

__global__ void __launch_bounds__(256)
k_orient_inplace(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
                 const int32_t* __restrict__ deg, int64_t n,
                 int32_t* __restrict__ od, int32_t* __restrict__ oadj,
                 int32_t* __restrict__ opos, int32_t* max_od,
                 unsigned long long* sum_od, int32_t* __restrict__ long_rows,
                 unsigned* __restrict__ n_long, const unsigned* __restrict__ status) {
  constexpr unsigned FULL = 0xffffffffu;
  __shared__ int scratch[8][64];
  if (*status & DEV_BADGRAPH) return;  // ids may be out of range
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;  // lanes below this one
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  unsigned long long local_sum = 0;
  int32_t local_max = 0;
  for (int64_t v0 = warp * 32; v0 < n; v0 += nwarps * 32) {
    const int64_t v = v0 + lane;
    int64_t b = 0;
    int32_t d = 0;
    if (v < n) { b = off[v]; d = deg[v]; }
    const bool is_long = d > LONG_ROW;
    if (is_long) long_rows[atomicAdd(n_long, 1u)] = (int32_t)v;
    if (v < n && d == 0) od[v] = 0;
    RowGroup g;
    g.init(is_long ? 0 : d, scratch[threadIdx.x >> 5]);
    const int64_t start = __shfl_sync(FULL, b, g.row);  // of lane's compacted row
    int32_t w = 0;                                      // its out-arcs placed so far
    for (int i0 = 0; i0 < g.total; i0 += 32) {
      const int k = g.chunk(i0);
      const int i = i0 + lane;
      const int64_t rb = __shfl_sync(FULL, start, k);
      const int vsk = __shfl_sync(FULL, g.vs, k), vek = __shfl_sync(FULL, g.ve, k);
      const int wk = __shfl_sync(FULL, w, k);
      const int32_t own = (int32_t)v0 + __shfl_sync(FULL, g.row, k);
      const bool act = i < g.total;
      const int p = i - vsk;  // position in the row
      int32_t x = 0;
      bool up = false;
      if (act) { x = adj[rb + p]; up = lower(vek - vsk, own, deg[x], x); }
      const unsigned m = __ballot_sync(FULL, up);
      // out-arcs of the row before this position: placed ones and lower lanes
      // from the row's first position in the chunk on
      const unsigned st = g.starts & (lt | (lt + 1u));
      const unsigned from = st ? ~((1u << (31 - __clz(st))) - 1u) : FULL;
      const int ups = wk + __popc(m & lt & from);
      if (act) {
        const int64_t dst = up ? rb + ups : rb + (vek - vsk) - 1 - (p - ups);
        oadj[dst] = x;
        opos[dst] = p;
      }
      // each row's owner lane adds its row's out-arcs of this chunk
      const int mlo = max(0, g.vs - i0), mhi = min(32, g.ve - i0);
      if (lane < g.cnt && mlo < mhi)
        w += __popc(m & (FULL >> (32 - mhi)) & (FULL << mlo));
    }
    if (lane < g.cnt) {
      od[v0 + g.row] = w;
      local_sum += (unsigned long long)w;
      local_max = max(local_max, w);
    }
  }
  for (int o = 16; o; o >>= 1) {
    local_sum += __shfl_xor_sync(FULL, local_sum, o);
    local_max = max(local_max, __shfl_xor_sync(FULL, local_max, o));
  }
  if (lane == 0) {
    if (local_sum) atomicAdd(sum_od, local_sum);
    if (local_max) atomicMax(max_od, local_max);
  }
}

// One CTA per listed long row: chunks of LONG_T positions, the out-arcs of a
// chunk placed by a block-wide prefix count (ballots, then a scan of the 32
// warp counts), so the out-list stays in id order; the in-arcs fill the rest
// of the row from its end.
__global__ void __launch_bounds__(LONG_T)
k_orient_long(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
              const int32_t* __restrict__ deg, const int32_t* __restrict__ long_rows,
              const unsigned* __restrict__ n_long, int32_t* __restrict__ od,
              int32_t* __restrict__ oadj, int32_t* __restrict__ opos, int32_t* max_od,
              unsigned long long* sum_od) {
  __shared__ int s_cnt[LONG_T / 32];
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const unsigned cnt = *n_long;
  for (unsigned r = blockIdx.x; r < cnt; r += gridDim.x) {
    const int32_t v = long_rows[r];
    const int64_t b = off[v], e = off[v + 1];
    const int32_t dv = deg[v];
    int64_t w = b, wi = 0;  // out-arcs placed from the front, in-arcs from the back
    for (int64_t i0 = b; i0 < e; i0 += LONG_T) {
      const int64_t i = i0 + t;
      bool up = false;
      int32_t x = 0;
      if (i < e) { x = adj[i]; up = lower(dv, v, deg[x], x); }
      const unsigned m = __ballot_sync(0xffffffffu, up);
      if (lane == 0) s_cnt[wid] = __popc(m);
      __syncthreads();
      // warp prefix over the 32 warp counts, computed by every warp
      int c = s_cnt[lane];
      int incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const int before = __shfl_sync(0xffffffffu, incl - c, wid);
      const int total = __shfl_sync(0xffffffffu, incl, 31);
      const int up_before = before + __popc(m & ((1u << lane) - 1u));
      if (up) {
        const int64_t dst = w + up_before;
        oadj[dst] = x;
        opos[dst] = (int32_t)(i - b);
      } else if (i < e) {
        const int64_t dst = e - 1 - (wi + (t - up_before));
        oadj[dst] = x;
        opos[dst] = (int32_t)(i - b);
      }
      w += total;
      wi += min((int64_t)LONG_T, e - i0) - total;
      __syncthreads();  // s_cnt is rewritten by the next chunk
    }
    if (t == 0) {
      od[v] = (int32_t)(w - b);
      atomicAdd(sum_od, (unsigned long long)(w - b));
      atomicMax(max_od, (int32_t)(w - b));
    }
  }
}

inline unsigned grid_for(int64_t work, int per_block, int cap = sm_count() * 32) {
  int64_t g = (work + per_block - 1) / per_block;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (unsigned)g;
}

}  // namespace

int exclusive_scan_i64(const int64_t* in, int64_t* out, int64_t n, Pool& pool, cudaStream_t s) {
  return scan_impl<int64_t>(in, out, n, pool, s);
}

int exclusive_scan_i32_to_i64(const int32_t* in, int64_t* out, int64_t n, Pool& pool,
                              cudaStream_t s) {
  return scan_impl<int32_t>(in, out, n, pool, s);
}

int launch_degrees(const int64_t* off, const int32_t* adj, int64_t n, int64_t arcs, int32_t* deg,
                   int32_t* maxdeg_dev, unsigned* status, Pool& pool, cudaStream_t s) {
  if (n == 0) return SCAN_OK;
  const int64_t max_long = arcs / DEG_LONG + 1;
  int32_t* long_rows = pool.tmp<int32_t>(max_long);
  unsigned* n_long = pool.tmp<unsigned>(1);
  if (!long_rows || !n_long) return SCAN_ENOMEM;
  GS_CUDA(cudaMemsetAsync(n_long, 0, sizeof(unsigned), s));
  k_degrees<<<grid_for(n, 256), 256, 0, s>>>(off, adj, n, arcs, deg, maxdeg_dev, status, long_rows,
                                             n_long, (unsigned)max_long);
  GS_LAUNCH();
  k_degrees_long<<<(unsigned)std::min<int64_t>(max_long, sm_count() * 2), 1024, 0, s>>>(
      off, adj, n, long_rows, n_long, (unsigned)max_long, status);
  GS_LAUNCH();
  pool.put(long_rows);
  pool.put(n_long);
  return SCAN_OK;
}

int launch_orient(const int64_t* off, const int32_t* adj, const int32_t* deg, int64_t n,
                  int64_t arcs, Pool& pool, int32_t** od_out, int32_t** oadj_out,
                  int32_t** opos_out, int32_t* max_od_dev, unsigned long long* sum_od_dev,
                  const unsigned* status, cudaStream_t s) {
  int32_t* od = pool.tmp<int32_t>(n > 0 ? n : 1);
  int32_t* oadj = pool.tmp<int32_t>(arcs > 0 ? arcs : 1);
  int32_t* opos = pool.tmp<int32_t>(arcs > 0 ? arcs : 1);
  // rows longer than LONG_ROW: at most arcs / LONG_ROW of them (the degree
  // pass has refused offsets that descend, and k_orient_inplace lists nothing
  // then)
  const int64_t max_long = arcs / LONG_ROW + 1;
  int32_t* long_rows = pool.tmp<int32_t>(max_long);
  unsigned* n_long = pool.tmp<unsigned>(1);
  if (!od || !oadj || !opos || !long_rows || !n_long) return SCAN_ENOMEM;
  if (n > 0) {
    GS_CUDA(cudaMemsetAsync(n_long, 0, sizeof(unsigned), s));
    k_orient_inplace<<<grid_for(n, 256), 256, 0, s>>>(off, adj, deg, n, od, oadj, opos, max_od_dev,
                                                    sum_od_dev, long_rows, n_long, status);
    GS_LAUNCH();
    k_orient_long<<<(unsigned)std::min<int64_t>(max_long, sm_count() * 2), LONG_T, 0, s>>>(
        off, adj, deg, long_rows, n_long, od, oadj, opos, max_od_dev, sum_od_dev);
    GS_LAUNCH();
  }
  pool.put(long_rows);
  pool.put(n_long);
  *od_out = od;
  *oadj_out = oadj;
  *opos_out = opos;
  return SCAN_OK;
}

}  // namespace gscan
