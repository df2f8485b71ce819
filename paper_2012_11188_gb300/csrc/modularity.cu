// Modularity of a clustering (Section 7.2) and the (mu, eps) sweep that
// selects the clustering of highest modularity (Section 7.3.4, over the
// parameter set Sigma: mu in {2, 4, ..., 2^18}, eps in {.01, ..., .99}).
//
// With unclustered vertices as singletons, the modularity of a clustering is
//   Q = I / 2m - (S_c + S_u) / (2m)^2,
// where I counts the arcs (u,v) with u, v in the same cluster, S_c sums
// D_c^2 over the clusters c, D_c being the sum of the degrees in c, and S_u
// sums d_v^2 over the unclustered vertices. All three are integers, summed
// exactly in 64 bits; only the last line is floating point. S_u is the sum
// of d^2 over all vertices (fixed per graph) minus that over the clustered
// ones, so a pass touches the rows of the clustered vertices only.
#include "scan_internal.cuh"

namespace gscan {

namespace {

// Per clustering: acc[0] = I, acc[1] = sum of d^2 over clustered vertices,
// acc[2] = S_c, acc[3] != 0 if a label was not a vertex id. dsum[c] (zero on
// entry and on exit) accumulates D_c at the cluster's label c. MANY: clustering
// blockIdx.y of several, rows of n labels and sums, four words of acc each;
// nothing is done where reached is `most` or more, what lies inside a row of more
// than `longest` is left to k_mod_long, and runs of one label are one addition.
template <bool MANY>
__global__ void k_mod_rows(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
                           const int32_t* __restrict__ labels, int64_t n,
                           unsigned long long* __restrict__ dsum,
                           unsigned long long* __restrict__ acc, const unsigned long long* reached,
                           unsigned long long most, int64_t longest) {
  if (MANY) {
    if (*reached >= most) return;
    labels += (int64_t)blockIdx.y * n;
    dsum += (int64_t)blockIdx.y * n;
    acc += 4 * blockIdx.y;
  }
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  unsigned long long inside = 0, dsq = 0, run = 0;  // run: of vertices with run_label
  int32_t run_label = -1;
  bool bad = false;
  for (int64_t v0 = warp * 32; v0 < n; v0 += nwarps * 32) {
    // 32 vertices per step: one label load per lane, then the clustered rows
    const int64_t vl = v0 + lane;
    int32_t ll = vl < n ? labels[vl] : -1;
    if (ll >= n) { bad = true; ll = -1; }
    unsigned todo = __ballot_sync(0xffffffffu, ll >= 0);
    while (todo) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      const int64_t v = v0 + src;
      const int32_t lv = __shfl_sync(0xffffffffu, ll, src);
      const int64_t b = off[v], e = off[v + 1];
      unsigned cnt = 0;
      const int64_t to = MANY && e - b > longest ? b : e;
      for (int64_t i = b + lane; i < to; i += 32) cnt += labels[adj[i]] == lv ? 1u : 0u;
      cnt = __reduce_add_sync(0xffffffffu, cnt);
      if (lane == 0) {
        const unsigned long long d = (unsigned long long)(e - b);
        inside += cnt;
        dsq += d * d;
        if (!MANY) {
          if (d) atomicAdd(&dsum[lv], d);
        } else {
          if (lv != run_label) {
            if (run) atomicAdd(&dsum[run_label], run);
            run_label = lv;
            run = 0;
          }
          run += d;
        }
      }
    }
  }
  if (lane == 0) {
    if (MANY && run) atomicAdd(&dsum[run_label], run);
    if (inside) atomicAdd(&acc[0], inside);
    if (dsq) atomicAdd(&acc[1], dsq);
  }
  if (bad) atomicOr(&acc[3], 1ull);
}

// The arcs inside the rows of more than MOD_LONG entries (CO[MOD_LONG + 2] lists
// them) of clustering blockIdx.y: a CTA per row, all CTAs on a row of more than
// MOD_HUGE. (One warp on a star's row of 4M entries: 1.5 ms for each clustering.)
constexpr int MOD_LONG = 2048, MOD_HUGE = 65536;

__global__ void __launch_bounds__(256)
k_mod_long(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
           const int32_t* __restrict__ labels, int64_t n, const int64_t* __restrict__ co_off,
           const int32_t* __restrict__ co_id, int32_t maxdeg,
           unsigned long long* __restrict__ acc, const unsigned long long* reached, unsigned long long most) {
  if (*reached >= most) return;
  labels += (int64_t)blockIdx.y * n;
  unsigned long long inside = 0;
  auto walk = [&](int64_t from, int64_t to, int64_t step, int32_t lv) {
    for (int64_t i = from; i < to; i += step) inside += labels[adj[i]] == lv ? 1u : 0u;
  };
  for (int64_t r = co_off[MOD_LONG] + blockIdx.x; r < co_off[MOD_LONG + 1]; r += gridDim.x) {
    const int32_t v = co_id[r], lv = labels[v];
    const int64_t b = off[v], e = off[v + 1];
    if (lv >= 0 && e - b <= MOD_HUGE) walk(b + threadIdx.x, e, blockDim.x, lv);
  }
  if (maxdeg > MOD_HUGE)
    for (int64_t r = co_off[MOD_HUGE]; r < co_off[MOD_HUGE + 1]; ++r) {
      const int32_t v = co_id[r], lv = labels[v];
      if (lv >= 0)
        walk(off[v] + (int64_t)blockIdx.x * blockDim.x + threadIdx.x, off[v + 1],
             (int64_t)gridDim.x * blockDim.x, lv);
    }
  for (int o = 16; o; o >>= 1) inside += __shfl_xor_sync(0xffffffffu, inside, o);
  if ((threadIdx.x & 31) == 0 && inside) atomicAdd(&acc[4 * blockIdx.y], inside);
}

// S_c = sum over the cluster labels c of D_c^2; dsum is cleared for the next
// clustering.
__global__ void k_mod_clusters(int64_t n, unsigned long long* __restrict__ dsum,
                               unsigned long long* __restrict__ acc) {
  unsigned long long s = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long d = dsum[v];
    if (d) {
      s += d * d;
      dsum[v] = 0;
    }
  }
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0 && s) atomicAdd(&acc[2], s);
}

// ---- Modularity of SWEEP_BATCH clusterings in one pass over the graph.
// One pass per clustering reads every row's ids and gathers one 4-byte label
// per arc, a 32-byte sector each; with the labels turned to lab[v][query]
// (32 queries, 128 bytes a vertex) lane q compares for query q, the ids are
// read once for all 32, and a gather is one full line. Warps take equal
// pieces of the arc array, so a hub's row is not one warp's. R-MAT s20, 594
// pairs: 44 ms for the passes of the single clusterings, 16 ms here (13 of them
// in k_mod_rows_all, at most 3.9 GB of label lines per batch). It is taken where
// the clusters hold arcs enough (MOD_TOGETHER).
constexpr int SWEEP_BATCH = 32;

// lab[q][v] (nq rows) -> lt[v][32], -1 for the queries past nq
__global__ void __launch_bounds__(256)
k_turn_labels(const int32_t* __restrict__ lab, int64_t n, int nq, int32_t* __restrict__ lt,
              const unsigned long long* reached,
              unsigned long long least) {
  __shared__ int32_t tile[32][33];
  if (reached && *reached < least) return;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int64_t v0 = (int64_t)blockIdx.x * 32; v0 < n; v0 += (int64_t)gridDim.x * 32) {
    for (int q = ty; q < 32; q += 8)
      tile[q][tx] = q < nq && v0 + tx < n ? lab[(int64_t)q * n + v0 + tx] : -1;
    __syncthreads();
    for (int r = ty; r < 32; r += 8)
      if (v0 + r < n) lt[(v0 + r) * 32 + tx] = tile[tx][r];
    __syncthreads();
  }
}

// acc and dsum as for k_mod_rows, acc[4 q ..] and dsum[q n ..] of query q.
// The warp's piece is MOD_PIECE arcs; the row that holds its first arc comes
// from a search. A row's degree is added by the warp of its first arc, runs of
// one label in a lane's own sum (a cluster of most vertices would otherwise
// be one address for all warps).
constexpr int MOD_PIECE = 512;

__global__ void __launch_bounds__(256)
k_mod_rows_all(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
               const int32_t* __restrict__ lt, int64_t n, int64_t arcs, int nq,
               unsigned long long* __restrict__ dsum, unsigned long long* __restrict__ acc,
               const unsigned long long* reached,
              unsigned long long least) {
  constexpr unsigned FULL = 0xffffffffu;
  if (reached && *reached < least) return;
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  unsigned long long inside = 0, dsq = 0, run = 0;
  int32_t run_label = -1;
  for (int64_t p0 = warp * MOD_PIECE; p0 < arcs; p0 += nwarps * MOD_PIECE) {
    const int64_t p1 = min(arcs, p0 + (int64_t)MOD_PIECE);
    int64_t lo = 0, hi = n;  // the last row that starts at or before p0 is not empty
    while (hi - lo > 1) {
      const int64_t mid = (lo + hi) >> 1;
      if (off[mid] <= p0) lo = mid; else hi = mid;
    }
    int64_t v = lo, b = off[v];
    for (int64_t p = p0; p < p1; ++v) {
      const int64_t e = off[v + 1];
      const int32_t lv = lt[v * 32 + lane];
      if (b >= p0 && e > b && lv >= 0) {
        const unsigned long long d = (unsigned long long)(e - b);
        dsq += d * d;
        if (run_label < 0) run_label = lv;
        if (lv == run_label) run += d;
        else atomicAdd(&dsum[(int64_t)lane * n + lv], d);
      }
      const int64_t end = min(e, p1);
      if (__any_sync(FULL, lv >= 0)) {
        const int32_t want = lv >= 0 ? lv : -4;  // no label
        unsigned cnt = 0;
        for (int64_t i0 = p; i0 < end; i0 += 32) {
          const int m = (int)min((int64_t)32, end - i0);
          const int32_t x = lane < m ? adj[i0 + lane] : 0;
          int k = 0;
          for (; k + 8 <= m; k += 8) {
            int32_t l[8];
#pragma unroll
            for (int t = 0; t < 8; ++t)
              l[t] = lt[(int64_t)__shfl_sync(FULL, x, k + t) * 32 + lane];
#pragma unroll
            for (int t = 0; t < 8; ++t) cnt += l[t] == want ? 1u : 0u;
          }
          for (; k < m; ++k)
            cnt += lt[(int64_t)__shfl_sync(FULL, x, k) * 32 + lane] == want ? 1u : 0u;
        }
        inside += cnt;
      }
      p = end > p ? end : p;
      b = e;
    }
  }
  if (lane < nq) {
    if (run) atomicAdd(&dsum[(int64_t)lane * n + run_label], run);
    if (inside) atomicAdd(&acc[4 * lane], inside);
    if (dsq) atomicAdd(&acc[4 * lane + 1], dsq);
  }
}

// S_c of query blockIdx.y; dsum is cleared for the next batch.
__global__ void k_mod_clusters_all(int64_t n, unsigned long long* __restrict__ dsum,
                                   unsigned long long* __restrict__ acc) {
  unsigned long long* ds = dsum + (int64_t)blockIdx.y * n;
  unsigned long long s = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long d = ds[v];
    if (d) {
      s += d * d;
      ds[v] = 0;
    }
  }
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0 && s) atomicAdd(&acc[4 * blockIdx.y + 2], s);
}

// Entries of the cores' prefixes over a batch's clusterings, per vertex, from which
// its labels are turned (16 pairs, turned and one by one, ms: grid of 4M vertices
// without clusters 1.17 and 0.61; R-MAT s22, few clusters, 1.49 and .49; 500k borders
// of 2000 cores 0.67 and 1.12; tree of 3M vertices, half of it clustered, 7.4 and
// 13.7).
constexpr double MOD_TOGETHER = 2.0;
// vertices from which the choice is made: turning the labels of fewer costs less
// than the launches that choose (SBM of 10k vertices, 16 pairs, 125 us and 140)
constexpr int64_t MOD_CHOOSE = 1 << 17;

// sum of d^2 over all vertices
__global__ void k_deg_sq(const int32_t* __restrict__ deg, int64_t n,
                         unsigned long long* __restrict__ out) {
  unsigned long long s = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long d = (unsigned long long)deg[v];
    s += d * d;
  }
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0 && s) atomicAdd(out, s);
}

unsigned grid_of(int64_t work, int per_block) {
  int64_t g = (work + per_block - 1) / per_block;
  if (g < 1) g = 1;
  if (g > sm_count() * 16) g = sm_count() * 16;
  return (unsigned)g;
}

double modularity_of(const unsigned long long* acc, unsigned long long deg_sq_all, int64_t arcs) {
  if (arcs == 0) return 0.0;
  const double two_m = (double)arcs;
  const unsigned long long su = deg_sq_all - acc[1];  // unclustered singletons
  return (double)acc[0] / two_m - (double)(acc[2] + su) / (two_m * two_m);
}

}  // namespace

// Launches the modularity passes of one clustering (device labels) into the
// four words acc (zeroed by the caller); dsum must be zero on entry.
int launch_modularity(const IndexData& ix, const int32_t* labels_dev, unsigned long long* dsum,
                      unsigned long long* acc, cudaStream_t s) {
  if (ix.n == 0) return SCAN_OK;
  k_mod_rows<false><<<grid_of(ix.n, 256), 256, 0, s>>>(ix.off, ix.adj, labels_dev, ix.n, dsum, acc,
                                                       nullptr, 0, 0);
  GS_LAUNCH();
  k_mod_clusters<<<grid_of(ix.n, 256 * 8), 256, 0, s>>>(ix.n, dsum, acc);
  GS_LAUNCH();
  return SCAN_OK;
}

int modularity_impl(const IndexData& ix, const int32_t* labels, double* q, cudaStream_t s) {
  Pool pool(s);
  const int64_t n = ix.n;
  if (n == 0 || ix.arcs == 0) {
    *q = 0.0;
    return SCAN_OK;
  }
  const bool dev_in = is_device_ptr(labels);
  const int32_t* lab = labels;
  if (!dev_in) {
    int32_t* tmp = pool.get<int32_t>(n);
    if (!tmp) return SCAN_ENOMEM;
    GS_CUDA(cudaMemcpyAsync(tmp, labels, n * sizeof(int32_t), cudaMemcpyHostToDevice, s));
    lab = tmp;
  }
  unsigned long long* dsum = pool.get<unsigned long long>(n);
  unsigned long long* acc = pool.get<unsigned long long>(5);  // 4 words + sum of d^2
  if (!dsum || !acc) return SCAN_ENOMEM;
  GS_CUDA(cudaMemsetAsync(dsum, 0, n * sizeof(unsigned long long), s));
  GS_CUDA(cudaMemsetAsync(acc, 0, 5 * sizeof(unsigned long long), s));
  k_deg_sq<<<grid_of(n, 256 * 8), 256, 0, s>>>(ix.deg, n, acc + 4);
  GS_LAUNCH();
  GS_TRY(launch_modularity(ix, lab, dsum, acc, s));
  unsigned long long h[5];
  GS_CUDA(cudaMemcpyAsync(h, acc, sizeof(h), cudaMemcpyDeviceToHost, s));
  GS_CUDA(cudaStreamSynchronize(s));
  if (h[3]) return SCAN_EINVAL;  // a label was >= n
  *q = modularity_of(h, h[4], ix.arcs);
  return SCAN_OK;
}

int sweep_impl(const IndexData& ix, int count, const int* mu, const double* eps, double* q,
               cudaStream_t s) {
  const int64_t n = ix.n;
  if (count == 0) return SCAN_OK;
  if (n == 0 || ix.arcs == 0) {
    for (int i = 0; i < count; ++i) q[i] = 0.0;
    return SCAN_OK;
  }
  Pool pool(s);
  // queries are answered SWEEP_BATCH at a time into one label buffer
  const int B = count < SWEEP_BATCH ? count : SWEEP_BATCH;
  int32_t* lab = pool.get<int32_t>((size_t)B * n);
  unsigned long long* acc = pool.get<unsigned long long>(4 * (size_t)count + 1);
  unsigned* st = pool.get<unsigned>(4);  // status, -, entries of a batch's prefixes (2 words)
  unsigned long long* reached =
      st && n >= MOD_CHOOSE ? reinterpret_cast<unsigned long long*>(st + 2) : nullptr;
  // all clusterings of a batch at once: 12 more bytes per vertex and query;
  // one at a time where there is no room for them, and for a few pairs: a
  // gather of turned labels is 128 bytes per arc whatever their number, one
  // of single labels a 32-byte sector per arc and query, and a pass of its
  // own skips the rows that its one clustering leaves out
  int32_t* lt = B >= 8 ? pool.get<int32_t>((size_t)SWEEP_BATCH * n) : nullptr;
  unsigned long long* dsum = lt ? pool.get<unsigned long long>((size_t)B * n) : nullptr;
  if (lt && !dsum) pool.put(lt);
  bool together = dsum != nullptr;
  if (!dsum) dsum = pool.get<unsigned long long>(n);
  if (!lab || !dsum || !acc || !st) return SCAN_ENOMEM;
  GS_CUDA(cudaMemsetAsync(dsum, 0, (together ? (size_t)B : 1) * n * sizeof(unsigned long long), s));
  GS_CUDA(cudaMemsetAsync(acc, 0, (4 * (size_t)count + 1) * sizeof(unsigned long long), s));
  GS_CUDA(cudaMemsetAsync(st, 0, 4 * sizeof(unsigned), s));
  // Turned labels cost 256 bytes a vertex and 132 per arc of rows with a label,
  // whatever the number of clusterings; single labels 36 bytes per arc of a
  // clustered row.
  const unsigned long long least = (unsigned long long)(MOD_TOGETHER * (double)n);
  k_deg_sq<<<grid_of(n, 256 * 8), 256, 0, s>>>(ix.deg, n, acc + 4 * (size_t)count);
  GS_LAUNCH();
  for (int b0 = 0; b0 < count; b0 += B) {
    const int nb = count - b0 < B ? count - b0 : B;
    if (reached) GS_CUDA(cudaMemsetAsync(reached, 0, sizeof(*reached), s));
    int rc = run_queries(ix, nb, mu + b0, eps + b0, lab, 0, pool, s, st, reached);
    if (rc == SCAN_ENOMEM && together) {  // the queries need the room themselves
      pool.put(lt);
      pool.put(dsum);
      together = false;
      dsum = pool.get<unsigned long long>(n);
      if (!dsum) return SCAN_ENOMEM;
      GS_CUDA(cudaMemsetAsync(dsum, 0, n * sizeof(unsigned long long), s));
      rc = run_queries(ix, nb, mu + b0, eps + b0, lab, 0, pool, s, st);
    }
    GS_TRY(rc);
    if (together) {
      k_turn_labels<<<grid_of(n, 32), 256, 0, s>>>(lab, n, nb, lt, reached, least);
      GS_LAUNCH();
      k_mod_rows_all<<<grid_of(ix.arcs, MOD_PIECE * 8), 256, 0, s>>>(
          ix.off, ix.adj, lt, n, ix.arcs, nb, dsum, acc + 4 * (size_t)b0, reached, least);
      GS_LAUNCH();
      if (reached) {
        k_mod_rows<true><<<dim3(grid_of(n, 256), nb), 256, 0, s>>>(
            ix.off, ix.adj, lab, n, dsum, acc + 4 * (size_t)b0, reached, least, MOD_LONG);
        GS_LAUNCH();
      }
      if (reached && ix.maxdeg > MOD_LONG) {
        k_mod_long<<<dim3(std::max(8, sm_count() * 8 / nb), nb), 256, 0, s>>>(
            ix.off, ix.adj, lab, n, ix.co_off, ix.co_id, ix.maxdeg, acc + 4 * (size_t)b0, reached,
            least);
        GS_LAUNCH();
      }
      k_mod_clusters_all<<<dim3(grid_of(n, 256 * 32), nb), 256, 0, s>>>(n, dsum,
                                                                       acc + 4 * (size_t)b0);
      GS_LAUNCH();
      continue;
    }
    for (int i = 0; i < nb; ++i)
      GS_TRY(launch_modularity(ix, lab + (size_t)i * n, dsum, acc + 4 * (size_t)(b0 + i), s));
  }
  std::vector<unsigned long long> h(4 * (size_t)count + 1);
  unsigned hst = 0;
  GS_CUDA(cudaMemcpyAsync(h.data(), acc, h.size() * sizeof(unsigned long long),
                          cudaMemcpyDeviceToHost, s));
  GS_CUDA(cudaMemcpyAsync(&hst, st, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
  GS_CUDA(cudaStreamSynchronize(s));
  if (hst & DEV_LIMIT) return SCAN_ETIMEOUT;
  for (int i = 0; i < count; ++i) q[i] = modularity_of(&h[4 * (size_t)i], h.back(), ix.arcs);
  return SCAN_OK;
}

}  // namespace gscan

using namespace gscan;

extern "C" {

int scan_modularity(scan_index* index, const int32_t* labels, double* q, uintptr_t stream) {
  if (!index || !q || (index->d.n > 0 && !labels)) return SCAN_EINVAL;
  return modularity_impl(index->d, labels, q, (cudaStream_t)stream);
}

int scan_sweep(scan_index* index, int count, const int* mu, const double* eps, double* q,
               uintptr_t stream) {
  if (!index || count < 0 || (count > 0 && (!mu || !eps || !q))) return SCAN_EINVAL;
  for (int i = 0; i < count; ++i) {
    if (mu[i] < 2) return SCAN_EINVAL;
    if (!(eps[i] >= 0.0 && eps[i] <= 1.0)) return SCAN_EINVAL;
  }
  return sweep_impl(index->d, count, mu, eps, q, (cudaStream_t)stream);
}

}  // extern "C"
