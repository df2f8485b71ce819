// LSH index mode (Sections 2.1.2, 5 and 6.3).
//
// Selection (Section 6.3 heuristic): an edge is approximated iff both of its
// endpoints have degree > T; only vertices of degree > T with at least one
// such neighbour are sketched (row[v] >= 0, numbered in id order).
//
// Random numbers: R(key, c) = output number c of SplitMix64 (Steele, Lea,
// Flood 2014) whose state starts at key, i.e. mix64(key + (c+1) * golden).
//  SimHash (Charikar): hyperplane j gives x in N̄(v) the sign +1 iff bit j%64 of
//    R(ks, x*1024 + j/64) is set, ks = mix64(seed ^ "SIMH"); s_j = sum of the
//    signs over N̄(v); bit j = [s_j >= 0], i.e. at least half of them are +1.
//    Estimate max(0, cos(pi h / k)) for Hamming distance h, from a table
//    computed on the host in double precision.
//  MinHash: h(x) = low 32 bits of R(km, x), km = mix64(seed ^ "MINH").
//    k-partition (one-permutation hashing): bin = top log2(k) bits, value =
//    the other bits, min per bin, empty = 0xFFFFFFFF; estimate = equal
//    non-empty bins / (k - bins empty in both). Standard: h_j(x) = low 32 bits
//    of R(km ^ ((j+1) * golden), x), min per j; estimate = equal / k.
#include <cmath>

#include "scan_internal.cuh"

namespace gscan {

namespace {

constexpr uint64_t GOLDEN = 0x9E3779B97F4A7C15ULL;

__host__ __device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

__device__ __forceinline__ uint64_t splitmix_out(uint64_t key, uint64_t c) {
  return mix64(key + (c + 1) * GOLDEN);
}

__global__ void k_select_flags(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
                               const int32_t* __restrict__ deg, int64_t n, int T,
                               int32_t* __restrict__ flag) {
  const int lane = threadIdx.x & 31;
  const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = w0; v < n; v += nw) {
    bool any = false;
    if (deg[v] > T) {  // uniform across the warp
      for (int64_t j = off[v] + lane; j < off[v + 1]; j += 32)
        if (deg[adj[j]] > T) { any = true; break; }
    }
    any = __any_sync(0xffffffffu, any);
    if (lane == 0) flag[v] = any ? 1 : 0;
  }
}

__global__ void k_select_rows(const int32_t* __restrict__ flag, const int64_t* __restrict__ pre,
                              int64_t n, int32_t* __restrict__ row) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    row[v] = flag[v] ? (int32_t)pre[v] : -1;
}

// ---- SimHash of unweighted graphs: vertical counters.
// s_j >= 0 iff at least half of the signs of hyperplane j are set, so only
// the number of set bits per hyperplane is needed. Each lane hashes its own
// elements of N̄(v) (SplitMix64 gives 64 hyperplanes at once) and adds them
// into bit-sliced counters: plane p of a word holds bit p of 32 hyperplanes'
// counts, so an element costs about five logical instructions per 32
// hyperplanes instead of one shared load, test and add per hyperplane (5.7 ms
// that way on R-MAT s22, k = 256; now 0.4 ms for the rows of one pass and
// 0.75 ms for the longer ones: the hashing is most of it).
// The lanes' counters are then added across the warp the same way, each
// exchange halving the words a lane keeps, and compared with the threshold
// plane by plane. SH_LANE elements fill the five planes of a lane.
constexpr int SH_LANE = 30;
constexpr int SH_ROW = 32 * SH_LANE;  // elements of one warp pass
constexpr int SH_W32 = 8;             // 32-hyperplane words per pass (256 hyperplanes)
constexpr int SH_PLANES = 10;         // counts up to SH_ROW < 2^10

// Set bits per hyperplane of elements c0 .. min(c0 + SH_ROW, cnt) of N̄(v)
// (element 0 is v itself, c >= 1 is adj[c - 1]) for the words w32_0 ..
// w32_0 + 7 of the hyperplanes: on return lane l holds, in pl[0..9], the
// bit-sliced counts of word w32_0 + l/4 (four lanes hold the same).
__device__ __forceinline__ void simhash_counts(const int32_t* __restrict__ adj, int32_t v,
                                               int64_t c0, int64_t cnt, int w64, int W,
                                               uint64_t key, uint32_t (&pl)[SH_PLANES]) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int64_t c1 = min(cnt, c0 + (int64_t)SH_ROW);
  uint32_t a[SH_W32][5];
#pragma unroll
  for (int w = 0; w < SH_W32; ++w)
#pragma unroll
    for (int p = 0; p < 5; ++p) a[w][p] = 0;
  for (int64_t c = c0 + lane; c < c1; c += 64) {
    const bool two = c + 32 < c1;
    const uint64_t x = c == 0 ? (uint64_t)v : (uint64_t)adj[c - 1];
    const uint64_t y = two ? (uint64_t)adj[c + 31] : 0;
#pragma unroll
    for (int q = 0; q < SH_W32 / 2; ++q) {
      if (w64 + q >= W) break;  // uniform
      const uint64_t hx = splitmix_out(key, x * 1024u + (uint64_t)(w64 + q));
      const uint64_t hy = two ? splitmix_out(key, y * 1024u + (uint64_t)(w64 + q)) : 0;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t(&r)[5] = a[2 * q + h];
        const uint32_t u = (uint32_t)(hx >> (32 * h)), t = (uint32_t)(hy >> (32 * h));
        uint32_t carry = (r[0] & u) | (r[0] & t) | (u & t);
        r[0] ^= u ^ t;
#pragma unroll
        for (int p = 1; p < 5; ++p) {
          const uint32_t n = r[p] & carry;
          r[p] ^= carry;
          carry = n;
        }
      }
    }
  }
  // add across lanes: at distance 16, 8 and 4 a lane keeps half of its words
  // and sends the other half; at 2 and 1 both sides keep the sum
  uint32_t b4[4][6], b2[2][7], b1[8], b0[9];
  auto add = [](const uint32_t* x, const uint32_t* y, int planes, uint32_t* out) {
    uint32_t carry = 0;
#pragma unroll
    for (int p = 0; p < SH_PLANES; ++p) {
      if (p >= planes) break;
      out[p] = x[p] ^ y[p] ^ carry;
      carry = (x[p] & y[p]) | (x[p] & carry) | (y[p] & carry);
    }
    out[planes] = carry;
  };
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    uint32_t mine[5], theirs[5];
#pragma unroll
    for (int p = 0; p < 5; ++p) {
      mine[p] = (lane & 16) ? a[w + 4][p] : a[w][p];
      theirs[p] = __shfl_xor_sync(FULL, (lane & 16) ? a[w][p] : a[w + 4][p], 16);
    }
    add(mine, theirs, 5, b4[w]);
  }
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    uint32_t mine[6], theirs[6];
#pragma unroll
    for (int p = 0; p < 6; ++p) {
      mine[p] = (lane & 8) ? b4[w + 2][p] : b4[w][p];
      theirs[p] = __shfl_xor_sync(FULL, (lane & 8) ? b4[w][p] : b4[w + 2][p], 8);
    }
    add(mine, theirs, 6, b2[w]);
  }
  {
    uint32_t mine[7], theirs[7];
#pragma unroll
    for (int p = 0; p < 7; ++p) {
      mine[p] = (lane & 4) ? b2[1][p] : b2[0][p];
      theirs[p] = __shfl_xor_sync(FULL, (lane & 4) ? b2[0][p] : b2[1][p], 4);
    }
    add(mine, theirs, 7, b1);
  }
  {
    uint32_t theirs[8];
#pragma unroll
    for (int p = 0; p < 8; ++p) theirs[p] = __shfl_xor_sync(FULL, b1[p], 2);
    add(b1, theirs, 8, b0);
  }
  {
    uint32_t theirs[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) theirs[p] = __shfl_xor_sync(FULL, b0[p], 1);
    add(b0, theirs, 9, pl);
  }
}

// A warp per sketched vertex of at most SH_ROW closed neighbours.
constexpr int SH_T = 256;

__global__ void __launch_bounds__(SH_T)
k_simhash(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
          const int32_t* __restrict__ hlist, int64_t nH, int W, uint64_t key,
          uint32_t* __restrict__ sig32) {
  const int lane = threadIdx.x & 31;
  const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t h = w0; h < nH; h += nw) {
    const int32_t v = hlist[h];
    const int64_t b = off[v], cnt = off[v + 1] - b + 1;
    if (cnt > SH_ROW) continue;  // k_simhash_long
    const uint32_t need = (uint32_t)((cnt + 1) / 2);
    for (int w64 = 0; w64 < W; w64 += SH_W32 / 2) {
      uint32_t pl[SH_PLANES];
      simhash_counts(adj + b, v, 0, cnt, w64, W, key, pl);
      uint32_t gt = 0, eq = 0xffffffffu;  // count > need, = need in the planes above
#pragma unroll
      for (int p = SH_PLANES - 1; p >= 0; --p) {
        const uint32_t bit = (need >> p & 1u) ? 0xffffffffu : 0u;
        gt |= eq & pl[p] & ~bit;
        eq &= ~(pl[p] ^ bit);
      }
      const int w = 2 * w64 + (lane >> 2);
      if ((lane & 3) == 0 && w < 2 * W) sig32[h * 2 * W + w] = gt | eq;
    }
  }
}

// A CTA per longer row: its warps take passes of SH_ROW elements and add
// their counts in shared memory. Four warps: most long rows have two to four
// passes, and a hub's 150 are still only 38 in a row (R-MAT s22, k = 256:
// 0.75 ms; eight warps 1.12, sixteen 1.29, two 1.45; one warp walking up to
// four passes alone and CTAs beyond them together 0.5 ms slower).
constexpr int SHL_T = 128;

__global__ void __launch_bounds__(SHL_T)
k_simhash_long(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
               const int32_t* __restrict__ hlist, int64_t nH, int W, uint64_t key,
               uint32_t* __restrict__ sig32) {
  __shared__ unsigned cnts[32 * SH_W32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int64_t h = blockIdx.x; h < nH; h += gridDim.x) {
    const int32_t v = hlist[h];
    const int64_t b = off[v], cnt = off[v + 1] - b + 1;
    if (cnt <= SH_ROW) continue;
    for (int w64 = 0; w64 < W; w64 += SH_W32 / 2) {
      for (int j = threadIdx.x; j < 32 * SH_W32; j += SHL_T) cnts[j] = 0;
      __syncthreads();
      for (int64_t c0 = (int64_t)wid * SH_ROW; c0 < cnt; c0 += (int64_t)(SHL_T / 32) * SH_ROW) {
        uint32_t pl[SH_PLANES];
        simhash_counts(adj + b, v, c0, cnt, w64, W, key, pl);
        // the four lanes of a word take eight hyperplanes each
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int bit = (lane & 3) * 8 + i;
          unsigned t = 0;
#pragma unroll
          for (int p = 0; p < SH_PLANES; ++p) t |= (pl[p] >> bit & 1u) << p;
          atomicAdd(&cnts[(lane >> 2) * 32 + bit], t);
        }
      }
      __syncthreads();
      for (int j = threadIdx.x; j < 32 * SH_W32; j += SHL_T) {
        const unsigned bal = __ballot_sync(0xffffffffu, 2 * (int64_t)cnts[j] >= cnt);
        const int w = 2 * w64 + (j >> 5);
        if (lane == 0 && w < 2 * W) sig32[h * 2 * W + w] = bal;
      }
      __syncthreads();
    }
  }
}

// SimHash of weighted graphs, one CTA per sketched vertex: elements of N̄(v)
// in chunks of SH_T; each thread hashes one element into W words, then
// hyperplane j adds +-w(v,x) (w(v,v) = 1) over the chunk in double precision,
// in the order v, then N(v) in id order: a fixed order that decides every
// sign reproducibly.
constexpr int SH_WMAX = 64;  // k <= 4096

__global__ void __launch_bounds__(SH_T)
k_simhash_w(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
            const int32_t* __restrict__ hlist, int64_t nH, int W, uint64_t key,
            const double* __restrict__ wcsr, uint64_t* __restrict__ sig) {
  extern __shared__ uint64_t bits[];  // [SH_T][W]
  __shared__ unsigned ballots[SH_WMAX * 2];
  __shared__ double wel[SH_T];
  const int k = 64 * W;
  const int per = (k + SH_T - 1) / SH_T;  // hyperplanes per thread (<= 16)
  double s[16];
  for (int64_t h = blockIdx.x; h < nH; h += gridDim.x) {
    const int32_t v = hlist[h];
    const int64_t b = off[v], e = off[v + 1];
    const int64_t cnt = e - b + 1;  // N̄(v)
#pragma unroll
    for (int t = 0; t < 16; ++t) s[t] = 0.0;
    for (int64_t c0 = 0; c0 < cnt; c0 += SH_T) {
      const int64_t c = c0 + threadIdx.x;
      if (c < cnt) {
        const int64_t x = c == 0 ? (int64_t)v : (int64_t)adj[b + c - 1];
        for (int w = 0; w < W; ++w)
          bits[threadIdx.x * W + w] = splitmix_out(key, (uint64_t)x * 1024u + (uint64_t)w);
        wel[threadIdx.x] = c == 0 ? 1.0 : wcsr[b + c - 1];
      }
      __syncthreads();
      const int m = (int)min((int64_t)SH_T, cnt - c0);
#pragma unroll
      for (int t = 0; t < 16; ++t) {
        if (t >= per) break;
        const int j = threadIdx.x + t * SH_T;
        if (j >= k) break;
        const int wj = j >> 6, bj = j & 63;
        double acc = s[t];
        for (int el = 0; el < m; ++el) {
          const bool up = (bits[el * W + wj] >> bj) & 1ull;
          acc = __dadd_rn(acc, up ? wel[el] : -wel[el]);
        }
        s[t] = acc;
      }
      __syncthreads();
    }
    // bit j = [s_j >= 0]; hyperplane j = threadIdx.x + t*SH_T, lanes hold 32 consecutive j
    const int lane = threadIdx.x & 31;
    for (int t = 0; t < per; ++t) {
      const int j = threadIdx.x + t * SH_T;
      const unsigned bal = __ballot_sync(0xffffffffu, j < k && s[t] >= 0.0);
      if (lane == 0 && j < k) ballots[j >> 5] = bal;
    }
    __syncthreads();
    for (int w = threadIdx.x; w < W; w += SH_T)
      sig[h * W + w] = (uint64_t)ballots[2 * w] | ((uint64_t)ballots[2 * w + 1] << 32);
    __syncthreads();
  }
}

// One CTA per sketched vertex; k <= 1024 bins/hashes in shared memory.
__global__ void __launch_bounds__(256)
k_minhash(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
          const int32_t* __restrict__ hlist, int64_t nH, int k, int L, int kpartition,
          uint64_t key, uint32_t* __restrict__ mh) {
  __shared__ uint32_t mins[1024];
  for (int64_t h = blockIdx.x; h < nH; h += gridDim.x) {
    const int32_t v = hlist[h];
    const int64_t b = off[v], e = off[v + 1];
    const int64_t cnt = e - b + 1;
    for (int j = threadIdx.x; j < k; j += blockDim.x) mins[j] = 0xFFFFFFFFu;
    __syncthreads();
    if (kpartition) {
      const uint32_t vmask = L == 0 ? 0x7FFFFFFFu : ((1u << (32 - L)) - 1u);
      for (int64_t c = threadIdx.x; c < cnt; c += blockDim.x) {
        const int64_t x = c == 0 ? (int64_t)v : (int64_t)adj[b + c - 1];
        const uint32_t hv = (uint32_t)splitmix_out(key, (uint64_t)x);
        const uint32_t bin = L == 0 ? 0u : hv >> (32 - L);
        atomicMin(&mins[bin], hv & vmask);
      }
    } else {
      for (int j = threadIdx.x; j < k; j += blockDim.x) {
        const uint64_t kj = key ^ ((uint64_t)(j + 1) * GOLDEN);
        uint32_t mn = 0xFFFFFFFFu;
        for (int64_t c = 0; c < cnt; ++c) {
          const int64_t x = c == 0 ? (int64_t)v : (int64_t)adj[b + c - 1];
          const uint32_t hv = (uint32_t)splitmix_out(kj, (uint64_t)x);
          mn = min(mn, hv);
        }
        mins[j] = mn;
      }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < k; j += blockDim.x) mh[h * k + j] = mins[j];
    __syncthreads();
  }
}

// ---- Estimates: overwrite the similarity of every approximated arc.
// Work items are pieces of at most LSH_PIECE arcs of the sketched vertices'
// rows (ipre: prefix of the pieces per row), a warp each: a hub's row is as
// many items as its length asks for. A warp collects the approximated arcs
// of its piece (row[x] >= 0) in a queue and estimates 32 at a time: G lanes
// read one neighbour's sketch together, as consecutive 16-byte vectors, so
// that a load touches 32/G sketches instead of 32 (a lane per arc read 32
// separate lines per load: on R-MAT s22 19.1 ms for the 256-byte MinHash
// sketches, now 3.7 ms; 5.3 ms for the 32-byte
// SimHash signatures, now 0.8 ms). The G lanes' partial
// sums are added while being dealt out: lane l ends with arc l's total.
constexpr int LSH_PIECE = 1024;

__device__ __forceinline__ int64_t piece_row(const int64_t* __restrict__ ipre, int64_t nH,
                                             int64_t it) {
  int64_t lo = 0, hi = nH;  // largest h with ipre[h] <= it
  while (hi - lo > 1) {
    const int64_t mid = (lo + hi) >> 1;
    if (ipre[mid] <= it) lo = mid; else hi = mid;
  }
  return lo;
}

// MinHash: equal non-empty bins in the low half, bins empty in both in the
// high half; SimHash: differing bits.
__device__ __forceinline__ uint32_t mh_bin(uint32_t x, uint32_t y) {
  return x == y ? (x == 0xFFFFFFFFu ? 0x10000u : 1u) : 0u;
}
template <bool SIMHASH>
__device__ __forceinline__ uint32_t sketch_part(const uint4& x, const uint4& y) {
  if (SIMHASH)
    return __popc(x.x ^ y.x) + __popc(x.y ^ y.y) + __popc(x.z ^ y.z) + __popc(x.w ^ y.w);
  return mh_bin(x.x, y.x) + mh_bin(x.y, y.y) + mh_bin(x.z, y.z) + mh_bin(x.w, y.w);
}

// nvec: 16-byte vectors per sketch, read G at a time. tab: cosine table
// (SimHash), k the length in bins (MinHash).
template <bool SIMHASH, int G>
__global__ void __launch_bounds__(256)
k_lsh_sims(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
           const int32_t* __restrict__ row, const int32_t* __restrict__ hlist, int64_t nH,
           const int64_t* __restrict__ ipre, int nvec, const uint4* __restrict__ sk,
           const double* __restrict__ tab, int k, int kpartition, double* __restrict__ sim_csr) {
  constexpr unsigned FULL = 0xffffffffu;
  __shared__ int32_t q_r[8][64], q_j[8][64];  // queued sketch rows, arc positions in the row
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int lg = lane & (G - 1), grp = lane & ~(G - 1);
  const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t items = ipre[nH];
  int32_t* qr = q_r[wid];
  int32_t* qj = q_j[wid];
  for (int64_t it = w0; it < items; it += nw) {
    const int64_t h = piece_row(ipre, nH, it);
    const int32_t u = hlist[h];
    const int64_t rb = off[u];
    const int len = (int)(off[u + 1] - rb);
    const int p0 = (int)(it - ipre[h]) * LSH_PIECE, p1 = min(len, p0 + LSH_PIECE);
    const uint4* own = sk + h * nvec;
    int n = 0;  // queued arcs
    auto flush = [&](int m) {  // estimate the first m <= 32 queued arcs
      uint32_t part[G];
#pragma unroll
      for (int s = 0; s < G; ++s) part[s] = 0;
      for (int t = lg; t - lg < nvec; t += G) {
        const bool in = t < nvec;
        const uint4 x = in ? own[t] : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int s = 0; s < G; ++s) {
          if (in && grp + s < m)
            part[s] += sketch_part<SIMHASH>(x, sk[(int64_t)qr[grp + s] * nvec + t]);
        }
      }
#pragma unroll
      for (int o = G / 2; o; o >>= 1)
#pragma unroll
        for (int s = 0; s < o; ++s) {
          const bool up = lane & o;
          const uint32_t keep = up ? part[s + o] : part[s], send = up ? part[s] : part[s + o];
          part[s] = keep + __shfl_xor_sync(FULL, send, o);
        }
      if (lane < m) {
        double v;
        if (SIMHASH) {
          v = tab[part[0]];
        } else {
          const int match = (int)(part[0] & 0xffffu), both_empty = (int)(part[0] >> 16);
          const int denom = kpartition ? k - both_empty : k;
          v = denom > 0 ? __ddiv_rn((double)match, (double)denom) : 0.0;
        }
        sim_csr[rb + qj[lane]] = v;
      }
    };
    for (int p = p0; p < p1; p += 32) {
      const int j = p + lane;
      const int32_t r = j < p1 ? row[adj[rb + j]] : -1;
      const unsigned m = __ballot_sync(FULL, r >= 0);
      if (r >= 0) {
        const int at = n + __popc(m & ((1u << lane) - 1u));
        qr[at] = r;
        qj[at] = j;
      }
      n += __popc(m);
      __syncwarp();
      if (n >= 32) {
        flush(32);
        n -= 32;
        __syncwarp();
        const int32_t r2 = qr[32 + lane], j2 = qj[32 + lane];  // at most 31 are left
        __syncwarp();
        qr[lane] = r2;
        qj[lane] = j2;
        __syncwarp();
      }
    }
    flush(n);
    __syncwarp();
  }
}

// Sketches that are no multiple of 16 bytes: a lane per arc.
template <bool SIMHASH>
__global__ void __launch_bounds__(256)
k_lsh_sims_odd(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
               const int32_t* __restrict__ row, const int32_t* __restrict__ hlist, int64_t nH,
               const int64_t* __restrict__ ipre, int words, const uint32_t* __restrict__ sk,
               const double* __restrict__ tab, int k, int kpartition,
               double* __restrict__ sim_csr) {
  const int lane = threadIdx.x & 31;
  const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t items = ipre[nH];
  for (int64_t it = w0; it < items; it += nw) {
    const int64_t h = piece_row(ipre, nH, it);
    const int32_t u = hlist[h];
    const int64_t rb = off[u];
    const int len = (int)(off[u + 1] - rb);
    const int p0 = (int)(it - ipre[h]) * LSH_PIECE, p1 = min(len, p0 + LSH_PIECE);
    for (int j = p0 + lane; j < p1; j += 32) {
      const int32_t r = row[adj[rb + j]];
      if (r < 0) continue;
      uint32_t part = 0;
      for (int t = 0; t < words; ++t) {
        const uint32_t x = sk[h * words + t], y = sk[(int64_t)r * words + t];
        part += SIMHASH ? (uint32_t)__popc(x ^ y) : mh_bin(x, y);
      }
      double v;
      if (SIMHASH) {
        v = tab[part];
      } else {
        const int match = (int)(part & 0xffffu), both_empty = (int)(part >> 16);
        const int denom = kpartition ? k - both_empty : k;
        v = denom > 0 ? __ddiv_rn((double)match, (double)denom) : 0.0;
      }
      sim_csr[rb + j] = v;
    }
  }
}

// sketched vertices in row order, and the pieces of their rows
__global__ void k_hlist(const int32_t* __restrict__ row, const int32_t* __restrict__ deg, int64_t n,
                        int32_t* __restrict__ hlist, int32_t* __restrict__ pieces) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    if (row[v] >= 0) {
      hlist[row[v]] = (int32_t)v;
      pieces[row[v]] = (deg[v] + LSH_PIECE - 1) / LSH_PIECE;
    }
}

// Estimates from sketches of `words` 32-bit words.
template <bool SIMHASH>
int launch_sims(const int64_t* off, const int32_t* adj, const int32_t* row, const int32_t* hlist,
                int64_t nH, const int64_t* ipre, int words, const uint32_t* sk, const double* tab,
                int k, int kpartition, double* sim_csr, cudaStream_t s) {
  const unsigned g = (unsigned)std::min<int64_t>((nH + 7) / 8, sm_count() * 32);
  const int nvec = words / 4;
  const uint4* v = reinterpret_cast<const uint4*>(sk);
  // lanes per sketch: enough for its vectors, up to a warp
  if (words % 4)
    k_lsh_sims_odd<SIMHASH><<<g, 256, 0, s>>>(off, adj, row, hlist, nH, ipre, words, sk, tab, k,
                                              kpartition, sim_csr);
  else if (nvec <= 1)
    k_lsh_sims<SIMHASH, 1><<<g, 256, 0, s>>>(off, adj, row, hlist, nH, ipre, nvec, v, tab, k,
                                             kpartition, sim_csr);
  else if (nvec <= 2)
    k_lsh_sims<SIMHASH, 2><<<g, 256, 0, s>>>(off, adj, row, hlist, nH, ipre, nvec, v, tab, k,
                                             kpartition, sim_csr);
  else if (nvec <= 4)
    k_lsh_sims<SIMHASH, 4><<<g, 256, 0, s>>>(off, adj, row, hlist, nH, ipre, nvec, v, tab, k,
                                             kpartition, sim_csr);
  else if (nvec <= 8)
    k_lsh_sims<SIMHASH, 8><<<g, 256, 0, s>>>(off, adj, row, hlist, nH, ipre, nvec, v, tab, k,
                                             kpartition, sim_csr);
  else if (nvec <= 16)
    k_lsh_sims<SIMHASH, 16><<<g, 256, 0, s>>>(off, adj, row, hlist, nH, ipre, nvec, v, tab, k,
                                              kpartition, sim_csr);
  else
    k_lsh_sims<SIMHASH, 32><<<g, 256, 0, s>>>(off, adj, row, hlist, nH, ipre, nvec, v, tab, k,
                                              kpartition, sim_csr);
  GS_LAUNCH();
  return SCAN_OK;
}

}  // namespace

int lsh_select(const int64_t* off, const int32_t* adj, const int32_t* deg, int64_t n, int T,
               int32_t* row, int64_t* nH_host, Pool& pool, cudaStream_t s) {
  int32_t* flag = pool.tmp<int32_t>(n > 0 ? n : 1);
  int64_t* pre = pool.tmp<int64_t>(n + 1);
  if (!flag || !pre) return SCAN_ENOMEM;
  if (n > 0) {
    k_select_flags<<<(unsigned)std::min<int64_t>((n + 7) / 8, sm_count() * 32), 256, 0, s>>>(off, adj, deg,
                                                                                     n, T, flag);
    GS_LAUNCH();
  }
  GS_TRY(exclusive_scan_i32_to_i64(flag, pre, n, pool, s));
  if (n > 0) {
    k_select_rows<<<(unsigned)std::min<int64_t>((n + 255) / 256, sm_count() * 32), 256, 0, s>>>(flag, pre,
                                                                                       n, row);
    GS_LAUNCH();
  }
  GS_CUDA(cudaMemcpyAsync(nH_host, pre + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  GS_CUDA(cudaStreamSynchronize(s));
  pool.put(flag);
  pool.put(pre);
  return SCAN_OK;
}

int lsh_apply(const scan_lsh_params& p, int kind, const int64_t* off, const int32_t* adj,
              const int32_t* deg, int64_t n, int64_t arcs, const int32_t* row, int64_t nH,
              double* sim_csr, Pool& pool, cudaStream_t s, const double* wcsr) {
  (void)arcs;
  if (nH <= 0) return SCAN_OK;
  int32_t* hlist = pool.tmp<int32_t>(nH);
  int32_t* pieces = pool.tmp<int32_t>(nH);
  int64_t* ipre = pool.tmp<int64_t>(nH + 1);
  if (!hlist || !pieces || !ipre) return SCAN_ENOMEM;
  k_hlist<<<(unsigned)std::min<int64_t>((n + 255) / 256, sm_count() * 32), 256, 0, s>>>(
      row, deg, n, hlist, pieces);
  GS_LAUNCH();
  GS_TRY(exclusive_scan_i32_to_i64(pieces, ipre, nH, pool, s));
  const unsigned gh = (unsigned)std::min<int64_t>(nH, sm_count() * 16);
  if (kind == SCAN_COSINE) {
    const int k = p.simhash_bits, W = k / 64;
    const uint64_t key = mix64(p.seed ^ 0x53494D48ULL);  // "SIMH"
    uint64_t* sig = pool.tmp<uint64_t>((size_t)nH * W);
    double* tab = pool.tmp<double>((size_t)k + 1);
    if (!sig || !tab) return SCAN_ENOMEM;
    std::vector<double> htab((size_t)k + 1);
    for (int h = 0; h <= k; ++h) {
      const double c = std::cos(M_PI * (double)h / (double)k);
      htab[h] = c > 0.0 ? c : 0.0;
    }
    GS_CUDA(cudaMemcpyAsync(tab, htab.data(), sizeof(double) * (k + 1), cudaMemcpyHostToDevice, s));
    if (wcsr) {
      const size_t smem = (size_t)SH_T * W * sizeof(uint64_t);
      GS_CUDA(cudaFuncSetAttribute(k_simhash_w, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)(SH_T * SH_WMAX * sizeof(uint64_t))));
      k_simhash_w<<<gh, SH_T, smem, s>>>(off, adj, hlist, nH, W, key, wcsr, sig);
      GS_LAUNCH();
    } else {
      uint32_t* sig32 = reinterpret_cast<uint32_t*>(sig);
      // the few long rows first: their CTAs run beside the warps' rows
      k_simhash_long<<<(unsigned)std::min<int64_t>(nH, sm_count() * 16), SHL_T, 0, s>>>(
          off, adj, hlist, nH, W, key, sig32);
      GS_LAUNCH();
      k_simhash<<<(unsigned)std::min<int64_t>((nH + 7) / 8, sm_count() * 32), SH_T, 0, s>>>(
          off, adj, hlist, nH, W, key, sig32);
      GS_LAUNCH();
    }
    GS_TRY(launch_sims<true>(off, adj, row, hlist, nH, ipre, 2 * W,
                             reinterpret_cast<const uint32_t*>(sig), tab, k, 0, sim_csr, s));
    GS_CUDA(cudaStreamSynchronize(s));  // the host table must outlive the copy
    pool.put(sig);
    pool.put(tab);
  } else {
    const int k = p.minhash_k;
    int L = 0;
    while ((1 << L) < k) ++L;
    const uint64_t key = mix64(p.seed ^ 0x4D494E48ULL);  // "MINH"
    uint32_t* mh = pool.tmp<uint32_t>((size_t)nH * k);
    if (!mh) return SCAN_ENOMEM;
    k_minhash<<<gh, 256, 0, s>>>(off, adj, hlist, nH, k, L, p.minhash_kpartition, key, mh);
    GS_LAUNCH();
    GS_TRY(launch_sims<false>(off, adj, row, hlist, nH, ipre, k, mh, nullptr, k,
                              p.minhash_kpartition, sim_csr, s));
    pool.put(mh);
  }
  pool.put(hlist);
  pool.put(pieces);
  pool.put(ipre);
  return SCAN_OK;
}

}  // namespace gscan
