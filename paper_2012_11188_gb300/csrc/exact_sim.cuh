// Cosine (Section 3.1) and Jaccard (Section 2.1.1) of whole numbers, rounded as
// IEEE double arithmetic rounds them, without the FP64 pipe.
//
// A warp's FP64 instruction occupies a multiprocessor's two FP64 lanes for 16
// clocks, and a correctly rounded square root and division are some 18 of
// them, 290 clocks for 32 edges; the 64-bit integer form below is about 130
// instructions that issue four a clock (builds: dense graph of 25,825 vertices,
// whose similarities the matrix product's epilogue forms, 24.4 -> 22.5 ms, 512
// SBM graphs 69.8 -> 68.7; R-MAT s24 within the noise, since its similarity
// pass waits for gathers and scattered stores). Both steps are Newton's iteration in
// fixed point from a 23-bit hardware approximation, of third order, to
// some 50 bits, one correction by the remainder, and then the exact whole remainder, which
// decides the last bit: the result does not depend on how good the
// approximation was, as long as it is within 2^-21.
#pragma once

#include <stdint.h>

#ifndef __CUDA_ARCH__
#include <cmath>
#include <cstring>
#ifndef GS_ES_ERROR
#define GS_ES_ERROR 0.0f  // relative error put on the host's approximations (tests)
#endif
#endif

namespace gscan {

#ifdef __CUDACC__
#define GS_HD __host__ __device__ __forceinline__
#else
#define GS_HD inline
#endif

GS_HD uint64_t es_mulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)((unsigned __int128)a * b >> 64);
#endif
}
GS_HD int64_t es_square(int64_t x, int shift) { return x * x >> shift; }
GS_HD int es_clz(uint64_t x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return __builtin_clzll(x);
#endif
}
// 1 / sqrt(x) and 1 / x (documented to 2 units in the last place and correctly
// rounded)
GS_HD float es_rsqrt(float x) {
#ifdef __CUDA_ARCH__
  return rsqrtf(x);
#else
  return 1.0f / std::sqrt(x) * (1.0f + GS_ES_ERROR);
#endif
}
GS_HD float es_rcp(float x) {
#ifdef __CUDA_ARCH__
  return __frcp_rn(x);
#else
  return 1.0f / x * (1.0f + GS_ES_ERROR);
#endif
}
GS_HD double es_double(uint64_t bits) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)bits);
#else
  double d;
  std::memcpy(&d, &bits, 8);
  return d;
#endif
}

// RN(c / (S 2^-k)) for 1 <= c < 2^32, 2^52 <= S <= 2^53 and y = 2^115 / S (1/x
// in units of 2^-62 for x = S 2^-53) to 46 bits; yf is the same as a float near
// 1 to 2. No quotient lies half-way between two doubles: (2 Q + 1) S = c 2^j
// would make an odd number above 2^53 divide c.
GS_HD double es_divide(uint32_t c, uint64_t S, int k, uint64_t y, float yf) {
  const int lz = es_clz(c) - 11;
  const uint64_t C = (uint64_t)c << lz;  // 2^52 <= C < 2^53
  const int sh = C >= S ? 52 : 53;       // quotient of C 2^sh in [2^52, 2^53)
  uint64_t q = es_mulhi(C << 11, y) >> (62 - sh);
  // remainder: below 2^61 in magnitude, so 64 bits hold it
  int64_t r = (int64_t)((C << sh) - q * S);
  const int d = (int)((float)(int32_t)(r >> 32) * yf * 0x1p-21f);  // r / S to +-1
  q += (int64_t)d;
  r -= (int64_t)d * (int64_t)S;
  if (r < 0) { --q; r += (int64_t)S; }
  if (r < 0) { --q; r += (int64_t)S; }
  if (r >= (int64_t)S) { ++q; r -= (int64_t)S; }
  if (r >= (int64_t)S) { ++q; r -= (int64_t)S; }
  if (2 * r > (int64_t)S) ++q;
  // q 2^(k - lz - sh); q = 2^53 carries into the exponent
  return es_double(((uint64_t)(k - lz - sh + 52 + 1023) << 52) + (q - (1ull << 52)));
}

// RN(c / RN(sqrt(P))), 1 <= P < 2^62, 1 <= c < 2^32.
GS_HD double exact_cosine(uint32_t c, uint64_t P) {
  const int e = es_clz(P) & ~1;
  const uint64_t a = P << e;  // x = a 2^-64 in [1/4, 1)
  const float yf = es_rsqrt((float)(uint32_t)(a >> 32) * 0x1p-32f);
  const uint32_t y0 = (uint32_t)(yf * 0x1p30f);  // units of 2^-30
  // y = y0 (1 + t), t = h / 2 + 3 h^2 / 8 with h = 1 - x y0^2 (units of 2^-60)
  const int64_t h = (int64_t)((1ull << 60) - es_mulhi(a, (uint64_t)y0 * y0));
  const int64_t t = (h >> 1) + es_square(h >> 12, 36) * 3 / 8;
  const uint64_t y = ((uint64_t)y0 << 32) + (uint64_t)(((int64_t)y0 * (t >> 9)) >> 19);
  // m = sqrt(a) 2^21, and what a 2^42 is above m^2
  uint64_t m = es_mulhi(a, y) >> 9;
  int64_t r = (int64_t)((a << 42) - m * m);
  const int d = (int)((float)(int32_t)(r >> 32) * yf * 0x1p-22f);  // r / 2 m to +-1
  r -= (int64_t)d * (int64_t)(2 * m + (int64_t)d);
  m += (int64_t)d;
  if (r < 0) { --m; r += (int64_t)(2 * m + 1); }
  if (r < 0) { --m; r += (int64_t)(2 * m + 1); }
  if (r > (int64_t)(2 * m)) { r -= (int64_t)(2 * m + 1); ++m; }
  if (r > (int64_t)(2 * m)) { r -= (int64_t)(2 * m + 1); ++m; }
  if (r > (int64_t)m) ++m;  // nearest: the root is irrational or whole
  return es_divide(c, m, 21 + e / 2, y, yf);
}

// RN(c / D), 1 <= c, D < 2^32.
GS_HD double exact_ratio(uint32_t c, uint32_t D) {
  const int lz = es_clz(D) - 11;
  const uint64_t S = (uint64_t)D << lz;  // x = S 2^-53 in [1/2, 1)
  const uint64_t x = S << 11;
  const float yf = es_rcp((float)(uint32_t)(x >> 32) * 0x1p-32f);
  const uint32_t y0 = (uint32_t)(yf * 0x1p30f);
  // y = y0 (1 + t), t = h + h^2 with h = 1 - x y0 (units of 2^-60)
  const int64_t h = (int64_t)((1ull << 62) - es_mulhi(x, (uint64_t)y0 << 32)) >> 2;
  const int64_t t = h + es_square(h >> 12, 36);
  const uint64_t y = ((uint64_t)y0 << 32) + (uint64_t)(((int64_t)y0 * (t >> 9)) >> 19);
  return es_divide(c, S, lz, y, yf);
}

#ifdef __CUDACC__
// Cosine (SCAN_COSINE = 0) or Jaccard from the closed count and the degrees.
// The cosine is that of the product as a double: one of 2^53 or more is
// rounded before the root is taken.
__device__ __forceinline__ double sim_of(int kind, int64_t c, int64_t du, int64_t dv) {
  if (kind != 0) return exact_ratio((uint32_t)c, (uint32_t)(du + dv + 2 - c));
  const uint64_t prod = (uint64_t)(du + 1) * (uint64_t)(dv + 1);
  if (prod >> 53) return __ddiv_rn((double)c, __dsqrt_rn((double)prod));
  return exact_cosine((uint32_t)c, prod);
}
#endif

}  // namespace gscan
