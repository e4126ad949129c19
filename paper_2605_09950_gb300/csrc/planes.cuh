// Device functions shared by record.cu and column.cu: packed class histograms,
// their prefix sums, float scores and exact comparisons.
#pragma once
#include "split.cuh"

namespace bgb {

namespace {

// Packed class weights: F = 2 classes of 16 bits or 3 of 10 bits a word (class
// c in field c % F of word c / F), W words a bin.
template <int CM, int ROWS>
struct Pack {
  static constexpr int F = ROWS <= 256 ? 3 : 2;
  static constexpr int BITS = F == 3 ? 10 : 16;
  static constexpr uint32_t MASK = (1u << BITS) - 1u;
  static constexpr int W = (CM + F - 1) / F;
  // a row's word: its weight in its class's field, and the class's word in bits 30..31
  static __device__ __forceinline__ uint32_t row(uint32_t e) {
    const uint32_t y = ent_y(e), w = y / F;
    return (ent_w<0>(e) << (BITS * (y - w * F))) | (w << 30);
  }
  static __device__ __forceinline__ uint32_t field(const uint32_t (&cum)[W], int c) {
    return (cum[c / F] >> (BITS * (c % F))) & MASK;
  }
};

// exact float of v < 2^16
__device__ __forceinline__ float u16_to_float(uint32_t v) { return __uint_as_float(0x4B000000u | v) - 8388608.0f; }

// A node's totals as the scores take them.
template <int CM>
struct Totals {
  uint32_t n, cp[CM];
  float fn, fcp[CM];
};

// Float score of the candidate whose left counts are cum (0: no decrease).
template <int CM, int ROWS>
__device__ __forceinline__ float plane_score(const uint32_t (&cum)[Pack<CM, ROWS>::W], const Totals<CM>& T) {
  using P = Pack<CM, ROWS>;
  float s = 0.0f;
  if (ROWS > 1024) {  // |q| < 2^30: exact modulo 2^32
    uint32_t l[CM], nL = 0u;
#pragma unroll
    for (int c = 0; c < CM; ++c) nL += l[c] = P::field(cum, c);
#pragma unroll
    for (int c = 0; c < (CM == 2 ? 1 : CM); ++c) {
      const float q = static_cast<float>(static_cast<int32_t>(l[c] * T.n - T.cp[c] * nL));
      s = fmaf(q, q, s);
    }
    const float den = u16_to_float(nL) * u16_to_float(T.n - nL);
    return den > 0.0f ? __fdividef(s, den) : 0.0f;
  }
  float l[CM], nL = 0.0f;  // n < 4096: products below 2^24, exact
#pragma unroll
  for (int c = 0; c < CM; ++c) nL += l[c] = u16_to_float(P::field(cum, c));
#pragma unroll
  for (int c = 0; c < (CM == 2 ? 1 : CM); ++c) {
    const float q = fmaf(l[c], T.fn, -(T.fcp[c] * nL));
    s = fmaf(q, q, s);
  }
  const float den = nL * (T.fn - nL);  // 0 below the first bin that holds a row, and from the last on
  return den > 0.0f ? __fdividef(s, den) : 0.0f;
}

// sign of sa / da - sb / db
__device__ __forceinline__ int frac64_cmp(unsigned long long sa, uint32_t da, unsigned long long sb, uint32_t db) {
  const unsigned long long xh = __umul64hi(sa, db), yh = __umul64hi(sb, da);
  if (xh != yh) return xh > yh ? 1 : -1;
  const unsigned long long x = sa * db, y = sb * da;
  return x == y ? 0 : (x > y ? 1 : -1);
}

template <int CM, int ROWS>
struct RecordBest {
  unsigned long long s = 0ull;
  uint32_t den = 1u, key = 0xFFFFFFFFu, slot = 0u;
  uint32_t cum[Pack<CM, ROWS>::W];
};

// Inclusive prefix sums of the lane's bpl bins of a built histogram.
template <int CM, int ROWS>
__device__ __forceinline__ void record_prefix(const uint32_t* hw, int bpl, uint32_t (&h)[Pack<CM, ROWS>::W][8]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int w = 0; w < Pack<CM, ROWS>::W; ++w) {
    ld_bins(hw + 256 * w + lane * bpl, bpl, h[w]);
#pragma unroll
    for (int q = 1; q < 8; ++q) h[w][q] += h[w][q - 1];
    const uint32_t pre = warp_excl_scan_u32(h[w][7], lane);
#pragma unroll
    for (int q = 0; q < 8; ++q) h[w][q] += pre;
  }
}

template <int CM, int ROWS>
__device__ __forceinline__ void record_zero(uint32_t* hw, int bpl) {
  const uint32_t zero[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll
  for (int w = 0; w < Pack<CM, ROWS>::W; ++w) st_bins(hw + 256 * w + (threadIdx.x & 31) * bpl, bpl, zero);
  __syncwarp();
}

// Exact comparison of a built histogram's candidates with the lanes' bests.
template <int CM, int ROWS>
__device__ __forceinline__ void record_best(const uint32_t* hw, int bpl, uint32_t n, const uint32_t* cp, uint32_t key,
                                            uint32_t slot, RecordBest<CM, ROWS>& best) {
  using P = Pack<CM, ROWS>;
  const int lane = threadIdx.x & 31;
  uint32_t h[P::W][8];
  record_prefix<CM, ROWS>(hw, bpl, h);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    if (q >= bpl) break;
    uint32_t cum[P::W], nL = 0u, l[CM];
#pragma unroll
    for (int w = 0; w < P::W; ++w) cum[w] = h[w][q];
#pragma unroll
    for (int c = 0; c < CM; ++c) nL += l[c] = P::field(cum, c);
    if (nL == 0u || nL >= n) continue;
    unsigned long long s = 0ull;
#pragma unroll
    for (int c = 0; c < CM; ++c) {
      const long long x = static_cast<int32_t>(l[c] * n - cp[c] * nL);  // |x| < 2^30: exact modulo 2^32
      s += static_cast<unsigned long long>(x * x);
    }
    const uint32_t den = nL * (n - nL), k = key | static_cast<uint32_t>(lane * bpl + q);
    const int c = frac64_cmp(s, den, best.s, best.den);
    if (c > 0 || (c == 0 && k < best.key)) {
      best.s = s;
      best.den = den;
      best.key = k;
      best.slot = slot;
#pragma unroll
      for (int w = 0; w < P::W; ++w) best.cum[w] = cum[w];
    }
  }
}

// Best of the warp's lanes, in all of them.
template <int CM, int ROWS>
__device__ __forceinline__ void record_reduce(RecordBest<CM, ROWS>& best) {
  constexpr int W = Pack<CM, ROWS>::W;
#pragma unroll
  for (int m = 1; m < 32; m <<= 1) {
    const unsigned long long os = __shfl_xor_sync(kFull, best.s, m);
    const uint32_t od = __shfl_xor_sync(kFull, best.den, m), ok = __shfl_xor_sync(kFull, best.key, m),
                   ot = __shfl_xor_sync(kFull, best.slot, m);
    uint32_t oc[W];
#pragma unroll
    for (int w = 0; w < W; ++w) oc[w] = __shfl_xor_sync(kFull, best.cum[w], m);
    const int c = frac64_cmp(os, od, best.s, best.den);
    if (c > 0 || (c == 0 && ok < best.key)) {
      best.s = os;
      best.den = od;
      best.key = ok;
      best.slot = ot;
#pragma unroll
      for (int w = 0; w < W; ++w) best.cum[w] = oc[w];
    }
  }
}

}  // namespace

}  // namespace bgb
