// Device functions shared by the split kernels (split.cu: nodes of many rows;
// small.cu: nodes of few rows): row entries, exact candidate scores, the
// record of a chosen split.
#pragma once
#include <cstdint>

#include "engine.cuh"

namespace bgb {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

// Class count of a variant: the kernels are instantiated with CM = 3, 4 and 5
// for exactly that many classes (their class loops then unroll to the real
// count), CM = 2 for one or two classes and CM = 8 for six to eight.
template <int CM>
__device__ __forceinline__ int ncls(const Dev& d) {
  return (CM == 3 || CM == 4 || CM == 5) ? CM : d.C;
}

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

__device__ __forceinline__ const uint8_t* column(const Dev& d, uint32_t f) {
  return d.Xaug + static_cast<int64_t>(f) * d.ldN;
}

// The bin of one row and column for a node's row-by-row reads, from the
// row-major copy: a row's sampled columns then share its few kilobytes
// instead of lying a column apart.
__device__ __forceinline__ uint32_t row_bin(const Dev& d, uint32_t row, uint32_t f) {
  return d.Xrow[static_cast<int64_t>(row) * d.ldP + f];
}

// L2 residency in the histogram kernels.  The bins are gathered band by band
// (the groups are sorted by feature band), and a band's columns must stay in
// L2 while its groups run; the nodes' row entries, streamed once per feature
// group, would otherwise push them out.  So the gathers carry an evict-last
// policy and the entry reads are streaming (evict-first) loads.
__device__ __forceinline__ uint64_t keep_policy() {
  uint64_t p;
  asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}

__device__ __forceinline__ uint32_t ld_keep(const uint8_t* a, uint64_t pol) {
  uint32_t v;
  asm("ld.global.L2::cache_hint.u8 %0, [%1], %2;" : "=r"(v) : "l"(a), "l"(pol));
  return v;
}

__device__ __forceinline__ uint32_t ld_stream(const uint32_t* a) { return __ldcs(a); }

__device__ __forceinline__ void prefetch_l2(const void* a) { asm volatile("prefetch.global.L2 [%0];" ::"l"(a)); }

// Row entries: row << 8 | low byte.  Classification: low byte = y << 5 | w
// (label < 8, bootstrap count < 32); regression: low byte = w (< 256).
template <int KIND>
__device__ __forceinline__ uint32_t ent_w(uint32_t e) {
  return KIND == 0 ? (e & 31u) : (e & 255u);
}
__device__ __forceinline__ uint32_t ent_y(uint32_t e) { return (e >> 5) & 7u; }

template <int CM>
struct Cand {
  U192 num;
  uint64_t den;
  uint32_t key;
  uint32_t nL;
  uint32_t cL[CM];
  long long SL;
  int32_t feat;
  int32_t bin;
  bool valid;
};

template <int CM>
__device__ __forceinline__ bool better(const Cand<CM>& a, const Cand<CM>& b) {
  if (!a.valid) return false;
  if (!b.valid) return true;
  const int c = frac_cmp(a.num, a.den, b.num, b.den);
  if (c != 0) return c > 0;
  return a.key < b.key;
}

__device__ __forceinline__ U192 u192_mul(u128 a, uint64_t b) {
  const u128 lo = static_cast<u128>(static_cast<uint64_t>(a)) * b;
  const u128 hi = static_cast<u128>(static_cast<uint64_t>(a >> 64)) * b + (lo >> 64);
  U192 r;
  r.w[0] = static_cast<uint64_t>(lo);
  r.w[1] = static_cast<uint64_t>(hi);
  r.w[2] = static_cast<uint64_t>(hi >> 64);
  return r;
}

__device__ __forceinline__ U192 u192_add(const U192& a, const U192& b) {
  U192 r;
  u128 s = static_cast<u128>(a.w[0]) + b.w[0];
  r.w[0] = static_cast<uint64_t>(s);
  s = static_cast<u128>(a.w[1]) + b.w[1] + (s >> 64);
  r.w[1] = static_cast<uint64_t>(s);
  r.w[2] = a.w[2] + b.w[2] + static_cast<uint64_t>(s >> 64);
  return r;
}

__device__ __forceinline__ u128 sq_i64(long long v) {
  const uint64_t m = v < 0 ? 0ull - static_cast<uint64_t>(v) : static_cast<uint64_t>(v);
  return static_cast<u128>(m) * m;
}

template <int CM>
struct NodeInfo {
  int64_t base;  // tree row-buffer offset + segment offset
  uint32_t len, n;
  uint32_t cp[CM];
  long long SP;
};

// ---- scores
// Exact u32 -> float for v < 2^24 on the integer and FP32 pipes: the bits
// 0x4B000000 | m are the float 2^23 + m for m < 2^23.
__device__ __forceinline__ float u24_to_float(uint32_t v) {
  const float b = __uint_as_float(0x4B000000u | (v & 0x7FFFFFu));
  return (v & 0x800000u) ? b : b - 8388608.0f;
}

// |v| as float for a 64-bit v, from three exact 22-bit pieces (all terms
// non-negative: relative error below 2^-22)
__device__ __forceinline__ float abs_i64_to_float(long long v) {
  const uint64_t a = v < 0 ? 0ull - static_cast<uint64_t>(v) : static_cast<uint64_t>(v);
  return (u24_to_float(static_cast<uint32_t>(a >> 44)) * 17592186044416.0f +
          u24_to_float(static_cast<uint32_t>(a >> 22) & 0x3FFFFFu) * 4194304.0f) +
         u24_to_float(static_cast<uint32_t>(a) & 0x3FFFFFu);
}

// Float scores of the pre-screen (counts and n below 2^24, so the integer
// inputs convert exactly).  Relative error below 2^-20.
template <int CM>
__device__ __forceinline__ float score_class_f(const uint32_t* cl, const uint32_t* cp, int C, uint32_t nL,
                                               uint32_t n) {
  float AL = 0.0f, AR = 0.0f;
#pragma unroll
  for (int k = 0; k < CM; ++k)
    if (k < C) {
      const float l = u24_to_float(cl[k]), r = u24_to_float(cp[k] - cl[k]);
      AL += l * l;
      AR += r * r;
    }
  return __fdividef(AL, u24_to_float(nL)) + __fdividef(AR, u24_to_float(n - nL));
}

__device__ __forceinline__ float score_reg_f(long long SL, long long SP, uint32_t nL, uint32_t n) {
  const float l = abs_i64_to_float(SL), r = abs_i64_to_float(SP - SL);
  return __fdividef(l * l, u24_to_float(nL)) + __fdividef(r * r, u24_to_float(n - nL));
}

// The same for sums below 2^53 (|y| < 2^33): a signed high part and 22 exact low
// bits, without the sign and with half the instructions.
__device__ __forceinline__ float i53_to_float(long long v) {
  const float lo = __uint_as_float(0x4B000000u | (static_cast<uint32_t>(v) & 0x3FFFFFu)) - 8388608.0f;
  return fmaf(static_cast<float>(static_cast<int32_t>(v >> 22)), 4194304.0f, lo);
}

__device__ __forceinline__ float score_reg_narrow(long long SL, long long SP, uint32_t nL, uint32_t n) {
  const float l = i53_to_float(SL), r = i53_to_float(SP - SL);
  return __fdividef(l * l, u24_to_float(nL)) + __fdividef(r * r, u24_to_float(n - nL));
}

// wide: whether a sum may reach 2^53 (uniform)
__device__ __forceinline__ float score_reg_any(bool wide, long long SL, long long SP, uint32_t nL, uint32_t n) {
  return wide ? score_reg_f(SL, SP, nL, n) : score_reg_narrow(SL, SP, nL, n);
}

template <int CM>
__device__ __forceinline__ void make_class(Cand<CM>& c, const uint32_t* cl, const uint32_t* cp, int C,
                                           uint32_t nL, uint32_t n) {
  uint64_t AL = 0, AR = 0;
#pragma unroll
  for (int k = 0; k < CM; ++k) {
    c.cL[k] = k < C ? cl[k] : 0u;
    if (k < C) {
      const uint64_t l = cl[k], r = cp[k] - cl[k];
      AL += l * l;
      AR += r * r;
    }
  }
  const uint32_t nR = n - nL;
  c.num = u192_from(static_cast<u128>(AL) * nR + static_cast<u128>(AR) * nL);
  c.den = static_cast<uint64_t>(nL) * nR;
  c.nL = nL;
  c.SL = 0;
  c.valid = true;
}

template <int CM>
__device__ __forceinline__ void make_reg(Cand<CM>& c, long long SL, long long SP, uint32_t nL, uint32_t n) {
  const uint32_t nR = n - nL;
  c.num = u192_add(u192_mul(sq_i64(SL), nR), u192_mul(sq_i64(SP - SL), nL));
  c.den = static_cast<uint64_t>(nL) * nR;
  c.nL = nL;
  c.SL = SL;
#pragma unroll
  for (int k = 0; k < CM; ++k) c.cL[k] = 0u;
  c.valid = true;
}

// Relative window of the float pre-screen.  A float score is within 2^-20 of
// the exact score, so every candidate whose exact score is the maximum has a
// float score above (1 - 2^-16) * (best float score); only those are compared
// exactly.
__device__ __forceinline__ float screen(float m) { return m - m * 0.0000152587890625f; }

// all lanes: out = best of the lane candidates flagged valid
template <int KIND, int CM>
__device__ void warp_select(const Cand<CM>& mine, Cand<CM>& out) {
  unsigned m = __ballot_sync(kFull, mine.valid);
  out.valid = false;
  while (m) {
    const int l = __ffs(m) - 1;
    m &= m - 1;
    Cand<CM> c;
    c.num.w[0] = __shfl_sync(kFull, mine.num.w[0], l);
    c.num.w[1] = __shfl_sync(kFull, mine.num.w[1], l);
    c.num.w[2] = __shfl_sync(kFull, mine.num.w[2], l);
    c.den = __shfl_sync(kFull, mine.den, l);
    c.key = __shfl_sync(kFull, mine.key, l);
    c.nL = __shfl_sync(kFull, mine.nL, l);
    c.feat = __shfl_sync(kFull, mine.feat, l);
    c.bin = __shfl_sync(kFull, mine.bin, l);
    if (KIND == 1) {
      c.SL = __shfl_sync(kFull, mine.SL, l);
#pragma unroll
      for (int k = 0; k < CM; ++k) c.cL[k] = 0u;
    } else {
      c.SL = 0;
#pragma unroll
      for (int k = 0; k < CM; ++k) c.cL[k] = __shfl_sync(kFull, mine.cL[k], l);
    }
    c.valid = true;
    if (better(c, out)) out = c;
  }
}

// Exact impurity decrease of the chosen split:
//   delta = num/den - A_P/n_P = (num*n_P - A_P*den) / (den*n_P), rounded as
//   RN(numerator) / RN(denominator) in the working precision.
template <int KIND, int CM>
__device__ bool split_delta(const Cand<CM>& c, const NodeInfo<CM>& nd, int C, int precision, double* delta) {
  u128 AP = 0;
  if (KIND == 1) {
    AP = sq_i64(nd.SP);
  } else {
#pragma unroll
    for (int k = 0; k < CM; ++k)
      if (k < C) AP += static_cast<u128>(static_cast<uint64_t>(nd.cp[k]) * nd.cp[k]);
  }
  uint64_t lhs[4], rhs[4];
  mul192x64(c.num, nd.n, lhs);
  mul192x64(u192_from(AP), c.den, rhs);
  if (cmp_limbs4(lhs, rhs) <= 0) return false;
  uint64_t dn[4];
  uint64_t borrow = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint64_t a = lhs[i], b = rhs[i];
    const uint64_t t = a - b;
    const uint64_t b1 = a < b;
    dn[i] = t - borrow;
    const uint64_t b2 = t < borrow;
    borrow = b1 | b2;
  }
  const u128 dd = static_cast<u128>(c.den) * nd.n;
  const uint64_t dl[2] = {static_cast<uint64_t>(dd), static_cast<uint64_t>(dd >> 64)};
  if (precision == 0)
    *delta = limbs_to_double(dn, 4, 0) / limbs_to_double(dl, 2, 0);
  else
    *delta = static_cast<double>(__fdiv_rn(limbs_to_float(dn, 4, 0), limbs_to_float(dl, 2, 0)));
  return true;
}

// Records the split of node k (or marks it a leaf); one thread.
template <int KIND, int CM>
__device__ uint32_t commit_split(const Dev& d, uint32_t k, const Cand<CM>& b, const NodeInfo<CM>& nd) {
  double delta = 0.0;
  uint32_t sp = kLeaf;
  if (b.valid && split_delta<KIND, CM>(b, nd, ncls<CM>(d), d.precision, &delta)) {
    sp = (static_cast<uint32_t>(b.feat) << 8) | static_cast<uint32_t>(b.bin);
    d.nd_delta[k] = delta;
    d.nd_ln[k] = b.nL;
    if (KIND == 1) {
      d.nd_lS[k] = b.SL;
    } else {
#pragma unroll
      for (int c = 0; c < CM; ++c)
        if (c < ncls<CM>(d)) d.nd_lcnt[static_cast<int64_t>(k) * d.C + c] = b.cL[c];
    }
    if (!d.permut) {  // Alg. 2: this node's gain x samples, summed exactly per (tree, feature)
      if (!csa_add(d.acc + (static_cast<int64_t>(d.nd_tree[k]) * d.p_aug + b.feat) * kCsaLimbs, delta))
        atomicOr(&d.status[0], kErrAcc);
    }
  }
  d.nd_split[k] = sp;
  return sp;
}

// Record of a split given by its counts: s / (n_L n_R n), s = sum_k q_k^2,
// q_k = l_k n - c_k n_L, is the impurity decrease, its
// numerator and denominator exact (the general form's numerator
// num n_P - A_P den equals s), each rounded once.  cL: left class counts.
template <int CM>
__device__ __noinline__ uint32_t commit_counts(const Dev& d, uint32_t k, bool valid, uint32_t feat, uint32_t bin, uint32_t nL,
                                  const uint32_t (&cL)[CM], unsigned long long s, uint32_t n) {
  uint32_t sp = kLeaf;
  if (valid) {
    const unsigned long long den = static_cast<unsigned long long>(nL) * (n - nL) * n;
    const double delta = d.precision == 0
                             ? __ull2double_rn(s) / __ull2double_rn(den)
                             : static_cast<double>(__fdiv_rn(__ull2float_rn(s), __ull2float_rn(den)));
    sp = (feat << 8) | bin;
    d.nd_delta[k] = delta;
    d.nd_ln[k] = nL;
#pragma unroll
    for (int c = 0; c < CM; ++c)
      if (c < ncls<CM>(d)) d.nd_lcnt[static_cast<int64_t>(k) * d.C + c] = cL[c];
    if (!d.permut) {  // Alg. 2: this node's gain x samples, summed exactly per (tree, feature)
      if (!csa_add(d.acc + (static_cast<int64_t>(d.nd_tree[k]) * d.p_aug + feat) * kCsaLimbs, delta))
        atomicOr(&d.status[0], kErrAcc);
    }
  }
  d.nd_split[k] = sp;
  return sp;
}

template <int KIND, int CM>
__device__ bool load_node(const Dev& d, uint32_t k, int level, NodeInfo<CM>& nd) {
  const uint32_t tau = d.nd_tree[k];
  nd.base = static_cast<int64_t>(tau) * d.N + d.nd_seg[k];
  nd.len = d.nd_len[k];
  nd.n = d.nd_n[k];
  nd.SP = 0;
  bool pure = false;
#pragma unroll
  for (int c = 0; c < CM; ++c) {
    nd.cp[c] = 0u;
    if (KIND == 0 && c < d.C) {
      nd.cp[c] = d.nd_cnt[static_cast<int64_t>(k) * d.C + c];
      pure |= nd.cp[c] == nd.n;
    }
  }
  if (KIND == 1) nd.SP = d.nd_S[k];
  return level < d.D && nd.len >= 2u && !pure;
}

__device__ __forceinline__ void node_perm(const Dev& d, uint32_t k, Perm& P) {
  perm_init(P, static_cast<uint32_t>(d.p_aug), d.seed, d.nd_heap[k], unit_word(d.t, d.nd_tree[k]),
            purpose_word(kPurposeMtry, d.job));
}

// Stable partition of a node's rows by warp: left rows in order from the
// front, right rows in order from the back (reversed); 8 gathers per lane
// in flight.  Returns the number of left rows.
__device__ uint32_t warp_partition(const Dev& d, int64_t base, uint32_t len, uint32_t sp, const uint32_t* rows_in,
                                   uint32_t* rows_out) {
  const int lane = threadIdx.x & 31;
  const uint8_t* col = column(d, sp >> 8);
  const uint32_t thr = sp & 255u;
  uint32_t lbase = 0, rbase = 0;
  const uint32_t lt = lanemask_lt();
  for (uint32_t r0 = 0; r0 < len; r0 += 256) {
    uint32_t e[8], b[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const uint32_t r = r0 + q * 32 + lane;
      e[q] = r < len ? rows_in[base + r] : 0u;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const uint32_t r = r0 + q * 32 + lane;
      b[q] = r < len ? col[e[q] >> 8] : 0u;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const bool v = r0 + q * 32 + lane < len;
      const bool gl = v && b[q] <= thr, gr = v && !gl;
      const unsigned bl = __ballot_sync(kFull, gl), br = __ballot_sync(kFull, gr);
      if (gl) rows_out[base + lbase + __popc(bl & lt)] = e[q];
      if (gr) rows_out[base + len - 1u - (rbase + __popc(br & lt))] = e[q];
      lbase += __popc(bl);
      rbase += __popc(br);
    }
  }
  return lbase;
}

// Bins of a lane in histograms of one 32-bit plane of 256 words per field.
__device__ __forceinline__ int lane_bins(int B) { return B > 128 ? 8 : (B > 64 ? 4 : (B > 32 ? 2 : 1)); }

// A lane's bpl (1, 2, 4 or 8) consecutive bins of a plane, by 4, 8 or 16 bytes:
// the plane starts on a 16-byte boundary (p = plane + lane * bpl).
__device__ __forceinline__ void ld_bins(const uint32_t* p, int bpl, uint32_t (&h)[8]) {
#pragma unroll
  for (int q = 0; q < 8; ++q) h[q] = 0u;
  if (bpl >= 4) {
    const uint4 a = reinterpret_cast<const uint4*>(p)[0];
    h[0] = a.x, h[1] = a.y, h[2] = a.z, h[3] = a.w;
    if (bpl == 8) {
      const uint4 b = reinterpret_cast<const uint4*>(p)[1];
      h[4] = b.x, h[5] = b.y, h[6] = b.z, h[7] = b.w;
    }
  } else if (bpl == 2) {
    const uint2 a = *reinterpret_cast<const uint2*>(p);
    h[0] = a.x, h[1] = a.y;
  } else {
    h[0] = *p;
  }
}

__device__ __forceinline__ void st_bins(uint32_t* p, int bpl, const uint32_t (&h)[8]) {
  if (bpl >= 4) {
    reinterpret_cast<uint4*>(p)[0] = make_uint4(h[0], h[1], h[2], h[3]);
    if (bpl == 8) reinterpret_cast<uint4*>(p)[1] = make_uint4(h[4], h[5], h[6], h[7]);
  } else if (bpl == 2) {
    *reinterpret_cast<uint2*>(p) = make_uint2(h[0], h[1]);
  } else {
    *p = h[0];
  }
}

// Stable partition of a node's rows by a block: left rows in order, then right
// rows in order.  Warp w holds in e[i] the entries of rows (w + WARPS i) 32 ..;
// goes_left(i, r) is asked for rows below len; left: a word of shared memory
// per 32 rows.  Returns the number of left rows.
template <int CH, int WARPS, typename F>
__device__ __forceinline__ uint32_t block_partition(const uint32_t (&e)[CH], uint32_t len, int64_t base, uint32_t* out,
                                                    uint32_t* left, F&& goes_left) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t chunks = (len + 31u) / 32u;
  unsigned bl[CH];
#pragma unroll
  for (int i = 0; i < CH; ++i) {
    const uint32_t c = warp + WARPS * i, r = c * 32u + lane;
    bl[i] = 0u;
    if (c < chunks) {
      bl[i] = __ballot_sync(kFull, r < len && goes_left(i, r));
      if (lane == 0) left[c] = __popc(bl[i]);
    }
  }
  __syncthreads();
  uint32_t total = 0u, before[CH];
#pragma unroll
  for (int i = 0; i < CH; ++i) before[i] = 0u;
  for (uint32_t c0 = 0; c0 < chunks; c0 += 32u) {
    const uint32_t v = c0 + lane < chunks ? left[c0 + lane] : 0u;
    const uint32_t x = total + warp_excl_scan_u32(v, lane);
#pragma unroll
    for (int i = 0; i < CH; ++i) {
      const uint32_t c = warp + WARPS * i;
      const uint32_t y = __shfl_sync(kFull, x, c & 31u);
      if (c >= c0 && c < c0 + 32u) before[i] = y;
    }
    total = __shfl_sync(kFull, x + v, 31);
  }
#pragma unroll
  for (int i = 0; i < CH; ++i) {
    const uint32_t c = warp + WARPS * i, r = c * 32u + lane;
    if (c < chunks && r < len) {
      const uint32_t l = before[i] + __popc(bl[i] & lanemask_lt());
      out[base + (((bl[i] >> lane) & 1u) ? l : total + (r - l))] = e[i];
    }
  }
  return total;
}

}  // namespace

}  // namespace bgb
