// Device functions shared by the regression kernels of threebin.cu and
// regress.cu: a lane's best candidate and its exact comparison.
#pragma once
#include "split.cuh"

namespace bgb {

namespace {

struct RegCand {
  float sf = -1.0f;
  long long S = 0;
  uint32_t nL = 0u, fb = 0xFFFFFFFFu;  // feature (or its draw slot) << 8 | threshold
};

// slot of a sampled column: the inverse permutation
__device__ __noinline__ uint32_t perm_slot(const Perm& P, uint32_t f) {
  if (P.n <= 1u) return f;
  uint32_t x = f;
  do {
    uint32_t left = x >> P.half, right = x & P.mask;
#pragma unroll
    for (int r = 7; r >= 0; --r) {
      const uint32_t prev = right ^ (murmur_fmix(left ^ P.key[r]) & P.mask);
      right = left;
      left = prev;
    }
    x = (left << P.half) | right;
  } while (x >= P.n);
  return x;
}

// whether the score of candidate a is above (1), equal to (0) or below (-1) b's
__device__ __noinline__ int reg_cmp(long long Sa, uint32_t na, long long Sb, uint32_t nb, long long SP, uint32_t n) {
  Cand<1> a, b;
  make_reg<1>(a, Sa, SP, na, n);
  make_reg<1>(b, Sb, SP, nb, n);
  return frac_cmp(a.num, a.den, b.num, b.den);
}

// P: the node's permutation, where candidates are given by column and equal
// scores go to the column drawn first
__device__ __forceinline__ void reg_offer(RegCand& b, float sf, long long S, uint32_t nL, uint32_t fb, long long SP,
                                          uint32_t n, const Perm* P) {
  if (sf < 0.0f || sf < screen(b.sf)) return;
  if (screen(sf) <= b.sf) {  // inside the window: exactly
    const bool same = (S == b.S && nL == b.nL) || (S == SP - b.S && nL == n - b.nL);  // the same partition
    const int c = same ? 0 : reg_cmp(S, nL, b.S, b.nL, SP, n);
    if (c < 0) return;
    if (c == 0) {
      if (P && (fb >> 8) != (b.fb >> 8)) {
        if (perm_slot(*P, fb >> 8) >= perm_slot(*P, b.fb >> 8)) return;
      } else if (fb >= b.fb) {
        return;
      }
    }
  }
  b.sf = sf;
  b.S = S;
  b.nL = nL;
  b.fb = fb;
}

__device__ __forceinline__ void reg_warp_best(RegCand& b, long long SP, uint32_t n, const Perm* P) {
#pragma unroll
  for (int m = 1; m < 32; m <<= 1) {
    const float sf = __shfl_xor_sync(kFull, b.sf, m);
    const long long S = __shfl_xor_sync(kFull, b.S, m);
    const uint32_t nL = __shfl_xor_sync(kFull, b.nL, m), fb = __shfl_xor_sync(kFull, b.fb, m);
    reg_offer(b, sf, S, nL, fb, SP, n, P);
  }
}

__device__ __forceinline__ uint32_t commit_reg(const Dev& d, uint32_t k, const RegCand& b, const NodeInfo<1>& nd) {
  Cand<1> c;
  c.valid = false;
  if (b.sf >= 0.0f) {
    make_reg<1>(c, b.S, nd.SP, b.nL, nd.n);
    c.feat = static_cast<int32_t>(b.fb >> 8);
    c.bin = static_cast<int32_t>(b.fb & 255u);
    c.key = 0u;
  }
  return commit_split<1, 1>(d, k, c, nd);
}

__device__ __forceinline__ uint32_t le_h2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("set.le.f16x2.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// half bits of an integer of at most 2048
__device__ __forceinline__ uint32_t half_bits(int v) {
  uint32_t r;
  asm("{.reg .b16 h; cvt.rn.f16.s32 h, %1; mov.b32 %0, {h, h};}" : "=r"(r) : "r"(v));
  return r & 0xFFFFu;
}

}  // namespace

}  // namespace bgb
