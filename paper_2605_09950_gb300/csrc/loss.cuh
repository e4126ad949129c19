// Losses of Alg. 3 between the leaf of a row and the leaf of its re-walk.
#pragma once
#include "engine.cuh"

namespace bgb {

namespace {

// loss between the unpermuted leaf q and the permuted leaf q2
__device__ double loss64(const Dev& d, uint32_t q, uint32_t q2) {
  const double na = static_cast<double>(d.nd_n[q]), nb = static_cast<double>(d.nd_n[q2]);
  if (d.kind != 0) {
    const double ma = static_cast<double>(d.nd_S[q]) / na, mb = static_cast<double>(d.nd_S[q2]) / nb;
    const double df = (ma - mb) * 0x1p-20;
    return df * df;
  }
  const double eps = d.kl_eps;
  const double norm = 1.0 + static_cast<double>(d.C) * eps;
  double kl = 0.0;
  for (int c = 0; c < d.C; ++c) {
    const double pa = (static_cast<double>(d.nd_cnt[static_cast<int64_t>(q) * d.C + c]) / na + eps) / norm;
    const double pb = (static_cast<double>(d.nd_cnt[static_cast<int64_t>(q2) * d.C + c]) / nb + eps) / norm;
    kl += pa * log(pa / pb);
  }
  return kl;
}

// phi(r) = r log r - r + 1 >= 0, accurate near r = 1 (series in r - 1)
__device__ __forceinline__ float kl_phi(float r) {
  const float dl = r - 1.0f;
  if (fabsf(dl) < 0.25f) {
    // dl^2 * sum_{n=2..14} (-1)^n dl^(n-2) / (n (n-1)), by Horner
    constexpr float c[13] = {1.0f / 2,   -1.0f / 6,   1.0f / 12,   -1.0f / 20,  1.0f / 30,
                             -1.0f / 42, 1.0f / 56,   -1.0f / 72,  1.0f / 90,   -1.0f / 110,
                             1.0f / 132, -1.0f / 156, 1.0f / 182};
    float s = c[12];
#pragma unroll
    for (int m = 11; m >= 0; --m) s = s * dl + c[m];
    return s * (dl * dl);
  }
  return r * logf(r) - dl;
}

__device__ float loss32(const Dev& d, uint32_t q, uint32_t q2) {
  const uint32_t na = d.nd_n[q], nb = d.nd_n[q2];
  if (d.kind != 0) {
    // mean difference from exact integers: (S_a n_b - S_b n_a) / (n_a n_b)
    const __int128 num = static_cast<__int128>(d.nd_S[q]) * nb - static_cast<__int128>(d.nd_S[q2]) * na;
    const u128 mag = num < 0 ? static_cast<u128>(-num) : static_cast<u128>(num);
    const uint64_t ml[2] = {static_cast<uint64_t>(mag), static_cast<uint64_t>(mag >> 64)};
    const uint64_t den = static_cast<uint64_t>(na) * nb;
    const float df = __fdiv_rn(limbs_to_float(ml, 2, -20), limbs_to_float(&den, 1, 0));
    return df * df;
  }
  const float eps = static_cast<float>(d.kl_eps);
  const float norm = 1.0f + static_cast<float>(d.C) * eps;
  float kl = 0.0f;
  for (int c = 0; c < d.C; ++c) {
    const float pa = __fdiv_rn(__fdiv_rn(static_cast<float>(d.nd_cnt[static_cast<int64_t>(q) * d.C + c]),
                                         static_cast<float>(na)) + eps, norm);
    const float pb = __fdiv_rn(__fdiv_rn(static_cast<float>(d.nd_cnt[static_cast<int64_t>(q2) * d.C + c]),
                                         static_cast<float>(nb)) + eps, norm);
    kl += pb * kl_phi(__fdiv_rn(pa, pb));
  }
  return kl;
}

}  // namespace

}  // namespace bgb
