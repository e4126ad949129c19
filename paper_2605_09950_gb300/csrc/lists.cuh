// A level's lists of active nodes by the kernel that splits them.
#pragma once
#include "engine.cuh"

namespace bgb {

namespace {

// The list of an active node of len rows and weight n: 1 `small` (17..32 rows,
// or all above 8 of threebin.cu), 2 `big` (column gathers), 3 tiny (9..16 rows,
// the end of `small`), 4 `micro` (<= 8 rows), 5 `mid` (classification: 33..64
// rows, or fewer with a weight above kFewWeight), 6 `rec`, 7 and 8 the start
// and the end of `rec2`.
__device__ __forceinline__ int node_class(const Dev& d, uint32_t len, uint32_t n) {
  const int cls = len > kFewRows ? 2 : (len > 16u ? 1 : (len > 8u ? 3 : 4));
  if (d.kind != 0) {
    if (d.three_bins) return len >= kThreeRows ? 2 : (len > 8u ? 1 : 4);
    if (cls == 2 && len <= d.rec_rows) return len > 256u ? 7 : 6;
    return cls;
  }
  if (len <= kMidRows && (cls == 2 || n > kFewWeight)) return 5;
  if (cls != 2 || n >= 65536u) return cls;
  if (d.columns) return len <= 256u && n < 1024u ? 6 : 7;
  if (len > d.rec_rows) return 2;
  // by record: 10-bit counts, exact f32 products below weight 4096, 16-bit counts
  return len <= 256u && n < 1024u ? 6
         : len <= 1024u && n < 4096u ? (d.rec_rows > 256u ? 7 : 2)
                                     : (d.rec_rows > 1024u ? 8 : 2);
}

__device__ __forceinline__ uint32_t* list_count(const Dev& d, int level, int cls) {
  switch (cls) {
    case 1: return &d.nsmall[level];
    case 2: return &d.work[level];
    case 3: return &d.ntiny[level];
    case 4: return &d.nmicro[level];
    case 5: return &d.nmid[level];
    default: return &d.nrec[3 * level + cls - 6];
  }
}

__device__ __forceinline__ void list_put(const Dev& d, int cls, uint32_t at, uint32_t k) {
  switch (cls) {
    case 1: d.small[at] = k; break;
    case 2: d.big[at] = k; break;
    case 3: d.small[d.small_cap - 1u - at] = k; break;
    case 4: d.micro[at] = k; break;
    case 5: d.mid[at] = k; break;
    case 6: d.rec[at] = k; break;
    case 7: d.rec2[at] = k; break;
    case 8: d.rec2[d.rec2_cap - 1u - at] = k; break;
    default: break;
  }
}

// Appends nodes k and k + 1 to the level's lists of their classes (0: none);
// all lanes of the warp together, one atomic per class and warp, all classes'
// at once.  Siblings stay neighbours: their rows share cache lines, and so do
// the nodes that a warp of the split kernels takes together.
__device__ __forceinline__ void list_pair(const Dev& d, int level, int cls0, int cls1, uint32_t k) {
  const int lane = static_cast<int>(threadIdx.x & 31u);
  const unsigned lt = (1u << lane) - 1u;
  uint32_t n = 0u, at0 = 0u, at1 = 0u;
#pragma unroll
  for (int c = 1; c <= 8; ++c) {
    const unsigned m0 = __ballot_sync(0xFFFFFFFFu, cls0 == c), m1 = __ballot_sync(0xFFFFFFFFu, cls1 == c);
    const uint32_t before = static_cast<uint32_t>(__popc(m0 & lt) + __popc(m1 & lt));
    if (lane == c) n = static_cast<uint32_t>(__popc(m0) + __popc(m1));
    if (cls0 == c) at0 = before;
    if (cls1 == c) at1 = before + (cls0 == c ? 1u : 0u);
  }
  const uint32_t first = n > 0u ? atomicAdd(list_count(d, level, lane), n) : 0u;
  at0 += __shfl_sync(0xFFFFFFFFu, first, cls0);
  at1 += __shfl_sync(0xFFFFFFFFu, first, cls1);
  list_put(d, cls0, at0, k);
  list_put(d, cls1, at1, k + 1u);
}

}  // namespace

}  // namespace bgb
