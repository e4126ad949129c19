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

// Appends node k to the level's list of its class (0: none); all lanes of the
// warp together, one atomic per class and warp, all classes' at once.
__device__ __forceinline__ void list_node(const Dev& d, int level, int cls, uint32_t k) {
  const int lane = static_cast<int>(threadIdx.x & 31u);
  const unsigned same = __match_any_sync(0xFFFFFFFFu, cls);
  const int leader = __ffs(static_cast<int>(same)) - 1;
  uint32_t* count = nullptr;
  switch (cls) {
    case 1: count = &d.nsmall[level]; break;
    case 2: count = &d.work[level]; break;
    case 3: count = &d.ntiny[level]; break;
    case 4: count = &d.nmicro[level]; break;
    case 5: count = &d.nmid[level]; break;
    case 6: case 7: case 8: count = &d.nrec[3 * level + cls - 6]; break;
    default: break;
  }
  uint32_t at = 0u;
  if (count && lane == leader) at = atomicAdd(count, static_cast<uint32_t>(__popc(same)));
  at = __shfl_sync(0xFFFFFFFFu, at, leader) + __popc(same & ((1u << lane) - 1u));
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

}  // namespace

}  // namespace bgb
