// Alg. 3 on out-of-bag rows with a tree's split nodes and the rows' records in
// shared memory.
//
// A walk step needs the node's split word and the row's bin of its feature, a
// random word and a random byte each; from global memory every lane's pair is
// its own sector, and a warp waits for an L2 or DRAM round trip a step.  Here a
// block copies the first split nodes of one tree, in level order (6 bytes each:
// split word with two flags, number of the first child that splits), and each
// warp the records of the rows it works on, read in order; only the deepest
// levels of the largest trees are still read from L2.
//
//   k_walk_trees  a block per tree: numbers its split nodes in level order and
//                 writes them packed; for classes (FP32 terms) also each
//                 leaf's probabilities, divided once per leaf.
//   k_walks       blocks take 2048 rows of a tree at a time, a warp 3 rows: a
//                 lane per row walks the path; then a lane per path node finds
//                 the re-walks (ballots and matches over the path's features);
//                 the 3 rows' re-walks, about 12 each, are dealt to the lanes.
//                 Segment by segment through all trees: blocks work on
//                 different trees, and L2 holds the segment's records.
//
// Measured: N = 1e6, p = 500, 300 trees, depth 20 (213,000 nodes a tree): 963 ->
// 889 ms an iteration; N = 1e5, p = 1000, 500 trees, depth 16: 86.4 -> 80.0.
// Bound by issue (about 750 warp instructions a row and tree, a third of them
// the losses) and by the latency of a step.  Which forests it takes: routes.h.
#include <algorithm>
#include <cstdint>

#include "loss.cuh"

namespace bgb {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
// Warps of a block x rows a warp: more warps hide the latency of a step, more
// rows fill a warp's lanes, both take shared memory from the tree.  N = 1e6,
// 300 trees / N = 1e5, 500 trees, ms an iteration: 16 x 4 957 / 84.3, 24 x 2
// 975 / 86.8, 24 x 4 902 / 80.7, 32 x 2 909 / 83.4, 32 x 3 889 / 79.9.
constexpr int kWarps = 32;
constexpr int kRows = 3;
constexpr uint32_t kSegment = 2048; // rows of a work item
constexpr uint32_t kSmem = 227 * 1024;
constexpr int kRecordBytes = 2048;  // longest record that is staged
constexpr uint32_t kEnd = 0x80000000u;  // a walk that reached the leaf 2 * (split node) + side

__host__ __device__ inline uint32_t warp_bytes(int D, int ldP) {
  // records; path: split words, node numbers, swapped starts and features (4
  // bytes each), the rows' bins (1); base leaves
  return (static_cast<uint32_t>(kRows * (ldP + D * 17 + 4)) + 15u) & ~15u;
}

__device__ __forceinline__ uint32_t excl_scan(uint32_t v, uint32_t* total, uint32_t* part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t x = warp_excl_scan_u32(v, lane);
  if (lane == 31) part[warp] = x + v;
  __syncthreads();
  uint32_t before = 0u, all = 0u;
  for (int w = 0; w < nw; ++w) {
    all += part[w];
    before += w < warp ? part[w] : 0u;
  }
  __syncthreads();
  *total = all;
  return before + x;
}

__global__ void __launch_bounds__(1024) k_walk_trees(Dev d) {
  __shared__ uint32_t part[32], next, from, level_lo[kMaxDepth + 2], level_n[kMaxDepth + 2];
  const int tau = blockIdx.x;
  uint32_t* number = d.nd_lrows;  // split nodes of the tree before the node (the rows were for the fit)
  uint32_t* child = d.nd_ln;
  const bool probs = d.kind == 0 && d.precision != 0;
  const float eps = static_cast<float>(d.kl_eps);
  const float norm = 1.0f + static_cast<float>(d.C) * eps;
  uint32_t lo = static_cast<uint32_t>(tau), n = 1u, done = 0u;
  int levels = 0;
  while (n > 0u && levels <= d.D) {
    if (threadIdx.x == 0) {
      level_lo[levels] = lo;
      level_n[levels] = n;
    }
    uint32_t splits = 0u;
    for (uint32_t i0 = 0u; i0 < n; i0 += blockDim.x) {
      const uint32_t k = lo + i0 + threadIdx.x;
      const bool in = i0 + threadIdx.x < n;
      const uint32_t s = in ? d.nd_split[k] : kLeaf;
      uint32_t tot;
      const uint32_t j = done + splits + excl_scan(s != kLeaf ? 1u : 0u, &tot, part);
      if (in) number[k] = j;
      if (s != kLeaf) {
        if (j == done) next = d.nd_child[k];
      } else if (in && probs) {
        const float nf = static_cast<float>(d.nd_n[k]);
        for (int q = 0; q < d.C; ++q) {
          const int64_t at = static_cast<int64_t>(k) * d.C + q;
          d.nd_lcnt[at] = __float_as_uint(__fdiv_rn(__fdiv_rn(static_cast<float>(d.nd_cnt[at]), nf) + eps, norm));
        }
      }
      splits += tot;
    }
    __syncthreads();
    lo = next;
    done += splits;
    n = 2u * splits;
    ++levels;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    from = atomicAdd(&d.wt_tree[d.M].x, done);  // at most half of the nodes split
    d.wt_tree[tau] = make_uint2(from, done);
  }
  __syncthreads();
  const uint32_t off = from;
  for (int l = 0; l < levels; ++l)
    for (uint32_t i = threadIdx.x; i < level_n[l]; i += blockDim.x) {
      const uint32_t k = level_lo[l] + i, s = d.nd_split[k];
      if (s == kLeaf) continue;
      const uint32_t c = d.nd_child[k], at = off + number[k];
      child[at] = c;
      d.nd_sc[at] = make_uint2(s | (d.nd_split[c] != kLeaf ? 0x80000000u : 0u) |
                                   (d.nd_split[c + 1u] != kLeaf ? 0x40000000u : 0u),
                               number[c]);
    }
}

__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}

// child of split node j (word w) on a side: its number, or kEnd | its leaf
__device__ __forceinline__ uint32_t step(uint32_t j, uint32_t w, uint32_t first, bool right) {
  const uint32_t left_splits = w >> 31;
  const uint32_t splits = right ? (w >> 30) & 1u : left_splits;
  return splits ? first + (right ? left_splits : 0u) : kEnd | (2u * j + (right ? 1u : 0u));
}

__device__ __forceinline__ uint32_t feature(uint32_t w) { return (w & 0x3FFFFFFFu) >> 8; }

// loss32 of a classification from the leaves' probabilities (k_walk_trees)
__device__ __forceinline__ float loss_probs(const Dev& d, uint32_t q, uint32_t q2) {
  const uint32_t* pa = d.nd_lcnt + static_cast<int64_t>(q) * d.C;
  const uint32_t* pb = d.nd_lcnt + static_cast<int64_t>(q2) * d.C;
  float kl = 0.0f;
  for (int c = 0; c < d.C; ++c) {
    const float b = __uint_as_float(pb[c]);
    kl += b * kl_phi(__fdiv_rn(__uint_as_float(pa[c]), b));
  }
  return kl;
}

// PREC: the terms' precision (0, FP64: regression only; walks_pay in routes.h)
template <int PREC>
__global__ void __launch_bounds__(kWarps * 32, 1) k_walks(Dev d, uint32_t nodes) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int D = d.D, ldP = d.ldP;
  uint32_t* tw = reinterpret_cast<uint32_t*>(smem);
  uint16_t* tb = reinterpret_cast<uint16_t*>(smem + 4u * nodes);
  unsigned char* mine = smem + 6u * nodes + warp * warp_bytes(D, ldP);
  uint8_t* rec = mine;
  uint32_t* pw = reinterpret_cast<uint32_t*>(mine + kRows * ldP);
  uint32_t* q_at = pw + kRows * D;
  uint32_t* q_fx = q_at + kRows * D;
  uint32_t* o_leaf = q_fx + kRows * D;
  uint32_t* pj = o_leaf + kRows;
  uint8_t* px = reinterpret_cast<uint8_t*>(pj + kRows * D);
  const uint32_t segments = (static_cast<uint32_t>(d.N) + kSegment - 1u) / kSegment;
  const uint64_t items = static_cast<uint64_t>(d.M) * segments;
  unsigned long long visits = 0;
  int held = -1;  // the tree in shared memory
  for (uint64_t item = blockIdx.x; item < items; item += gridDim.x) {
    const int tau = static_cast<int>(item % static_cast<uint64_t>(d.M));
    const uint32_t r0 = static_cast<uint32_t>(item / static_cast<uint64_t>(d.M)) * kSegment;
    const uint32_t noob = d.oob_cnt[tau];
    const uint2 tree = d.wt_tree[tau];
    if (r0 >= noob || tree.y == 0u) continue;  // block-uniform
    const uint32_t* child = d.nd_ln + tree.x;
    const uint2* all = d.nd_sc + tree.x;
    const uint32_t top = min(tree.y, nodes);  // in shared memory
    if (tau != held) {
      held = tau;
      __syncthreads();  // the last tree's walks are over
#pragma unroll 8
      for (uint32_t j = threadIdx.x; j < top; j += blockDim.x) {
        const uint2 v = all[j];
        tw[j] = v.x;
        tb[j] = static_cast<uint16_t>(v.y);
      }
      __syncthreads();
    }
    const uint32_t* oob = d.oob + static_cast<int64_t>(tau) * d.N;
    const uint32_t end = min(noob, r0 + kSegment);
    for (uint32_t g0 = r0 + warp * kRows; g0 < end; g0 += kWarps * kRows) {
      const int rows = static_cast<int>(min(static_cast<uint32_t>(kRows), end - g0));
      const uint32_t i = lane < rows ? oob[g0 + lane] : 0u;
      const uint32_t pi = lane < rows ? d.piv[i] : 0u;
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        const uint8_t* src = d.Xrow + static_cast<int64_t>(__shfl_sync(kFull, i, r)) * ldP;
        if (r < rows)
          for (int o = 16 * lane; o < ldP; o += 512) copy16(rec + r * ldP + o, src + o);
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncwarp();
      // the rows' paths
      int depth = 0;
      if (lane < rows) {
        const uint8_t* x = rec + lane * ldP;
        uint32_t j = 0u;
        while (depth < D && !(j & kEnd)) {
          const uint2 v = j < top ? make_uint2(tw[j], tb[j]) : all[j];
          const uint8_t b = x[feature(v.x)];
          pw[lane * D + depth] = v.x;
          pj[lane * D + depth] = j;
          px[lane * D + depth] = b;
          ++depth;
          j = step(j, v.x, v.y, b > (v.x & 255u));
        }
        visits += static_cast<unsigned long long>(depth);
        const uint32_t leaf = j & ~kEnd;
        o_leaf[lane] = child[leaf >> 1] + (leaf & 1u);
      }
      __syncwarp();
      // The re-walks, a lane per node of a path: the row with feature f swapped
      // leaves the path at the first node that tests f and sends the swapped
      // bin the other way (if there is none, it reaches the same leaf).
      uint32_t w[kRows], xp[kRows];
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        const bool in = lane < __shfl_sync(kFull, depth, r);
        const uint8_t* x = d.Xrow + static_cast<int64_t>(__shfl_sync(kFull, pi, r)) * ldP;
        w[r] = in ? pw[r * D + lane] : 0xFFFFFFFFu;
        xp[r] = in ? x[feature(w[r])] : 0u;
      }
      uint32_t W = 0u;
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        const bool in = w[r] != 0xFFFFFFFFu;
        const uint32_t f = feature(w[r]);
        const bool right = xp[r] > (w[r] & 255u);
        const bool other = in && right != (px[r * D + min(lane, D - 1)] > (w[r] & 255u));
        const unsigned same = __match_any_sync(kFull, in ? f : kEnd | static_cast<uint32_t>(lane));
        const unsigned others = __ballot_sync(kFull, other);
        const bool leaves = other && (same & others & lt) == 0u;
        const unsigned them = __ballot_sync(kFull, leaves);
        if (leaves) {
          const uint32_t at = W + static_cast<uint32_t>(__popc(them & lt)), j = pj[r * D + lane];
          q_at[at] = step(j, w[r], j < top ? tb[j] : all[j].y, right);
          q_fx[at] = static_cast<uint32_t>(r) << 28 | f << 8 | xp[r];
        }
        W += static_cast<uint32_t>(__popc(them));
      }
      __syncwarp();
      // two re-walks a lane advance together
      for (uint32_t e0 = 0u; e0 < W; e0 += 64u) {
        uint32_t at[2], fx[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const uint32_t e = e0 + 32u * u + lane;
          at[u] = e < W ? q_at[e] : kEnd;
          fx[u] = e < W ? q_fx[e] : 0u;
        }
        for (int guard = 0; guard <= kMaxDepth; ++guard) {  // trees are at most kMaxDepth deep
          if ((at[0] & at[1]) >> 31) break;
          uint2 v[2];
#pragma unroll
          for (int u = 0; u < 2; ++u)
            if (!(at[u] & kEnd)) v[u] = at[u] < top ? make_uint2(tw[at[u]], tb[at[u]]) : all[at[u]];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            if (at[u] & kEnd) continue;
            ++visits;
            const uint32_t f = feature(v[u].x);
            const uint32_t own = rec[(fx[u] >> 28) * ldP + f];
            const uint32_t b = f == ((fx[u] >> 8) & 0xFFFFFu) ? fx[u] & 255u : own;
            at[u] = step(at[u], v[u].x, v[u].y, b > (v[u].x & 255u));
          }
        }
        uint32_t q2[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const uint32_t leaf = at[u] & ~kEnd;
          q2[u] = e0 + 32u * u + lane < W ? child[leaf >> 1] + (leaf & 1u) : 0u;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          if (e0 + 32u * u + lane >= W) continue;
          const uint32_t qo = o_leaf[fx[u] >> 28];
          double L;
          if constexpr (PREC == 0)
            L = loss64(d, qo, q2[u]);
          else
            L = static_cast<double>(d.kind == 0 ? loss_probs(d, qo, q2[u]) : loss32(d, qo, q2[u]));
          if (!csa_add(d.acc + (static_cast<int64_t>(tau) * d.p_aug + ((fx[u] >> 8) & 0xFFFFFu)) * kCsaLimbs, L))
            atomicOr(&d.status[0], kErrAcc);
        }
      }
      __syncwarp();  // the records and the pool are refilled
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) visits += __shfl_xor_sync(kFull, visits, off);
  if (lane == 0 && visits) atomicAdd(&d.counters[3], visits);
}

}  // namespace

// split nodes that fit beside the records (the first children of so many are
// numbered below 2^16)
uint32_t walk_nodes(int D, int ldP) {
  if (ldP > kRecordBytes) return 0u;
  const uint32_t rows = kWarps * warp_bytes(D, ldP);
  return rows < kSmem ? std::min((kSmem - rows) / 6u, 32760u) & ~7u : 0u;
}

int setup_walks() {
  cudaError_t e = cudaFuncSetAttribute(k_walks<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_walks<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  return static_cast<int>(e);
}

int launch_walks(const Dev& d, int sms, cudaStream_t st) {
  cudaMemsetAsync(d.wt_tree + d.M, 0, sizeof(uint2), st);
  k_walk_trees<<<d.M, 1024, 0, st>>>(d);
  uint32_t nodes = walk_nodes(d.D, d.ldP);
  if (d.D < 15) nodes = std::min(nodes, 1u << d.D);
  nodes = (nodes + 7u) & ~7u;
  const size_t bytes = 6u * nodes + kWarps * warp_bytes(d.D, d.ldP);
  if (d.precision == 0)
    k_walks<0><<<sms, kWarps * 32, bytes, st>>>(d, nodes);
  else
    k_walks<1><<<sms, kWarps * 32, bytes, st>>>(d, nodes);
  return 2;
}

}  // namespace bgb
