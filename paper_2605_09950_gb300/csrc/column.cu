// Split search of a level's larger classification nodes where a whole column
// fits in shared memory: one block per column, which it loads once for all the
// nodes that sample it.
//
// A random byte from shared memory costs a bank cycle instead of a 32-byte
// sector, so the gathers of a level (rows x sampled columns) run at the rate
// of the row lists, which are read in order.  Per level:
//   k_col_count / k_col_scan / k_col_fill  the (node, draw slot) items sorted
//                  by column;
//   k_column       a block per column: warps take its items as they come free,
//                  count the node's rows in a warp-private packed histogram
//                  (planes.cuh) and keep the best float score of the item;
//   k_col_finish   a block per node: the items inside the window of the node's
//                  best score (usually one) are counted again and compared
//                  exactly; split record and partition.
// Nodes of at most 256 rows stay with record.cu: an item's fixed work (its
// record, the scan of 256 bins) would be most of it.
//
// Measured: N = 1e5, p = 1000, 2 classes, 500 trees, depth 16: 141 -> 93 ms
// an iteration; 1.2 to 2.2 ms a level here (6 to 9 by column gathers from L2).
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "planes.cuh"

namespace bgb {

namespace {

constexpr int kColWarps = 32;
constexpr int kColPack = 1024;  // Pack<CM, kColPack>: two classes a word
constexpr int kFinishThreads = 256;

template <int CM>
using ColPack = Pack<CM, kColPack>;

// totals of the column list's nodes, and the number of items per column
template <int CM>
__global__ void __launch_bounds__(256) k_col_count(Dev d, int level) {
  const int lane = threadIdx.x & 31;
  const uint32_t nn = d.nrec[3 * level + 1];
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t rank = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; rank < nn; rank += nwarps) {
    const uint32_t k = d.rec2[rank];
    if (lane == 0) {
      NodeInfo<CM> nd;
      load_node<0, CM>(d, k, level, nd);
      reinterpret_cast<NodeInfo<CM>*>(d.ninfo)[rank] = nd;
    }
    Perm P;
    node_perm(d, k, P);
    for (int s = lane; s < d.mtry; s += 32) atomicAdd(&d.col_cnt[perm_apply(P, static_cast<uint32_t>(s))], 1u);
  }
}

// exclusive scan of the counts in place (one block)
__global__ void __launch_bounds__(1024) k_col_scan(Dev d, int level) {
  __shared__ uint32_t warps[32];
  if (d.nrec[3 * level + 1] == 0u) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t carry = 0u;
  for (int f0 = 0; f0 < d.p_aug; f0 += 1024) {
    const int f = f0 + threadIdx.x;
    const uint32_t v = f < d.p_aug ? d.col_cnt[f] : 0u;
    const uint32_t x = warp_excl_scan_u32(v, lane);
    if (lane == 31) warps[warp] = x + v;
    __syncthreads();
    const uint32_t t = warp_excl_scan_u32(warps[lane], lane);
    const uint32_t before = __shfl_sync(kFull, t, warp), all = __shfl_sync(kFull, t + warps[lane], 31);
    if (f < d.p_aug) d.col_cnt[f] = carry + before + x;
    carry += all;
    __syncthreads();
  }
}

// the items, each in its column's range; the starts become the ends
__global__ void __launch_bounds__(256) k_col_fill(Dev d, int level) {
  const int lane = threadIdx.x & 31;
  const uint32_t nn = d.nrec[3 * level + 1];
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t rank = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; rank < nn; rank += nwarps) {
    Perm P;
    node_perm(d, d.rec2[rank], P);
    for (int s = lane; s < d.mtry; s += 32)
      d.items_u[atomicAdd(&d.col_cnt[perm_apply(P, static_cast<uint32_t>(s))], 1u)] =
          (static_cast<uint64_t>(rank) << 32) | static_cast<uint32_t>(s);
  }
}

template <int CM>
__global__ void __launch_bounds__(kColWarps * 32, 1) k_column(Dev d, int level) {
  using P = ColPack<CM>;
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ uint32_t next;
  if (d.nrec[3 * level + 1] == 0u) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int f = blockIdx.x;
  const uint32_t start = f ? d.col_cnt[f - 1] : 0u, count = d.col_cnt[f] - start;
  if (blockIdx.y >= count) return;  // block-uniform
  uint8_t* col = raw;
  uint32_t* hw = reinterpret_cast<uint32_t*>(raw + d.ldN) + warp * (P::W * 256);
  const uint4* src = reinterpret_cast<const uint4*>(column(d, static_cast<uint32_t>(f)));
  for (int i = threadIdx.x; i < d.ldN / 16; i += kColWarps * 32) reinterpret_cast<uint4*>(col)[i] = src[i];
  for (int i = lane; i < P::W * 256; i += 32) hw[i] = 0u;
  if (threadIdx.x == 0) next = blockIdx.y;
  __syncthreads();
  const uint32_t* rows_in = d.rows[level & 1];
  const int bpl = lane_bins(d.B);
  float* fmax = reinterpret_cast<float*>(d.fbest);
  for (;;) {
    uint32_t at = 0u;
    if (lane == 0) at = atomicAdd(&next, gridDim.y);
    at = __shfl_sync(kFull, at, 0);
    if (at >= count) break;
    const uint64_t item = d.items_u[start + at];
    const uint32_t rank = static_cast<uint32_t>(item >> 32);
    const NodeInfo<CM> nd = reinterpret_cast<const NodeInfo<CM>*>(d.ninfo)[rank];
    const uint32_t* rows = rows_in + nd.base;
    const uint32_t len = nd.len;
    uint32_t e[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) e[q] = q * 32u + lane < len ? ld_stream(rows + q * 32 + lane) : 0u;
    for (uint32_t r0 = 0; r0 < len; r0 += 256u) {
      uint32_t n[8];  // the next rows, in flight
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const uint32_t r = r0 + 256u + q * 32u + lane;
        n[q] = r < len ? ld_stream(rows + r) : 0u;
      }
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (r0 + q * 32u + lane < len)
          atomicAdd(hw + col[e[q] >> 8] + (P::W > 1 ? ((e[q] >> 6) & 3u) << 8 : 0u),
                    ent_w<0>(e[q]) << ((e[q] >> 1) & 16u));  // class y: half y & 1 of word y >> 1
#pragma unroll
      for (int q = 0; q < 8; ++q) e[q] = n[q];
    }
    __syncwarp();
    Totals<CM> T;
    T.n = nd.n;
    T.fn = u24_to_float(nd.n);
#pragma unroll
    for (int c = 0; c < CM; ++c) {
      T.cp[c] = nd.cp[c];
      T.fcp[c] = u24_to_float(nd.cp[c]);
    }
    uint32_t h[P::W][8], cum[P::W];
    record_prefix<CM, kColPack>(hw, bpl, h);
    float mine = 0.0f;
    const bool narrow = nd.n < 4096u;
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (q < bpl) {
#pragma unroll
        for (int w = 0; w < P::W; ++w) cum[w] = h[w][q];
        mine = fmaxf(mine, narrow ? plane_score<CM, 1024>(cum, T) : plane_score<CM, 4096>(cum, T));
      }
    record_zero<CM, kColPack>(hw, bpl);
    const uint32_t mx = __reduce_max_sync(kFull, __float_as_uint(mine));
    if (lane == 0)
      fmax[static_cast<uint64_t>(rank) * d.mtry + static_cast<uint32_t>(item)] = __uint_as_float(mx);
  }
}

template <int CM>
__global__ void __launch_bounds__(kFinishThreads) k_col_finish(Dev d, int level) {
  using P = ColPack<CM>;
  constexpr int kWarps = kFinishThreads / 32;
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ __align__(16) uint32_t hist[P::W * 256];  // read and cleared 16 bytes at a time
  __shared__ uint32_t red[kWarps], cps[CM], s_sp, s_total;
  uint32_t* bits = reinterpret_cast<uint32_t*>(raw);  // per 32 rows: which go left
  uint32_t* before = bits + (d.N + 31) / 32;          // and how many before them
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t nn = d.nrec[3 * level + 1];
  const uint32_t* rows_in = d.rows[level & 1];
  uint32_t* rows_out = d.rows[(level & 1) ^ 1];
  const int bpl = lane_bins(d.B);
  for (uint32_t i = threadIdx.x; i < P::W * 256; i += kFinishThreads) hist[i] = 0u;
  for (uint32_t rank = blockIdx.x; rank < nn; rank += gridDim.x) {
    const uint32_t k = d.rec2[rank];
    const NodeInfo<CM> nd = reinterpret_cast<const NodeInfo<CM>*>(d.ninfo)[rank];
    const float* fmax = reinterpret_cast<const float*>(d.fbest) + static_cast<uint64_t>(rank) * d.mtry;
    const uint32_t* rows = rows_in + nd.base;
    uint32_t mx = 0u;
    for (int s = threadIdx.x; s < d.mtry; s += kFinishThreads) mx = max(mx, __float_as_uint(fmax[s]));
    mx = __reduce_max_sync(kFull, mx);
    if (lane == 0) red[warp] = mx;
    if (threadIdx.x == 0) {
#pragma unroll
      for (int c = 0; c < CM; ++c) cps[c] = nd.cp[c];
    }
    Perm Q;
    node_perm(d, k, Q);
    __syncthreads();
    mx = red[0];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) mx = max(mx, red[w]);
    const float thr = screen(__uint_as_float(mx));
    RecordBest<CM, kColPack> best;
#pragma unroll
    for (int w = 0; w < P::W; ++w) best.cum[w] = 0u;
    for (int s = 0; mx != 0u && s < d.mtry; ++s) {
      if (fmax[s] < thr) continue;  // block-uniform
      const uint32_t f = perm_apply(Q, static_cast<uint32_t>(s));
      const uint8_t* col = column(d, f);
      for (uint32_t r = threadIdx.x; r < nd.len; r += kFinishThreads) {
        const uint32_t e = rows[r];
        atomicAdd(hist + col[e >> 8] + (P::W > 1 ? ((e >> 6) & 3u) << 8 : 0u), ent_w<0>(e) << ((e >> 1) & 16u));
      }
      __syncthreads();
      if (warp == 0) {
        record_best<CM, kColPack>(hist, bpl, nd.n, cps, (d.tie_break == 1 ? static_cast<uint32_t>(s) : f) << 8,
                                  static_cast<uint32_t>(s), best);
        record_zero<CM, kColPack>(hist, bpl);
      }
      __syncthreads();
    }
    if (warp == 0) {
      record_reduce<CM, kColPack>(best);
      if (lane == 0) {
        uint32_t cL[CM], nL = 0u;
#pragma unroll
        for (int c = 0; c < CM; ++c) nL += cL[c] = P::field(best.cum, c);
        const bool ok = best.s > 0ull;
        uint32_t feat = best.key >> 8;
        if (ok && d.tie_break == 1) feat = perm_apply(Q, best.slot);
        s_sp = commit_counts<CM>(d, k, ok, feat, best.key & 255u, nL, cL, best.s, nd.n);
        const uint32_t rd = static_cast<uint32_t>(d.mtry) + 4u + (ok ? 5u : 0u);
        atomicAdd(&d.counters[0], static_cast<unsigned long long>(nd.len) * rd);
        atomicAdd(&d.counters[2], static_cast<unsigned long long>(nd.len) * (d.mtry + kRowStateClass));
      }
    }
    __syncthreads();
    const uint32_t sp = s_sp;
    if (sp != kLeaf) {
      // stable partition: left rows in order, then right rows in order
      const uint8_t* col = column(d, sp >> 8);
      const uint32_t chunks = (nd.len + 31u) / 32u;
      for (uint32_t c = warp; c < chunks; c += kWarps) {
        const uint32_t r = c * 32u + lane;
        const unsigned b = __ballot_sync(kFull, r < nd.len && col[rows[r < nd.len ? r : 0u] >> 8] <= (sp & 255u));
        if (lane == 0) bits[c] = b;
      }
      __syncthreads();
      if (warp == 0) {
        uint32_t total = 0u;
        for (uint32_t c0 = 0; c0 < chunks; c0 += 32u) {
          const uint32_t v = c0 + lane < chunks ? __popc(bits[c0 + lane]) : 0u;
          const uint32_t x = total + warp_excl_scan_u32(v, lane);
          if (c0 + lane < chunks) before[c0 + lane] = x;
          total = __shfl_sync(kFull, x + v, 31);
        }
        if (lane == 0) {
          s_total = total;
          d.nd_lrows[k] = total;
        }
      }
      __syncthreads();
      for (uint32_t r = threadIdx.x; r < nd.len; r += kFinishThreads) {
        const uint32_t b = bits[r >> 5], l = before[r >> 5] + __popc(b & lanemask_lt());
        rows_out[nd.base + (((b >> lane) & 1u) ? l : s_total + (r - l))] = rows[r];
      }
    }
    __syncthreads();
  }
}

template <typename F>
auto with_classes(int variant, F&& f) {
  switch (variant) {
    case 0: return f(std::integral_constant<int, 2>{});
    case 1: return f(std::integral_constant<int, 3>{});
    case 2: return f(std::integral_constant<int, 4>{});
    case 3: return f(std::integral_constant<int, 5>{});
    default: return f(std::integral_constant<int, 8>{});
  }
}

template <int CM>
size_t column_smem(const Dev& d) {
  return static_cast<size_t>(d.ldN) + kColWarps * ColPack<CM>::W * 1024;
}

size_t finish_smem(const Dev& d) { return static_cast<size_t>((d.N + 31) / 32) * 8; }

constexpr size_t kColSmemMax = 226 * 1024;

}  // namespace

// Whether the session's columns fit, and the grid of k_col_finish (0: not).
int setup_column(const Dev& d, int sms, int* grid) {
  *grid = 0;
  return with_classes(split_variant(d.kind, d.C), [&](auto cm) {
    constexpr int CM = decltype(cm)::value;
    if (column_smem<CM>(d) > kColSmemMax) return 0;
    // one limit for every session of the process
    cudaError_t e = cudaFuncSetAttribute(k_column<CM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(kColSmemMax));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_col_finish<CM>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
    int per_sm = 0;
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_col_finish<CM>, kFinishThreads, finish_smem(d));
    *grid = per_sm * sms;
    return static_cast<int>(e);
  });
}

// The level's nodes of the column list (rec2, nrec[1]): at most `nodes`.
int launch_column(const Dev& d, int level, int sms, int finish_grid, uint64_t nodes, cudaStream_t st) {
  return with_classes(split_variant(d.kind, d.C), [&](auto cm) {
    constexpr int CM = decltype(cm)::value;
    const unsigned warps8 = static_cast<unsigned>(std::max<uint64_t>(1, std::min<uint64_t>((nodes + 7) / 8, 8ull * sms)));
    const unsigned fin =
        static_cast<unsigned>(std::max<uint64_t>(1, std::min<uint64_t>(nodes, static_cast<uint64_t>(finish_grid))));
    // blocks per column: enough of them for two rounds of the GPU
    const unsigned parts = static_cast<unsigned>(std::max(1, (2 * sms + d.p_aug - 1) / d.p_aug));
    cudaMemsetAsync(d.col_cnt, 0, static_cast<size_t>(d.p_aug) * sizeof(uint32_t), st);
    k_col_count<CM><<<warps8, 256, 0, st>>>(d, level);
    k_col_scan<<<1, 1024, 0, st>>>(d, level);
    k_col_fill<<<warps8, 256, 0, st>>>(d, level);
    k_column<CM><<<dim3(static_cast<unsigned>(d.p_aug), parts), kColWarps * 32, column_smem<CM>(d), st>>>(d, level);
    k_col_finish<CM><<<fin, kFinishThreads, finish_smem(d), st>>>(d, level);
    return 5;
  });
}

}  // namespace bgb
