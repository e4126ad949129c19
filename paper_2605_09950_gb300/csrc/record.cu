// Split search of a level's larger classification nodes whose rows are a
// sparse subset of the matrix: one block per node, rows read by record.
//
// Gathering a column at a node's rows moves a 32-byte sector per bin once the
// node holds fewer than one row in 32.  The row-major copy holds a row's bins
// together, and a node samples the same columns for all its rows, so reading
// records moves fewer sectors (about 20 for 31 of 1000 columns), 4 times fewer
// lines per load instruction, and needs no grouping of (node, feature) items
// by column band.  The block loads 32 features of all the node's rows into a
// byte tile in shared memory (lanes over features, 16 rows in flight a warp),
// then each warp takes features of the tile: a warp-private histogram, its
// prefix sums and the best float score.  The features inside the window of the
// node's best score (usually one) are then counted again and compared exactly;
// the block commits the best split and partitions the rows, so a node is read
// and finished by one launch.
//
// Histograms: class weights are packed into 32-bit words (native shared-memory
// atomics), 3 classes of 10 bits in the smallest tile (nodes of weight below
// 1024) and 2 of 16 bits in the others, one plane of 256 words per word.  Scores are s / (n_L n_R) with
// s = sum_k q_k^2, q_k = l_k n - c_k n_L (see small.cu): exact products in f32
// while n < 4096, in 32-bit integers above.
//
// Measured (one iteration; before: the column gathers of split.cu for all
// nodes above 64 rows): N = 1e6, p = 500, 5 classes, 300 trees: 1148 -> 955 ms;
// N = 30011, 8 classes: 10.2 -> 8.1 ms.  At 257 rows and more the record reads
// bind (4.6 TB/s of DRAM in the 1024-row tile: 64-byte granules make 880 of a
// record's 1000 bytes move), below it the work per (node, feature), about 400
// warp instructions.
//
// Sizes: tiles of 256, 1024 and 4096 rows (4, 8 and 16 warps a block), so that
// a block's shared memory and threads follow its node.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "planes.cuh"

namespace bgb {

namespace {

template <int CM, int ROWS, int WARPS>
struct RecordSmem {
  using P = Pack<CM, ROWS>;
  uint32_t rw[ROWS];                          // per row: P::row of its entry
  uint32_t hist[WARPS][P::W * 256];
  uint32_t tile[32 * (ROWS / 4 + 1)];         // [feature][row] bins; odd word pitch
  unsigned long long bs[WARPS];
  uint32_t bden[WARPS], bkey[WARPS], bslot[WARPS], bcum[WARPS][P::W];
  uint32_t feat[32], fmax[32];
  uint32_t left[ROWS / 32];
  uint32_t cp[CM];
  uint32_t split, slot;
};

// A feature's histogram by one warp (zero on entry).
template <int CM, int ROWS>
__device__ __forceinline__ void record_count(const uint32_t* tile, const uint32_t* rw, uint32_t* hw, uint32_t len) {
  using P = Pack<CM, ROWS>;
  const uint32_t lane = threadIdx.x & 31;
  for (uint32_t wi = lane; wi * 4u < len; wi += 32u) {
    const uint32_t tw = tile[wi];
    const uint4 r4 = reinterpret_cast<const uint4*>(rw)[wi];
    const uint32_t r[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t b = (tw >> (8 * u)) & 255u;
      if (P::W == 1)
        atomicAdd(hw + b, r[u]);
      else
        atomicAdd(hw + b + ((r[u] >> 30) << 8), r[u] & 0x3FFFFFFFu);
    }
  }
  __syncwarp();
}

// The exact best of a feature into the lanes' bests (the one or two features
// of a node whose float best lies inside the window).
template <int CM, int ROWS>
__device__ __noinline__ void record_exact(const uint32_t* tile, const uint32_t* rw, uint32_t* hw, uint32_t len, int B,
                                          uint32_t n, const uint32_t* cp, uint32_t key, uint32_t slot,
                                          RecordBest<CM, ROWS>& best) {
  using P = Pack<CM, ROWS>;
  const int bpl = lane_bins(B);
  record_count<CM, ROWS>(tile, rw, hw, len);
  record_best<CM, ROWS>(hw, bpl, n, cp, key, slot, best);
  record_zero<CM, ROWS>(hw, bpl);
}

// Best float score of one feature by one warp, as its bits (0: no decrease).
// The candidates are all bins, each lane its own, from registers (an empty
// bin repeats the partition of the one below, which has the lower key); in
// the smallest tile, where a node has fewer rows than bins, the rows' own
// bins.  The histogram is zero on entry and on return.
template <int CM, int ROWS>
__device__ __forceinline__ uint32_t record_screen(const uint32_t* tile, const uint32_t* rw, uint32_t* hw, uint32_t len,
                                                  int B, const Totals<CM>& T) {
  using P = Pack<CM, ROWS>;
  const uint32_t lane = threadIdx.x & 31;
  const int bpl = lane_bins(B);
  record_count<CM, ROWS>(tile, rw, hw, len);
  uint32_t h[P::W][8], cum[P::W];
  record_prefix<CM, ROWS>(hw, bpl, h);
  float mine = 0.0f;
  if (ROWS <= 256) {
#pragma unroll
    for (int w = 0; w < P::W; ++w) st_bins(hw + 256 * w + lane * bpl, bpl, h[w]);
    __syncwarp();
    const bool by_row = len <= static_cast<uint32_t>(B);
    const uint32_t count = by_row ? len : static_cast<uint32_t>(B);
#pragma unroll 2
    for (uint32_t i = lane; i < count; i += 32u) {
      const uint32_t b = by_row ? reinterpret_cast<const uint8_t*>(tile)[i] : i;
#pragma unroll
      for (int w = 0; w < P::W; ++w) cum[w] = hw[256 * w + b];
      mine = fmaxf(mine, plane_score<CM, ROWS>(cum, T));
    }
    __syncwarp();  // other lanes may still read this lane's prefix sums
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (q < bpl) {
#pragma unroll
        for (int w = 0; w < P::W; ++w) cum[w] = h[w][q];
        mine = fmaxf(mine, plane_score<CM, ROWS>(cum, T));
      }
  }
  record_zero<CM, ROWS>(hw, bpl);
  return __reduce_max_sync(kFull, __float_as_uint(mine));  // non-negative floats order as their bits
}

template <int CM, int ROWS, int WARPS>
__device__ __forceinline__ void record_node(const Dev& d, int level, uint32_t k, RecordSmem<CM, ROWS, WARPS>& sm) {
  using Pk = Pack<CM, ROWS>;
  constexpr int NW = Pk::W, CH = ROWS / (32 * WARPS), PITCH = ROWS / 4 + 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t* rows_in = d.rows[level & 1];
  NodeInfo<CM> nd;
  load_node<0, CM>(d, k, level, nd);
  const uint32_t len = nd.len, chunks = (len + 31u) / 32u;
  uint32_t e[CH];
#pragma unroll
  for (int i = 0; i < CH; ++i) {
    const uint32_t c = warp + WARPS * i, r = c * 32u + lane;
    e[i] = r < len ? rows_in[nd.base + r] : 0u;
    if (c < chunks) sm.rw[r] = Pk::row(e[i]);
  }
  if (threadIdx.x == 0) {
#pragma unroll
    for (int c = 0; c < CM; ++c) sm.cp[c] = nd.cp[c];
  }
  uint32_t seen = 0u;  // best float score of the block so far, as its bits
  Perm P;
  if (warp == 0) node_perm(d, k, P);
  Totals<CM> T;
  T.n = nd.n;
  T.fn = u24_to_float(nd.n);
#pragma unroll
  for (int c = 0; c < CM; ++c) {
    T.cp[c] = nd.cp[c];
    T.fcp[c] = u24_to_float(nd.cp[c]);
  }
  RecordBest<CM, ROWS> best;
#pragma unroll
  for (int w = 0; w < NW; ++w) best.cum[w] = 0u;
  uint32_t* hw = sm.hist[warp];
  for (int r0 = 0; r0 < d.mtry; r0 += 32) {
    const int nf = min(32, d.mtry - r0);
    if (warp == 0) sm.feat[lane] = lane < nf ? perm_apply(P, static_cast<uint32_t>(r0 + lane)) : 0u;
    __syncthreads();
    const uint32_t f = sm.feat[lane];
#pragma unroll
    for (int i = 0; i < CH; ++i) {
      const uint32_t c = warp + WARPS * i;
      if (c >= chunks) break;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t b[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          const uint32_t r = __shfl_sync(kFull, e[i], 16 * h + q) >> 8;
          b[q] = 0u;
          if (lane < nf && c * 32u + 16u * h + q < len) b[q] = row_bin(d, r, f);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
          sm.tile[lane * PITCH + c * 8u + 4 * h + q] =
              b[4 * q] | (b[4 * q + 1] << 8) | (b[4 * q + 2] << 16) | (b[4 * q + 3] << 24);
      }
    }
    __syncthreads();
    for (int j = warp; j < nf; j += WARPS) {
      const uint32_t mx = record_screen<CM, ROWS>(sm.tile + j * PITCH, sm.rw, hw, len, d.B, T);
      if (lane == 0) sm.fmax[j] = mx;
    }
    __syncthreads();
    // every candidate whose exact score is the best has a float score inside
    // the window of the best one: usually one feature's
    const uint32_t mine = lane < nf ? sm.fmax[lane] : 0u;
    seen = max(seen, __reduce_max_sync(kFull, mine));
    unsigned in = __ballot_sync(kFull, mine != 0u && __uint_as_float(mine) >= screen(__uint_as_float(seen)));
    for (int i = 0; in; ++i) {
      const int j = __ffs(in) - 1;
      in &= in - 1;
      if (i % WARPS != warp) continue;
      record_exact<CM, ROWS>(sm.tile + j * PITCH, sm.rw, hw, len, d.B, nd.n, sm.cp,
                             (d.tie_break == 1 ? static_cast<uint32_t>(r0 + j) : sm.feat[j]) << 8, r0 + j, best);
    }
    if (r0 + 32 < d.mtry) __syncthreads();  // the tile is refilled
  }
  // the block's best
  record_reduce<CM, ROWS>(best);
  if (lane == 0) {
    sm.bs[warp] = best.s;
    sm.bden[warp] = best.den;
    sm.bkey[warp] = best.key;
    sm.bslot[warp] = best.slot;
#pragma unroll
    for (int w = 0; w < NW; ++w) sm.bcum[warp][w] = best.cum[w];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int b = 0;
    for (int w = 1; w < WARPS; ++w) {
      const int c = frac64_cmp(sm.bs[w], sm.bden[w], sm.bs[b], sm.bden[b]);
      if (c > 0 || (c == 0 && sm.bkey[w] < sm.bkey[b])) b = w;
    }
    uint32_t cum[NW], cL[CM], nL = 0u;
#pragma unroll
    for (int w = 0; w < NW; ++w) cum[w] = sm.bcum[b][w];
#pragma unroll
    for (int c = 0; c < CM; ++c) nL += cL[c] = Pk::field(cum, c);
    const uint32_t slot = sm.bslot[b], key = sm.bkey[b];
    const bool ok = sm.bs[b] > 0ull;
    uint32_t feat = key >> 8;
    if (ok && d.tie_break == 1) feat = perm_apply(P, slot);
    sm.split = commit_counts<CM>(d, k, ok, feat, key & 255u, nL, cL, sm.bs[b], nd.n);
    sm.slot = slot;
    const uint32_t rd = static_cast<uint32_t>(d.mtry) + 4u + (ok ? 5u : 0u);
    atomicAdd(&d.counters[0], static_cast<unsigned long long>(len) * rd);
    atomicAdd(&d.counters[2], static_cast<unsigned long long>(len) * (d.mtry + kRowStateClass));
  }
  __syncthreads();
  const uint32_t sp = sm.split;
  if (sp != kLeaf) {
    const bool in_tile = d.mtry <= 32;
    const uint8_t* tb = reinterpret_cast<const uint8_t*>(sm.tile + sm.slot * PITCH);
    const uint32_t total = block_partition<CH, WARPS>(
        e, len, nd.base, d.rows[(level & 1) ^ 1], sm.left,
        [&](int i, uint32_t r) {
          return (in_tile ? static_cast<uint32_t>(tb[r]) : row_bin(d, e[i] >> 8, sp >> 8)) <= (sp & 255u);
        });
    if (threadIdx.x == 0) d.nd_lrows[k] = total;
  }
  __syncthreads();  // the next node refills the block's shared memory
}

// which: 0 = nodes of at most 256 rows (`rec`), 1 = at most 1024 (the start of
// `rec2`), 2 = at most 4096 (the end of `rec2`)
template <int CM, int ROWS, int WARPS, int MINB>
__global__ void __launch_bounds__(WARPS * 32, MINB) k_record(Dev d, int level) {
  extern __shared__ __align__(16) unsigned char raw[];
  auto& sm = *reinterpret_cast<RecordSmem<CM, ROWS, WARPS>*>(raw);
  const uint32_t nn = d.nrec[3 * level + (ROWS == 256 ? 0 : (ROWS == 1024 ? 1 : 2))];
  if (blockIdx.x >= nn) return;
  for (uint32_t i = threadIdx.x; i < WARPS * Pack<CM, ROWS>::W * 256; i += WARPS * 32) sm.hist[0][i] = 0u;
  __syncthreads();
  for (uint32_t i = blockIdx.x; i < nn; i += gridDim.x)
    record_node<CM, ROWS, WARPS>(
        d, level, ROWS == 256 ? d.rec[i] : (ROWS == 1024 ? d.rec2[i] : d.rec2[d.rec2_cap - 1u - i]), sm);
}

template <int CM, int ROWS, int WARPS, int MINB>
cudaError_t setup(int sms, int* grid) {
  auto* f = &k_record<CM, ROWS, WARPS, MINB>;
  const int smem = static_cast<int>(sizeof(RecordSmem<CM, ROWS, WARPS>));
  cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  int per_sm = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, WARPS * 32, smem);
  *grid = (per_sm < 1 ? 1 : per_sm) * sms;
  return e;
}

template <int CM>
int launch(const Dev& d, int level, const int* grids, uint64_t nodes, cudaStream_t st) {
  auto grid = [&](int i, uint64_t most) {
    return static_cast<unsigned>(std::max<uint64_t>(1, std::min<uint64_t>(static_cast<uint64_t>(grids[i]), most)));
  };
  const uint64_t M = static_cast<uint64_t>(d.M), N = static_cast<uint64_t>(d.N);
  int n = 0;
  if (d.rec_rows > 1024u) {
    k_record<CM, 4096, 16, 1><<<grid(2, std::min(nodes, M * (N / 1025 + 1))), 512,
                               sizeof(RecordSmem<CM, 4096, 16>), st>>>(d, level);
    ++n;
  }
  if (d.rec_rows > 256u) {
    k_record<CM, 1024, 8, 3><<<grid(1, std::min(nodes, M * (N / 257 + 1))), 256, sizeof(RecordSmem<CM, 1024, 8>),
                               st>>>(d, level);
    ++n;
  }
  k_record<CM, 256, 4, 8><<<grid(0, std::min(nodes, M * (N / 65 + 1))), 128, sizeof(RecordSmem<CM, 256, 4>), st>>>(
      d, level);
  return n + 1;
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

}  // namespace

int setup_record(int variant, int sms, int* grids) {
  return with_classes(variant, [&](auto cm) {
    constexpr int CM = decltype(cm)::value;
    cudaError_t e = setup<CM, 256, 4, 8>(sms, grids);
    if (e == cudaSuccess) e = setup<CM, 1024, 8, 3>(sms, grids + 1);
    if (e == cudaSuccess) e = setup<CM, 4096, 16, 1>(sms, grids + 2);
    return static_cast<int>(e);
  });
}

int launch_record(const Dev& d, int level, const int* grids, uint64_t nodes, cudaStream_t st) {
  return with_classes(split_variant(d.kind, d.C),
                      [&](auto cm) { return launch<decltype(cm)::value>(d, level, grids, nodes, st); });
}

}  // namespace bgb
