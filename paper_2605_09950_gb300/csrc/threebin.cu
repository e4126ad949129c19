// Split search of regression nodes over columns of at most three bins
// (genotypes), where a node samples many of them (three_bins_pay in routes.h).
//
// Two thresholds per column, and every threshold's left totals are sums over
// the node's rows: with Le[(f, b)][s] = 1 where bin_s(f) <= b, the sums for all
// columns are the product of Le by the rows' values, a matrix product of
// (2 x columns) x rows x 8.  The values are exact: a row's weighted target
// (|sum| < 2^62) is cut into seven 9-bit limbs, the last one signed, and the
// eighth column is its weight; products of 0/1 by integers below 512 are exact
// in f16, and their f32 sums stay below 2^23 for fewer than 16384 rows.
//
//   k_three_rows    nodes of more than 8 rows, a block each: the rows' records
//                   are read whole (a third of the columns are sampled, so the
//                   16-byte-aligned record is dense), 128 columns a warp;
//                   16 rows x 128 bins go through a tile in shared memory as
//                   half pairs of consecutive rows, from which the 0/1 operand
//                   comes by two comparisons a register; one mma.sync covers
//                   8 columns x 2 thresholds x 16 rows.
//   k_three_few     nodes of at most 8 rows, a warp each: a threshold selects
//                   one of at most 256 subsets of the rows, whose scores are
//                   tabulated once; a column then costs its bits and two
//                   table reads.
// The node's sampled columns are a bit map (its permutation is evaluated by
// lanes that take the next slot as soon as theirs falls inside the domain).
// Every lane keeps its best candidate: by the float score where it is outside
// the window of the exact one's error, exactly (192-bit fractions) inside it,
// so the chosen split is that of an exhaustive exact comparison.
//
// Measured: N = 20000, p = 5003, 100 trees, depth 12, a third of the columns
// sampled: 556 -> 88 ms an iteration (gathers of columns and warp reductions
// before); about 6 ms a level down to depth 7, 13.5 ms at depth 11.  Bound by
// the ALU pipe (62% busy at depth 10): bytes to half pairs, comparisons, scores.
#include <cstdint>

#include "regress.cuh"

namespace bgb {

namespace {

constexpr int kTbWarps = 8;       // warps of a k_three_rows block
constexpr int kTbRows = 512;      // rows staged at a time
constexpr int kTbPitch = 136;     // words per row pair of a warp's tile (128 columns; 8 mod 32)

// Bits of the columns a node samples: slots first, first + step, ... by this
// thread.
__device__ __forceinline__ void mark_columns(const Perm& P, int mtry, uint32_t first, uint32_t step, uint32_t* bits) {
  uint32_t s = first, x = first;
  bool live = s < static_cast<uint32_t>(mtry);
  while (__any_sync(kFull, live)) {
    if (live) {
      if (P.n > 1u) x = feistel8(P, x);
      if (x < P.n) {
        atomicOr(&bits[x >> 5], 1u << (x & 31u));
        s += step;
        x = s;
        live = s < static_cast<uint32_t>(mtry);
      }
    }
  }
}

// ---------------------------------------------------------------- more than 8 rows
struct TbSmem {
  uint32_t tile[kTbWarps][8 * kTbPitch];  // [row pair][column] halves of two rows
  uint32_t val[kTbRows / 2][8];           // [row pair][limb] halves of two rows
  uint32_t row[kTbRows];
  RegCand best[kTbWarps];
  Perm perm;
  uint32_t sp;
};

template <typename T>
__device__ __forceinline__ T quad_own(const T (&p)[4], int t) {
  const bool o = t & 1, h = t & 2;
  const T x = __shfl_xor_sync(kFull, o ? p[0] : p[1], 1), y = __shfl_xor_sync(kFull, o ? p[2] : p[3], 1);
  const T k0 = (o ? p[1] : p[0]) + x, k1 = (o ? p[3] : p[2]) + y;
  return (h ? k1 : k0) + __shfl_xor_sync(kFull, h ? k0 : k1, 2);
}

__device__ void three_rows(const Dev& d, int level, uint32_t k, TbSmem& sm, uint32_t* bits) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  const uint32_t* rows_in = d.rows[level & 1];
  NodeInfo<1> nd;
  load_node<1, 1>(d, k, level, nd);
  const uint32_t len = nd.len, words = (static_cast<uint32_t>(d.p_aug) + 31u) / 32u;
  for (uint32_t i = threadIdx.x; i < words; i += kTbWarps * 32) bits[i] = 0u;
  if (threadIdx.x == 0) node_perm(d, k, sm.perm);
  const bool short_sums = !d.wide_y && len < 4096u;  // five limbs (45 bits and a sign) and 32-bit partial sums
  auto stage = [&](uint32_t r0) {  // rows r0 .. of the node
    const uint32_t nr = min(static_cast<uint32_t>(kTbRows), (len - r0 + 15u) & ~15u);
    for (uint32_t i = threadIdx.x; i < nr; i += kTbWarps * 32) {
      const bool v = r0 + i < len;
      const uint32_t e = rows_in[nd.base + (v ? r0 + i : 0u)];
      const uint32_t w = v ? ent_w<1>(e) : 0u;
      sm.row[i] = e >> 8;
      const long long x = v ? static_cast<long long>(w) * d.yreg[e >> 8] : 0ll;
      uint16_t* h = reinterpret_cast<uint16_t*>(&sm.val[i >> 1][0]) + (i & 1u);
#pragma unroll
      for (int j = 0; j < 6; ++j) {
        const int limb = static_cast<int>((x >> (9 * j)) & 511);
        h[2 * j] = static_cast<uint16_t>(half_bits(short_sums && j >= 4 ? (j == 4 ? static_cast<int>(x >> 36) : 0) : limb));
      }
      h[12] = static_cast<uint16_t>(half_bits(short_sums ? 0 : static_cast<int>(x >> 54)));
      h[14] = static_cast<uint16_t>(half_bits(static_cast<int>(w)));
    }
    return nr;
  };
  uint32_t nr = stage(0u);
  __syncthreads();
  const Perm P = sm.perm;
  mark_columns(P, d.mtry, threadIdx.x, kTbWarps * 32, bits);
  __syncthreads();
  const Perm* order = d.tie_break == 1 ? &sm.perm : nullptr;
  RegCand best;
  uint32_t* tile = sm.tile[warp];
  const uint32_t ldP = static_cast<uint32_t>(d.ldP);
  const float bias = t == 3 ? 12582912.0f : 8388608.0f;  // the last limb is signed
  const int ibias = __float_as_int(bias);
  const uint32_t blocks = (static_cast<uint32_t>(d.p_aug) + 127u) / 128u;
  for (uint32_t fb0 = 0; fb0 < blocks; fb0 += kTbWarps) {
    const uint32_t f0 = (fb0 + warp) * 128u;
    const bool mine = f0 < static_cast<uint32_t>(d.p_aug);
    const bool in = mine && f0 + 4u * lane < ldP;
    const uint8_t* src = d.Xrow + f0 + 4u * lane;
    float acc[16][4];
#pragma unroll
    for (int q = 0; q < 16; ++q)
#pragma unroll
      for (int x = 0; x < 4; ++x) acc[q][x] = 0.0f;
    for (uint32_t r0 = 0; r0 < len; r0 += kTbRows) {
      if (len > kTbRows) {  // (one chunk stays staged)
        __syncthreads();
        nr = stage(r0);
        __syncthreads();
      }
      if (!mine) continue;
      uint32_t w[16];
      auto fetch = [&](uint32_t c0) {
#pragma unroll
        for (int q = 0; q < 16; ++q)
          w[q] = in ? *reinterpret_cast<const uint32_t*>(src + static_cast<uint64_t>(sm.row[c0 + q]) * ldP) : 0u;
      };
      fetch(0u);
      for (uint32_t c0 = 0; c0 < nr; c0 += 16u) {
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 8; ++q) {  // bytes of two rows to half pairs by column
          const uint32_t a = w[2 * q] & 0x00FF00FFu, b = w[2 * q + 1] & 0x00FF00FFu;
          const uint32_t c = (w[2 * q] >> 8) & 0x00FF00FFu, e = (w[2 * q + 1] >> 8) & 0x00FF00FFu;
          *reinterpret_cast<uint4*>(tile + q * kTbPitch + 4 * lane) =
              make_uint4(__byte_perm(a, b, 0x5410), __byte_perm(c, e, 0x5410), __byte_perm(a, b, 0x7632),
                         __byte_perm(c, e, 0x7632));
        }
        __syncwarp();
        if (c0 + 16u < nr) fetch(c0 + 16u);  // the next rows, in flight during the products
        const uint32_t b0 = sm.val[c0 / 2u + t][g], b1 = sm.val[c0 / 2u + t + 4][g];
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          const uint32_t p0 = tile[t * kTbPitch + 8 * q + g], p1 = tile[(t + 4) * kTbPitch + 8 * q + g];
          const uint32_t a0 = le_h2(p0, 0u), a1 = le_h2(p0, 0x00010001u), a2 = le_h2(p1, 0u),
                         a3 = le_h2(p1, 0x00010001u);
          asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
              "{%0,%1,%2,%3};"
              : "+f"(acc[q][0]), "+f"(acc[q][1]), "+f"(acc[q][2]), "+f"(acc[q][3])
              : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
        }
      }
    }
    if (!mine) continue;
    if (short_sums) {
      // Limbs 0..4 (the last one signed; its lane's other column is 0) and the
      // weight: a lane's two columns in 32 bits (rows < 4096).  The quads' parts
      // go through the tile, so that the lanes then score the sampled columns
      // only, one after another.
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 16; ++q)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          const int m0 = __float_as_int(acc[q][2 * b] + 12582912.0f) - 0x4B400000;
          const int m1 = __float_as_int(acc[q][2 * b + 1] + 12582912.0f) - 0x4B400000;
          tile[((8 * q + g) * 2 + b) * 4 + t] = static_cast<uint32_t>(t == 3 ? m1 : m0 + (m1 << 9));
        }
      uint8_t* list = reinterpret_cast<uint8_t*>(tile + 1024);  // the block's sampled columns
      uint32_t count = 0u;
#pragma unroll
      for (uint32_t w = 0; w < 4; ++w) {
        const uint32_t bw = (f0 >> 5) + w < words ? bits[(f0 >> 5) + w] : 0u;
        if ((bw >> lane) & 1u) list[count + __popc(bw & lanemask_lt())] = static_cast<uint8_t>(32u * w + lane);
        count += __popc(bw);
      }
      __syncwarp();
      for (uint32_t i = lane; i < 2u * count; i += 32u) {
        const uint32_t c = list[i >> 1], b = i & 1u;
        const int4 m = reinterpret_cast<const int4*>(tile)[2u * c + b];
        const long long S = static_cast<long long>(m.x) + (static_cast<long long>(m.y) << 18) +
                            static_cast<long long>(m.z) * (1ll << 36);
        const uint32_t nL = static_cast<uint32_t>(m.w);
        if (nL > 0u && nL < nd.n)
          reg_offer(best, score_reg_narrow(S, nd.SP, nL, nd.n), S, nL, ((f0 + c) << 8) | b, nd.SP, nd.n, order);
      }
      continue;
    }
    // two column groups at a time: lane t of a quad takes group t / 2, threshold t % 2
#pragma unroll
    for (int q = 0; q < 16; q += 2) {
      long long part[4];
      uint32_t cnt[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int m0 = __float_as_int(acc[q + (i >> 1)][2 * (i & 1)] + bias) - ibias;
        const int m1 = __float_as_int(acc[q + (i >> 1)][2 * (i & 1) + 1] + bias) - ibias;
        // (modulo 2^64: the total fits)
        part[i] = static_cast<long long>(
            static_cast<unsigned long long>(static_cast<long long>(m0) + (t == 3 ? 0ll : 512ll * m1)) << (18 * t));
        cnt[i] = t == 3 ? static_cast<uint32_t>(m1) : 0u;
      }
      const long long S = quad_own(part, t);
      const uint32_t nL = quad_own(cnt, t);
      const uint32_t f = f0 + 8u * (q + (t >> 1)) + g;
      const bool drawn = f < static_cast<uint32_t>(d.p_aug) && ((bits[f >> 5] >> (f & 31u)) & 1u);
      if (drawn && nL > 0u && nL < nd.n)
        reg_offer(best, score_reg_any(d.wide_y, S, nd.SP, nL, nd.n), S, nL, (f << 8) | static_cast<uint32_t>(t & 1),
                  nd.SP, nd.n, order);
    }
  }
  reg_warp_best(best, nd.SP, nd.n, order);
  if (lane == 0) sm.best[warp] = best;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kTbWarps; ++w)
      reg_offer(best, sm.best[w].sf, sm.best[w].S, sm.best[w].nL, sm.best[w].fb, nd.SP, nd.n, order);
    sm.sp = commit_reg(d, k, best, nd);
    const unsigned long long rd = static_cast<unsigned long long>(d.mtry) + 12u + (sm.sp != kLeaf ? 5u : 0u);
    atomicAdd(&d.counters[0], len * rd);
    atomicAdd(&d.counters[2], static_cast<unsigned long long>(len) * (d.mtry + kRowStateReg));
  }
  __syncthreads();
  const uint32_t sp = sm.sp;
  if (sp != kLeaf && warp == 0) {
    const uint32_t nl = warp_partition(d, nd.base, len, sp, rows_in, d.rows[(level & 1) ^ 1]);
    if (lane == 0) d.nd_lrows[k] = nl;
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kTbWarps * 32, 2) k_three_rows(Dev d, int level) {
  extern __shared__ __align__(16) unsigned char raw[];
  TbSmem& sm = *reinterpret_cast<TbSmem*>(raw);
  uint32_t* bits = reinterpret_cast<uint32_t*>(raw + sizeof(TbSmem));
  const uint32_t nn = d.nsmall[level];
  for (uint32_t i = blockIdx.x; i < nn; i += gridDim.x) three_rows(d, level, d.small[i], sm, bits);
}

// ---------------------------------------------------------------- at most 8 rows
struct TbFew {
  float score[256];  // by subset of the rows; -1 where a side is empty
  long long v[8];    // weighted targets
  uint32_t w[8];
  Perm perm;
};

__device__ void three_few(const Dev& d, int level, uint32_t k, TbFew& sm, uint32_t* bits) {
  const int lane = threadIdx.x & 31;
  const uint32_t* rows_in = d.rows[level & 1];
  uint32_t* rows_out = d.rows[(level & 1) ^ 1];
  NodeInfo<1> nd;
  load_node<1, 1>(d, k, level, nd);
  const int len = static_cast<int>(nd.len);
  const uint32_t words = (static_cast<uint32_t>(d.p_aug) + 31u) / 32u;
  __syncwarp();
  Perm P;
  node_perm(d, k, P);
  if (lane == 0) sm.perm = P;
  const bool v = lane < len;
  const uint32_t e = v ? rows_in[nd.base + lane] : 0u;
  if (lane < 8) {
    sm.w[lane] = v ? ent_w<1>(e) : 0u;
    sm.v[lane] = v ? static_cast<long long>(ent_w<1>(e)) * d.yreg[e >> 8] : 0ll;
  }
  for (uint32_t i = lane; i < words; i += 32u) bits[i] = 0u;
  __syncwarp();
  auto subset = [&](uint32_t m, long long& S, uint32_t& nL) {
    S = 0;
    nL = 0u;
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if ((m >> r) & 1u) {
        S += sm.v[r];
        nL += sm.w[r];
      }
  };
  for (uint32_t m = lane; m < (1u << len); m += 32u) {
    long long S;
    uint32_t nL;
    subset(m, S, nL);
    sm.score[m] = nL > 0u && nL < nd.n ? score_reg_any(d.wide_y, S, nd.SP, nL, nd.n) : -1.0f;
  }
  mark_columns(P, d.mtry, static_cast<uint32_t>(lane), 32u, bits);
  __syncwarp();
  const Perm* order = d.tie_break == 1 ? &sm.perm : nullptr;
  RegCand best;
  uint32_t bestm = 0u;
  const uint32_t quads = (static_cast<uint32_t>(d.p_aug) + 3u) / 4u;
  for (uint32_t q = lane; q < ((quads + 31u) & ~31u); q += 32u) {
    uint32_t x[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const uint32_t row = __shfl_sync(kFull, e, r) >> 8;
      x[r] = (r < len && q < quads)
                 ? *reinterpret_cast<const uint32_t*>(d.Xrow + static_cast<uint64_t>(row) * d.ldP + 4u * q)
                 : 0x02020202u;
    }
    uint32_t m0 = 0u, m1 = 0u;  // per column's byte: the rows with bin <= 0, <= 1
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      m0 |= (~(x[r] | (x[r] >> 1)) & 0x01010101u) << r;
      m1 |= (~(x[r] >> 1) & 0x01010101u) << r;
    }
    const uint32_t drawn = q < quads ? (bits[q >> 3] >> (4u * (q & 7u))) & 15u : 0u;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint32_t m = ((u & 1) ? m1 : m0) >> (8 * (u >> 1)) & 255u;
      const float sf = sm.score[m];
      if (!((drawn >> (u >> 1)) & 1u) || sf < 0.0f || sf < screen(best.sf)) continue;
      const uint32_t fb = ((4u * q + (u >> 1)) << 8) | (u & 1);
      // keys ascend within a lane unless equal scores go by drawing order
      if (m == bestm && !order && best.sf >= 0.0f) continue;
      long long S;
      uint32_t nL;
      subset(m, S, nL);
      const uint32_t before = best.fb;
      reg_offer(best, sf, S, nL, fb, nd.SP, nd.n, order);
      if (best.fb != before) bestm = m;
    }
  }
  reg_warp_best(best, nd.SP, nd.n, order);
  uint32_t sp = kLeaf;
  if (lane == 0) {
    sp = commit_reg(d, k, best, nd);
    atomicAdd(&d.counters[0], nd.len * (static_cast<unsigned long long>(d.mtry) + 12u + (sp != kLeaf ? 5u : 0u)));
  }
  sp = __shfl_sync(kFull, sp, 0);
  const bool split = sp != kLeaf;
  const uint32_t b = (v && split) ? row_bin(d, e >> 8, sp >> 8) : 0u;
  const bool gl = v && split && b <= (sp & 255u), gr = v && split && !gl;
  const unsigned bl = __ballot_sync(kFull, gl), br = __ballot_sync(kFull, gr);
  if (gl) rows_out[nd.base + __popc(bl & lanemask_lt())] = e;
  if (gr) rows_out[nd.base + __popc(bl) + __popc(br & lanemask_lt())] = e;
  if (split && lane == 0) d.nd_lrows[k] = __popc(bl);
}

__global__ void __launch_bounds__(256, 4) k_three_few(Dev d, int level) {
  extern __shared__ __align__(16) unsigned char raw[];
  const uint32_t words = (static_cast<uint32_t>(d.p_aug) + 31u) / 32u;
  const int warp = threadIdx.x >> 5;
  TbFew& sm = reinterpret_cast<TbFew*>(raw)[warp];
  uint32_t* bits = reinterpret_cast<uint32_t*>(raw + 8 * sizeof(TbFew)) + warp * words;
  const uint32_t nn = d.nmicro[level];
  const uint32_t nwarps = gridDim.x * 8u;
  for (uint32_t i = blockIdx.x * 8u + warp; i < nn; i += nwarps) three_few(d, level, d.micro[i], sm, bits);
}

size_t rows_smem(int p_aug) { return sizeof(TbSmem) + static_cast<size_t>((p_aug + 31) / 32) * 4; }
size_t few_smem(int p_aug) { return 8 * (sizeof(TbFew) + static_cast<size_t>((p_aug + 31) / 32) * 4); }

}  // namespace

// Grid sizes for a matrix of p_aug columns (the most of the session); 0 where
// the bit maps do not fit.
int setup_three_bins(int p_aug, int sms, int* grids) {
  grids[0] = grids[1] = 0;
  if (rows_smem(p_aug) > 113 * 1024 || few_smem(p_aug) > 113 * 1024) return 0;
  cudaError_t e = cudaSuccess;
  const void* f[2] = {reinterpret_cast<const void*>(&k_three_rows), reinterpret_cast<const void*>(&k_three_few)};
  const size_t smem[2] = {rows_smem(p_aug), few_smem(p_aug)};
  for (int i = 0; i < 2 && e == cudaSuccess; ++i) {
    int per_sm = 0;
    // one limit for every session of the process: what the check above allows
    e = cudaFuncSetAttribute(f[i], cudaFuncAttributeMaxDynamicSharedMemorySize, 113 * 1024);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f[i], 256, smem[i]);
    grids[i] = per_sm * sms;
  }
  return static_cast<int>(e);
}

int launch_three_bins(const Dev& d, int level, const int* grids, uint64_t nodes, cudaStream_t st, cudaStream_t st2) {
  const unsigned g0 = static_cast<unsigned>(nodes < static_cast<uint64_t>(grids[0]) ? nodes : grids[0]);
  const uint64_t warps8 = (nodes + 7u) / 8u;
  const unsigned g1 = static_cast<unsigned>(warps8 < static_cast<uint64_t>(grids[1]) ? warps8 : grids[1]);
  k_three_rows<<<g0 ? g0 : 1, kTbWarps * 32, rows_smem(d.p_aug), st>>>(d, level);
  k_three_few<<<g1 ? g1 : 1, 256, few_smem(d.p_aug), st2>>>(d, level);
  return 2;
}

}  // namespace bgb
