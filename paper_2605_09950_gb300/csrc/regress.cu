// Split search of regression nodes of at most 1024 rows over binned columns.
//
//   reg_few      nodes of at most 8 rows, a warp each, a column per lane: the
//                candidate of a row is the subset of the rows whose bins do not
//                exceed its own, one of at most 256, whose scores are
//                tabulated once per node.
//   reg_rows     9..32 rows (two nodes or one a warp): the left sums of all
//                candidates of a column are the product of the 0/1 matrix
//                "bin_s <= bin_r" by the rows' values, as in small.cu.  The
//                weighted targets are cut into six 11-bit limbs (the last one
//                signed) beside the weight: integers below 2048 are exact in
//                f16, their sums over 32 rows in f32, and a transpose over the
//                quad of lanes that shares a row gives every lane the exact
//                64-bit sum of its own row's candidate.
//   k_reg_record 33..1024 rows, a block each: 32 columns of all rows in a byte
//                tile (rows read by record, lanes over columns), a histogram
//                per warp and column of the weight and of 21-bit limbs of the
//                weighted target in separate 32-bit planes (native shared
//                memory atomics; a limb's sum over 1024 rows stays below 2^32),
//                then prefix sums and scores, each lane its own bins.
// Every lane keeps its best candidate exactly (regress.cuh).
//
// Measured: N = 10000, p = 50, all 100 columns tried, 100 trees, depth 16,
// 128 bins: 26.3 -> 16.1 ms an iteration (row-by-row sums through shuffles and
// 64-bit shared-memory atomics before).  Which problems they take: routes.h.
#include <algorithm>
#include <cstdint>

#include "regress.cuh"

namespace bgb {

namespace {

constexpr uint32_t kNoNode = 0xFFFFFFFFu;

// The node's columns in drawing order (in their own where every one is
// sampled and the order decides nothing): slots first, first + step, ... by
// this thread, each taken up as soon as the one before falls inside the
// permutation's domain.  Candidates are then keyed by slot (equal scores to
// the first drawn) or by column.
__device__ __forceinline__ void list_columns(const Dev& d, const Perm& P, uint32_t first, uint32_t step,
                                             uint16_t* feat) {
  const uint32_t mtry = static_cast<uint32_t>(d.mtry);
  if (mtry == P.n && d.tie_break == 0) {
    for (uint32_t s = first; s < P.n; s += step) feat[s] = static_cast<uint16_t>(s);
    return;
  }
  uint32_t s = first, x = first;
  while (s < mtry) {
    if (P.n > 1u) x = feistel8(P, x);
    if (x < P.n) {
      feat[s] = static_cast<uint16_t>(x);
      s += step;
      x = s;
    }
  }
}

__device__ __forceinline__ uint32_t key_of(const Dev& d, int slot, uint32_t f) {
  return (d.tie_break == 1 ? static_cast<uint32_t>(slot) : f) << 8;
}

// the candidate with its column in place of its slot
__device__ __forceinline__ RegCand by_column(const Dev& d, RegCand b, const uint16_t* feat) {
  if (d.tie_break == 1 && b.sf >= 0.0f) b.fb = (static_cast<uint32_t>(feat[b.fb >> 8]) << 8) | (b.fb & 255u);
  return b;
}

// ---------------------------------------------------------------- at most 8 rows
struct RegFew {
  float score[256];  // by subset of the rows; -1 where a side is empty
  long long v[8];    // weighted targets
  uint32_t w[8];
};

// ---------------------------------------------------------------- 9..32 rows
struct RegTile {
  uint32_t bins[32 * 17];  // [column][slot] halves, odd word pitch
};

struct RegWarp {
  union {
    RegFew few;
    RegTile tile;
  };
  uint16_t feat[2][kRegColumns];
};

__device__ void reg_few(const Dev& d, int level, uint32_t k, RegWarp& sm, unsigned long long& bytes) {
  const int lane = threadIdx.x & 31;
  const uint32_t* rows_in = d.rows[level & 1];
  uint32_t* rows_out = d.rows[(level & 1) ^ 1];
  NodeInfo<1> nd;
  load_node<1, 1>(d, k, level, nd);
  const int len = static_cast<int>(nd.len);
  Perm P;
  node_perm(d, k, P);
  __syncwarp();
  const bool v = lane < len;
  const uint32_t e = v ? rows_in[nd.base + lane] : 0u;
  if (lane < 8) {
    sm.few.w[lane] = v ? ent_w<1>(e) : 0u;
    sm.few.v[lane] = v ? static_cast<long long>(ent_w<1>(e)) * d.yreg[e >> 8] : 0ll;
  }
  list_columns(d, P, static_cast<uint32_t>(lane), 32u, sm.feat[0]);
  __syncwarp();
  auto subset = [&](uint32_t m, long long& S, uint32_t& nL) {
    S = 0;
    nL = 0u;
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if ((m >> r) & 1u) {
        S += sm.few.v[r];
        nL += sm.few.w[r];
      }
  };
  for (uint32_t m = lane; m < (1u << len); m += 32u) {
    long long S;
    uint32_t nL;
    subset(m, S, nL);
    sm.few.score[m] = nL > 0u && nL < nd.n ? score_reg_any(d.wide_y, S, nd.SP, nL, nd.n) : -1.0f;
  }
  __syncwarp();
  RegCand best;
  for (int j = lane; j < ((d.mtry + 31) & ~31); j += 32) {
    const bool in = j < d.mtry;
    const uint32_t f = in ? sm.feat[0][j] : 0u;
    uint32_t b[8], m[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const uint32_t row = __shfl_sync(kFull, e, r) >> 8;
      b[r] = (r < len && in) ? row_bin(d, row, f) : 0u;
      m[r] = 1u << r;
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      if (r >= len) break;
#pragma unroll
      for (int s = 0; s < r; ++s) {
        if (b[s] <= b[r]) m[r] |= 1u << s;
        if (b[r] <= b[s]) m[s] |= 1u << r;
      }
    }
    // the candidates that may come first (few), their subsets and bins by byte
    uint32_t cand = 0u;
    unsigned long long ms = 0ull, xs = 0ull;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      if (r >= len) break;
      const float sf = sm.few.score[m[r]];
      if (in && sf >= 0.0f && sf >= screen(best.sf)) cand |= 1u << r;
      ms |= static_cast<unsigned long long>(m[r]) << (8 * r);
      xs |= static_cast<unsigned long long>(b[r]) << (8 * r);
    }
    for (; cand; cand &= cand - 1u) {
      const int r = __ffs(cand) - 1;
      const uint32_t sub = static_cast<uint32_t>(ms >> (8 * r)) & 255u;
      long long S;
      uint32_t nL;
      subset(sub, S, nL);
      reg_offer(best, sm.few.score[sub], S, nL, key_of(d, j, f) | (static_cast<uint32_t>(xs >> (8 * r)) & 255u), nd.SP,
                nd.n, nullptr);
    }
  }
  reg_warp_best(best, nd.SP, nd.n, nullptr);
  uint32_t sp = kLeaf;
  if (lane == 0) {
    sp = commit_reg(d, k, by_column(d, best, sm.feat[0]), nd);
    bytes += nd.len * (static_cast<unsigned long long>(d.mtry) + 12u + (sp != kLeaf ? 5u : 0u));
  }
  sp = __shfl_sync(kFull, sp, 0);
  const bool split = sp != kLeaf;
  const uint32_t x = (v && split) ? row_bin(d, e >> 8, sp >> 8) : 0u;
  const bool gl = v && split && x <= (sp & 255u), gr = v && split && !gl;
  const unsigned bl = __ballot_sync(kFull, gl), br = __ballot_sync(kFull, gr);
  if (gl) rows_out[nd.base + __popc(bl & lanemask_lt())] = e;
  if (gr) rows_out[nd.base + __popc(bl) + __popc(br & lanemask_lt())] = e;
  if (split && lane == 0) d.nd_lrows[k] = __popc(bl);
}

template <int SEG>
__device__ void reg_rows(const Dev& d, int level, uint32_t k, RegWarp& sm, unsigned long long& bytes) {
  constexpr int NSEG = 32 / SEG;
  const int lane = threadIdx.x & 31;
  const int hl = lane & (SEG - 1), seg = lane / SEG;  // slot order: a node's rows are consecutive lanes
  const int g = lane >> 2, t = lane & 3;              // fragment order: this lane scores slot 8 t + g
  const int sseg = SEG == 16 ? t >> 1 : 0;
  const uint32_t* rows_in = d.rows[level & 1];
  uint32_t* rows_out = d.rows[(level & 1) ^ 1];
  const bool has = k != kNoNode;
  NodeInfo<1> nd;
  nd.base = 0;
  nd.len = 0u;
  nd.n = 0u;
  nd.SP = 0;
  __syncwarp();
  if (has) {
    load_node<1, 1>(d, k, level, nd);
    Perm P;
    node_perm(d, k, P);
    list_columns(d, P, static_cast<uint32_t>(hl), SEG, sm.feat[seg]);
  }
  const bool v = hl < static_cast<int>(nd.len);
  const uint32_t e = v ? rows_in[nd.base + hl] : 0u;
  const uint32_t row = e >> 8;
  const long long val = v ? static_cast<long long>(ent_w<1>(e)) * d.yreg[row] : 0ll;
  const unsigned vmask = __ballot_sync(kFull, v);
  __syncwarp();
  // value factor: column g < 6 holds limb g, column 7 the weight
  uint32_t B[2][2];
#pragma unroll
  for (int kb = 0; kb < 2; ++kb)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t x[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int slot = 16 * kb + 8 * h + 2 * t + u;
        const long long y = __shfl_sync(kFull, val, slot);
        const uint32_t w = ent_w<1>(__shfl_sync(kFull, e, slot));
        const int limb = g < 5 ? static_cast<int>(y >> (11 * g)) & 2047 : static_cast<int>(y >> 55);
        x[u] = half_bits(g < 6 ? limb : (g == 7 ? static_cast<int>(w) : 0));
      }
      B[kb][h] = x[0] | (x[1] << 16);
    }
  const uint32_t n_own = __shfl_sync(kFull, nd.n, sseg * SEG);
  const long long SP_own = __shfl_sync(kFull, nd.SP, sseg * SEG);
  const bool own = (vmask >> (8 * t + g)) & 1u;
  RegCand best;
  for (int r0 = 0; r0 < d.mtry; r0 += 32) {
    const int nf = min(32, d.mtry - r0);
    uint32_t f[NSEG];
#pragma unroll
    for (int s = 0; s < NSEG; ++s) f[s] = lane < nf ? sm.feat[s][r0 + lane] : 0u;
    if (r0 > 0) __syncwarp();
#pragma unroll
    for (int hb = 0; hb < 2; ++hb) {
      uint32_t b[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int slot = 16 * hb + q;
        const uint32_t r = __shfl_sync(kFull, row, slot);
        b[q] = 0u;
        if (lane < nf && ((vmask >> slot) & 1u)) b[q] = row_bin(d, r, f[slot / SEG]);
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) sm.tile.bins[lane * 17 + 8 * hb + q] = b[2 * q] | (b[2 * q + 1] << 16);
    }
    __syncwarp();
    for (int j = 0; j < nf; ++j) {
      const uint32_t* tw = sm.tile.bins + j * 17;
      const uint16_t* th = reinterpret_cast<const uint16_t*>(tw);
      uint32_t A[4], R[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        A[i] = tw[4 * i + t];
        const uint32_t h = th[8 * i + g];
        R[i] = __byte_perm(h, h, 0x1010);
      }
      // the quad's parts of the sums of slots 8 i + g: limbs 2 t and 2 t + 1, or the weight
      int m[4];
#pragma unroll
      for (int mb = 0; mb < 2; ++mb) {
        float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int kb = 0; kb < 2; ++kb) {
          if (SEG < 32 && mb != kb) continue;
          const uint32_t a0 = le_h2(A[2 * kb], R[2 * mb]), a1 = le_h2(A[2 * kb], R[2 * mb + 1]),
                         a2 = le_h2(A[2 * kb + 1], R[2 * mb]), a3 = le_h2(A[2 * kb + 1], R[2 * mb + 1]);
          asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
              "{%0,%1,%2,%3};"
              : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
              : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(B[kb][0]), "r"(B[kb][1]));
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {  // integers of magnitude below 2^22 by their float's bits
          const int x = __float_as_int(c[2 * r] + 12582912.0f) - 0x4B400000,
                    y = __float_as_int(c[2 * r + 1] + 12582912.0f) - 0x4B400000;
          m[2 * mb + r] = t == 3 ? y : x + (y << 11);
        }
      }
      // transpose over the quad: this lane's slot is 8 t + g
      const bool o = t & 1, h = t & 2;
      const int x0 = __shfl_xor_sync(kFull, o ? m[0] : m[1], 1), x1 = __shfl_xor_sync(kFull, o ? m[2] : m[3], 1);
      const int a0 = o ? m[1] : m[0], a1 = o ? m[3] : m[2];
      const int p2 = __shfl_xor_sync(kFull, h ? a0 : a1, 2), p3 = __shfl_xor_sync(kFull, h ? x0 : x1, 2);
      const int p0 = h ? a1 : a0, p1 = h ? x1 : x0;  // of lanes t, t ^ 1; p2, p3: of t ^ 2, t ^ 3
      const int u0 = o ? p1 : p0, u1 = o ? p0 : p1, u2 = o ? p3 : p2, u3 = o ? p2 : p3;
      const int v0 = h ? u2 : u0, v1 = h ? u3 : u1, v2 = h ? u0 : u2, v3 = h ? u1 : u3;  // of lanes 0..3
      const long long S = static_cast<long long>(v0) + static_cast<long long>(v1) * (1ll << 22) +
                          static_cast<long long>(static_cast<unsigned long long>(static_cast<long long>(v2)) << 44);
      const uint32_t nL = static_cast<uint32_t>(v3);
      if (own && nL < n_own)
        reg_offer(best, score_reg_any(d.wide_y, S, SP_own, nL, n_own), S, nL,
                  key_of(d, r0 + j, sm.feat[sseg][r0 + j]) | th[8 * t + g], SP_own, n_own, nullptr);
    }
  }
#pragma unroll
  for (int x = 1; x < 32; x <<= 1) {
    if (x == 2 && SEG == 16) continue;
    const float sf = __shfl_xor_sync(kFull, best.sf, x);
    const long long S = __shfl_xor_sync(kFull, best.S, x);
    const uint32_t nL = __shfl_xor_sync(kFull, best.nL, x), fb = __shfl_xor_sync(kFull, best.fb, x);
    reg_offer(best, sf, S, nL, fb, SP_own, n_own, nullptr);
  }
  const int src = SEG == 16 ? 2 * seg : 0;  // a lane that scored this lane's node
  best.sf = __shfl_sync(kFull, best.sf, src);
  best.S = __shfl_sync(kFull, best.S, src);
  best.nL = __shfl_sync(kFull, best.nL, src);
  best.fb = __shfl_sync(kFull, best.fb, src);
  uint32_t sp = kLeaf;
  if (has && hl == 0) {
    sp = commit_reg(d, k, by_column(d, best, sm.feat[seg]), nd);
    bytes += nd.len * (static_cast<unsigned long long>(d.mtry) + 12u + (sp != kLeaf ? 5u : 0u));
  }
  sp = __shfl_sync(kFull, sp, seg * SEG);
  const bool split = has && sp != kLeaf;
  const uint32_t x = (v && split) ? row_bin(d, row, sp >> 8) : 0u;
  const bool gl = v && split && x <= (sp & 255u), gr = v && split && !gl;
  const unsigned sm_mask = SEG == 32 ? kFull : (((1u << (SEG & 31)) - 1u) << (seg * SEG));
  const unsigned bl = __ballot_sync(kFull, gl) & sm_mask, br = __ballot_sync(kFull, gr) & sm_mask;
  if (gl) rows_out[nd.base + __popc(bl & lanemask_lt())] = e;
  if (gr) rows_out[nd.base + __popc(bl) + __popc(br & lanemask_lt())] = e;
  if (split && hl == 0) d.nd_lrows[k] = __popc(bl);
}

__global__ void __launch_bounds__(256, 3) k_reg_rows(Dev d, int level) {
  __shared__ RegWarp warps[8];
  RegWarp& sm = warps[threadIdx.x >> 5];
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t nsmall = d.nsmall[level], ntiny = d.ntiny[level];
  const uint32_t end16 = nsmall + (ntiny + 1u) / 2u, end8 = end16 + d.nmicro[level];
  unsigned long long bytes = 0;
  for (uint32_t it = gwarp; it < end8; it += nwarps) {
    if (it < nsmall) {
      reg_rows<32>(d, level, d.small[it], sm, bytes);
    } else if (it < end16) {
      const uint32_t i = 2u * (it - nsmall) + (lane >> 4);
      reg_rows<16>(d, level, i < ntiny ? d.small[d.small_cap - 1u - i] : kNoNode, sm, bytes);
    } else {
      reg_few(d, level, d.micro[it - end16], sm, bytes);
    }
  }
  if (bytes) atomicAdd(&d.counters[0], bytes);
}

// ---------------------------------------------------------------- 33..1024 rows
template <int ROWS, int WARPS>
struct RegSmem {
  uint4 rw[ROWS];                      // per row: weight, 21-bit limbs of the weighted target (the last
                                       //   one signed: the third, or the second where two are enough)
  uint32_t hist[WARPS][4 * 256];       // planes of the four, by bin
  uint32_t tile[32 * (ROWS / 4 + 1)];  // [column][row] bins; odd word pitch
  RegCand best[WARPS];
  Perm perm;
  uint32_t left[ROWS / 32];
  uint16_t feat[kRegColumns];
  uint32_t sp;
};

template <int ROWS, int WARPS>
__device__ __forceinline__ void reg_record(const Dev& d, int level, uint32_t k, RegSmem<ROWS, WARPS>& sm) {
  constexpr int CH = ROWS / (32 * WARPS), PITCH = ROWS / 4 + 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t* rows_in = d.rows[level & 1];
  NodeInfo<1> nd;
  load_node<1, 1>(d, k, level, nd);
  const uint32_t len = nd.len, chunks = (len + 31u) / 32u;
  if (threadIdx.x == 0) node_perm(d, k, sm.perm);
  uint32_t e[CH];
#pragma unroll
  for (int i = 0; i < CH; ++i) {
    const uint32_t c = warp + WARPS * i, r = c * 32u + lane;
    e[i] = r < len ? rows_in[nd.base + r] : 0u;
    if (c < chunks) {
      const uint32_t w = r < len ? ent_w<1>(e[i]) : 0u;
      const long long v = r < len ? static_cast<long long>(w) * d.yreg[e[i] >> 8] : 0ll;
      const uint32_t hi = static_cast<uint32_t>(v >> 21);
      sm.rw[r] = make_uint4(w, static_cast<uint32_t>(v) & 0x1FFFFFu, d.wide_y ? hi & 0x1FFFFFu : hi,
                            static_cast<uint32_t>(v >> 42));
    }
  }
  __syncthreads();
  const Perm P = sm.perm;
  list_columns(d, P, threadIdx.x, WARPS * 32, sm.feat);
  __syncthreads();
  const int bpl = lane_bins(d.B);
  uint32_t* hw = sm.hist[warp];
  RegCand best;
  for (int r0 = 0; r0 < d.mtry; r0 += 32) {
    const int nf = min(32, d.mtry - r0);
    const uint32_t f = lane < nf ? sm.feat[r0 + lane] : 0u;
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
      const uint8_t* tb = reinterpret_cast<const uint8_t*>(sm.tile + j * PITCH);
      for (uint32_t r = lane; r < len; r += 32u) {
        const uint32_t b = tb[r];
        const uint4 x = sm.rw[r];
        atomicAdd(hw + b, x.x);
        atomicAdd(hw + 256 + b, x.y);
        atomicAdd(hw + 512 + b, x.z);
        if (d.wide_y) atomicAdd(hw + 768 + b, x.w);
      }
      __syncwarp();
      // the lane's bins: weight and exact sum each, then their prefix sums
      uint32_t h[4][8];
#pragma unroll
      for (int w = 0; w < 4; ++w)
        if (w < 3 || d.wide_y) ld_bins(hw + 256 * w + lane * bpl, bpl, h[w]);
      long long bs[8];
      uint32_t wsum = 0u;
      long long ssum = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const long long top = static_cast<long long>(static_cast<int32_t>(d.wide_y ? h[3][q] : h[2][q]));
        bs[q] = d.wide_y ? h[1][q] + (static_cast<long long>(h[2][q]) << 21) + top * (1ll << 42)
                         : h[1][q] + top * (1ll << 21);
        wsum += h[0][q];
        ssum += bs[q];
      }
      uint32_t nL = warp_excl_scan_u32(wsum, lane);
      long long S = warp_excl_scan_i64(ssum, lane);
      const uint32_t key = key_of(d, r0 + j, sm.feat[r0 + j]);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (q >= bpl || h[0][q] == 0u) continue;  // an empty bin repeats the partition of the one below
        nL += h[0][q];
        S += bs[q];
        if (nL < nd.n)
          reg_offer(best, score_reg_any(d.wide_y, S, nd.SP, nL, nd.n), S, nL, key | static_cast<uint32_t>(lane * bpl + q), nd.SP,
                    nd.n, nullptr);
      }
      const uint32_t zero[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll
      for (int w = 0; w < 4; ++w)
        if (w < 3 || d.wide_y) st_bins(hw + 256 * w + lane * bpl, bpl, zero);
      __syncwarp();
    }
    if (r0 + 32 < d.mtry) __syncthreads();  // the tile is refilled
  }
  reg_warp_best(best, nd.SP, nd.n, nullptr);
  if (lane == 0) sm.best[warp] = best;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < WARPS; ++w)
      reg_offer(best, sm.best[w].sf, sm.best[w].S, sm.best[w].nL, sm.best[w].fb, nd.SP, nd.n, nullptr);
    sm.sp = commit_reg(d, k, by_column(d, best, sm.feat), nd);
    const unsigned long long rd = static_cast<unsigned long long>(d.mtry) + 12u + (sm.sp != kLeaf ? 5u : 0u);
    atomicAdd(&d.counters[0], len * rd);
    atomicAdd(&d.counters[2], static_cast<unsigned long long>(len) * (d.mtry + kRowStateReg));
  }
  __syncthreads();
  const uint32_t sp = sm.sp;
  if (sp != kLeaf) {
    const uint32_t total = block_partition<CH, WARPS>(
        e, len, nd.base, d.rows[(level & 1) ^ 1], sm.left,
        [&](int i, uint32_t) { return row_bin(d, e[i] >> 8, sp >> 8) <= (sp & 255u); });
    if (threadIdx.x == 0) d.nd_lrows[k] = total;
  }
  __syncthreads();
}

template <int ROWS, int WARPS, int MINB>
__global__ void __launch_bounds__(WARPS * 32, MINB) k_reg_record(Dev d, int level) {
  extern __shared__ __align__(16) unsigned char raw[];
  auto& sm = *reinterpret_cast<RegSmem<ROWS, WARPS>*>(raw);
  const uint32_t nn = d.nrec[3 * level + (ROWS == 256 ? 0 : 1)];
  if (blockIdx.x >= nn) return;
  for (uint32_t i = threadIdx.x; i < WARPS * 1024; i += WARPS * 32) sm.hist[0][i] = 0u;
  __syncthreads();
  for (uint32_t i = blockIdx.x; i < nn; i += gridDim.x)
    reg_record<ROWS, WARPS>(d, level, ROWS == 256 ? d.rec[i] : d.rec2[i], sm);
}

template <int ROWS, int WARPS, int MINB>
cudaError_t setup(int sms, int* grid) {
  auto* f = &k_reg_record<ROWS, WARPS, MINB>;
  const int smem = static_cast<int>(sizeof(RegSmem<ROWS, WARPS>));
  cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  int per_sm = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, WARPS * 32, smem);
  *grid = (per_sm < 1 ? 1 : per_sm) * sms;
  return e;
}

}  // namespace

int setup_regress(int sms, int* grids) {
  cudaError_t e = setup<256, 4, 5>(sms, grids);
  if (e == cudaSuccess) e = setup<1024, 8, 2>(sms, grids + 1);
  int per_sm = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_reg_rows, 256, 0);
  grids[2] = (per_sm < 1 ? 1 : per_sm) * sms;
  return static_cast<int>(e);
}

int launch_regress(const Dev& d, int level, const int* grids, uint64_t nodes, cudaStream_t st, cudaStream_t st2) {
  auto grid = [&](int i, uint64_t most) {
    return static_cast<unsigned>(std::max<uint64_t>(1, std::min<uint64_t>(static_cast<uint64_t>(grids[i]), most)));
  };
  const uint64_t M = static_cast<uint64_t>(d.M), N = static_cast<uint64_t>(d.N);
  int n = 0;
  if (d.reg_rows) {
    k_reg_rows<<<grid(2, (nodes + 7) / 8), 256, 0, st2>>>(d, level);
    ++n;
  }
  if (d.rec_rows > 256u) {
    k_reg_record<1024, 8, 2><<<grid(1, std::min(nodes, M * (N / 257 + 1))), 256, sizeof(RegSmem<1024, 8>), st>>>(d, level);
    ++n;
  }
  if (d.rec_rows > 0u) {
    k_reg_record<256, 4, 5><<<grid(0, std::min(nodes, M * (N / 33 + 1))), 128, sizeof(RegSmem<256, 4>), st>>>(d, level);
    ++n;
  }
  return n;
}

}  // namespace bgb
