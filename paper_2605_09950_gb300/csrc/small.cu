// Split search of a level's nodes of few rows (classification): the left
// class counts of every candidate of a (node, feature) come from one small
// matrix product on the tensor cores.
//
// A candidate is "rows with bin <= the bin of row r go left" (an empty bin
// repeats the partition of the nearest bin below that holds a row, and loses
// the tie to it).  With Le[r][s] = 1 where bin_s <= bin_r, the left totals of
// all candidates of a feature are the product Le (rows x rows) by the rows'
// weights per class (rows x classes): both exact in f16 with f32 sums (0/1
// times integers of at most 2048, sums below 2^24).  The factor Le is built in
// registers by half-precision comparisons straight into mma.sync operand
// fragments, and the other factor is the same for all features of a node, so a
// feature costs a warp 4 to 16 comparisons, 4 to 12 matrix instructions and
// one score per row.  These products are 32 x 32 x 8 (64 x 64 x 8): far below
// the 128-row tiles of tcgen05.mma, whose operands would also have to go
// through shared memory; the warp-level instruction takes them from registers.
//
// Nodes and layouts: slots are a warp's rows.
//   few_rows<SEG>  nodes of at most SEG rows and total weight <= kFewWeight,
//                  32 / SEG nodes a warp, one slot per lane (SEG = 8, 16, 32);
//                  off-diagonal blocks of Le between nodes are not computed.
//   mid_rows       one node of at most 64 rows a warp, any weight.
// A node's bins are read by record from the row-major copy, lanes over the
// features of one row, 32 features at a time: one load instruction then
// touches the row's own record (8 lines of 128 B at 1000 columns) instead of
// 32 of them.
//
// Scores: with q_k = l_k n - c_k n_L (l, c: left and node counts of class k),
// the impurity decrease of a candidate is s / (n_L n_R n), s = sum_k q_k^2.
// few_rows folds n and c into the weights, so the product gives q_k, and s is
// exact in f32 (below 2^23 for n <= 66); every lane keeps its row's best
// candidate exactly, comparing s_a den_b with s_b den_a in 64-bit integers.
// mid_rows takes every feature's best float score first, then compares the
// features inside the window of the best one exactly.
//
// Measured (one iteration, before: ballots over the bin bits and 5 population
// counts per class for <= 32 rows, a 256-bin shared-memory histogram for
// 33..64): N = 1e6, p = 500, 5 classes, 300 trees, depth 20: 1424 -> 1148 ms;
// N = 30011, p = 203, 8 classes, 100 trees: 13.4 -> 10.2 ms; N = 1e5,
// p = 1000, 2 classes, 500 trees: 185 -> 164 ms.  Bound by the record reads
// (about 20 sectors of 32 B for 31 of 1000 columns) and by issue.
#include <cstdint>
#include <type_traits>

#include <cuda_fp16.h>

#include "split.cuh"

namespace bgb {

namespace {

constexpr uint32_t kNoNode = 0xFFFFFFFFu;

// 1.0 in each half where a <= b (bins as the bit patterns of halves: the order
// of non-negative halves is the order of their bits)
__device__ __forceinline__ uint32_t le_h2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("set.le.f16x2.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t pack_h2(int lo, int hi) {
  const __half2 h = __halves2half2(__int2half_rn(lo), __int2half_rn(hi));
  return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ uint32_t dup_h(uint32_t h) { return __byte_perm(h, h, 0x1010); }

// integer value of a float in [0, 2^23) that holds one
__device__ __forceinline__ uint32_t f23_to_u32(float v) { return __float_as_uint(v + 8388608.0f) & 0x7FFFFFu; }

// Four values per lane, one per row group i, summed over the four lanes of a
// quad: lane t of the quad gets the sum of group t.
template <typename T>
__device__ __forceinline__ T quad_sum_own(const T (&p)[4], int t) {
  const bool o = t & 1, h = t & 2;
  const T x = __shfl_xor_sync(kFull, o ? p[0] : p[1], 1), y = __shfl_xor_sync(kFull, o ? p[2] : p[3], 1);
  const T k0 = (o ? p[1] : p[0]) + x, k1 = (o ? p[3] : p[2]) + y;
  return (h ? k1 : k0) + __shfl_xor_sync(kFull, h ? k0 : k1, 2);
}

template <typename T>
__device__ __forceinline__ T pick4(T v0, T v1, T v2, T v3, int t) {
  const T a = (t & 1) ? v1 : v0, b = (t & 1) ? v3 : v2;
  return (t & 2) ? b : a;
}

// ---------------------------------------------------------------- at most 32 rows
// A warp's tile: the bins of 32 features by slot, one half each (an odd word
// pitch: lanes over features write, and lanes over slots read, without bank
// conflicts), the features' keys, and the nodes' class totals.
struct FewTile {
  uint32_t bins[32 * 17];
  uint32_t key[32 * 4];  // [feature][node]
  uint32_t tot[4 * 8];   // [node][class]
};

template <int CM, int SEG>
__device__ void few_rows(const Dev& d, int level, uint32_t k, FewTile& sm, unsigned long long& bytes) {
  constexpr int NSEG = 32 / SEG;
  const int lane = threadIdx.x & 31;
  const int hl = lane & (SEG - 1), seg = lane / SEG;  // slot order: a node's rows are consecutive lanes
  const int g = lane >> 2, t = lane & 3;              // fragment order: this lane scores slot 8 t + g
  const int sseg = SEG == 8 ? t : (SEG == 16 ? t >> 1 : 0);
  const uint32_t* rows_in = d.rows[level & 1];
  uint32_t* rows_out = d.rows[(level & 1) ^ 1];
  const bool has = k != kNoNode;
  NodeInfo<CM> nd;
  nd.base = 0;
  nd.len = 0u;
  nd.n = 0u;
#pragma unroll
  for (int c = 0; c < CM; ++c) nd.cp[c] = 0u;
  Perm P;
  if (has) {
    load_node<0, CM>(d, k, level, nd);
    node_perm(d, k, P);
  }
  __syncwarp();  // the previous nodes' tile is read no more
  if (hl == 0) {
#pragma unroll
    for (int c = 0; c < 8; ++c) sm.tot[seg * 8 + c] = c < CM ? nd.cp[c < CM ? c : 0] : 0u;
  }
  const bool v = hl < static_cast<int>(nd.len);
  const uint32_t e = v ? rows_in[nd.base + hl] : 0u;
  const uint32_t row = e >> 8;
  const unsigned vmask = __ballot_sync(kFull, v);
  __syncwarp();
  // weight factor, as matrix fragments: slot s of class column g holds
  // w_s (n [y_s = g] - c_g); two classes need one column (q_1 = -q_0), so even
  // columns hold it and odd ones w_s, which gives n_L in the same product
  uint32_t Bq[2][2], Bw[2][2];
#pragma unroll
  for (int kb = 0; kb < 2; ++kb)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int s = (16 * kb + 8 * h) / SEG;
      const int ns = static_cast<int>(__shfl_sync(kFull, nd.n, s * SEG));
      const int cls = CM == 2 ? 0 : g;
      const int cg = static_cast<int>(sm.tot[s * 8 + cls]);
      int q[2], w[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const uint32_t ek = __shfl_sync(kFull, e, 16 * kb + 8 * h + 2 * t + u);
        w[u] = static_cast<int>(ent_w<0>(ek));
        q[u] = w[u] * ((static_cast<int>(ent_y(ek)) == cls ? ns : 0) - cg);
        if (CM == 2 && (g & 1)) q[u] = w[u];
      }
      Bq[kb][h] = pack_h2(q[0], q[1]);
      if (CM > 2) Bw[kb][h] = pack_h2(w[0], w[1]);
    }
  const uint32_t n_own = __shfl_sync(kFull, nd.n, sseg * SEG);
  const bool own = (vmask >> (8 * t + g)) & 1u;
  uint32_t bs = 0u, bden = 1u, bkey = 0xFFFFFFFFu;  // this slot's best candidate: s, n_L n_R, key
  for (int r0 = 0; r0 < d.mtry; r0 += 32) {
    const int nf = min(32, d.mtry - r0);
    uint32_t f[NSEG];
#pragma unroll
    for (int s = 0; s < NSEG; ++s) {
      Perm Q;
      Q.n = static_cast<uint32_t>(d.p_aug);
      Q.half = __shfl_sync(kFull, P.half, s * SEG);
      Q.mask = __shfl_sync(kFull, P.mask, s * SEG);
#pragma unroll
      for (int q = 0; q < 8; ++q) Q.key[q] = __shfl_sync(kFull, P.key[q], s * SEG);
      const bool any = (vmask >> (s * SEG)) & 1u;
      f[s] = (any && lane < nf) ? perm_apply(Q, static_cast<uint32_t>(r0 + lane)) : 0u;
    }
    if (r0 > 0) __syncwarp();
#pragma unroll
    for (int s = 0; s < NSEG; ++s)
      sm.key[lane * NSEG + s] = (d.tie_break == 1 ? static_cast<uint32_t>(r0 + lane) : f[s]) << 8;
#pragma unroll
    for (int hb = 0; hb < 2; ++hb) {  // 16 rows' records in flight
      uint32_t b[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int slot = 16 * hb + q;
        const uint32_t r = __shfl_sync(kFull, row, slot);
        b[q] = 0u;
        if (lane < nf && ((vmask >> slot) & 1u)) b[q] = row_bin(d, r, f[slot / SEG]);
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) sm.bins[lane * 17 + 8 * hb + q] = b[2 * q] | (b[2 * q + 1] << 16);
    }
    __syncwarp();
    for (int j = 0; j < nf; ++j) {
      const uint32_t* tw = sm.bins + j * 17;
      const uint16_t* th = reinterpret_cast<const uint16_t*>(tw);
      uint32_t A[4], R[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        A[i] = tw[4 * i + t];       // bins of slots 8 i + 2 t and + 1
        R[i] = dup_h(th[8 * i + g]);  // bin of slot 8 i + g
      }
      float q[2][4], w[2][4];
#pragma unroll
      for (int mb = 0; mb < 2; ++mb) {
#pragma unroll
        for (int x = 0; x < 4; ++x) q[mb][x] = w[mb][x] = 0.0f;
#pragma unroll
        for (int kb = 0; kb < 2; ++kb) {
          if (SEG < 32 && mb != kb) continue;
          const uint32_t a0 = le_h2(A[2 * kb], R[2 * mb]);
          const uint32_t a1 = SEG == 8 ? 0u : le_h2(A[2 * kb], R[2 * mb + 1]);
          const uint32_t a2 = SEG == 8 ? 0u : le_h2(A[2 * kb + 1], R[2 * mb]);
          const uint32_t a3 = le_h2(A[2 * kb + 1], R[2 * mb + 1]);
          mma16816(q[mb], a0, a1, a2, a3, Bq[kb][0], Bq[kb][1]);
          if (CM > 2) mma16816(w[mb], a0, a1, a2, a3, Bw[kb][0], Bw[kb][1]);
        }
      }
      float s, nL;
      if (CM == 2) {
        const float q0 = pick4(q[0][0], q[0][2], q[1][0], q[1][2], t);
        nL = pick4(q[0][1], q[0][3], q[1][1], q[1][3], t);
        s = 2.0f * q0 * q0;
      } else {
        float p[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float x = q[i >> 1][2 * (i & 1)], y = q[i >> 1][2 * (i & 1) + 1];
          p[i] = fmaf(x, x, y * y);
        }
        s = quad_sum_own(p, t);
        nL = pick4(w[0][0], w[0][2], w[1][0], w[1][2], t);
      }
      const uint32_t si = f23_to_u32(s), nl = f23_to_u32(nL);
      if (own && si > 0u) {  // s = 0: no decrease (n_L = n among them)
        const uint32_t den = nl * (n_own - nl);
        const uint64_t x = static_cast<uint64_t>(si) * bden, y = static_cast<uint64_t>(bs) * den;
        if (x >= y) {
          const uint32_t key = sm.key[j * NSEG + sseg] | th[8 * t + g];
          if (x > y || key < bkey) {
            bs = si;
            bden = den;
            bkey = key;
          }
        }
      }
    }
  }
  // the node's best: butterfly over the lanes that score its slots
#pragma unroll
  for (int m = 1; m < 32; m <<= 1) {
    if ((m == 1 && SEG == 8) || (m == 2 && SEG <= 16)) continue;
    const uint32_t os = __shfl_xor_sync(kFull, bs, m), od = __shfl_xor_sync(kFull, bden, m),
                   ok = __shfl_xor_sync(kFull, bkey, m);
    const uint64_t x = static_cast<uint64_t>(os) * bden, y = static_cast<uint64_t>(bs) * od;
    if (x > y || (x == y && ok < bkey)) {
      bs = os;
      bden = od;
      bkey = ok;
    }
  }
  const int src = SEG == 8 ? seg : (SEG == 16 ? 2 * seg : 0);
  bs = __shfl_sync(kFull, bs, src);
  bkey = __shfl_sync(kFull, bkey, src);
  const bool split = has && bs > 0u;
  uint32_t feat = bkey >> 8;
  if (split && d.tie_break == 1) feat = perm_apply(P, feat);
  const uint32_t bin = bkey & 255u;
  const uint32_t br = (v && split) ? row_bin(d, row, feat) : 0u;
  const bool gl = v && split && br <= bin, gr = v && split && !gl;
  // left class counts: bytes of one 64-bit word (at most kFewWeight each)
  unsigned long long cnt = gl ? static_cast<unsigned long long>(ent_w<0>(e)) << (8 * ent_y(e)) : 0ull;
#pragma unroll
  for (int m = SEG / 2; m > 0; m >>= 1) cnt += __shfl_xor_sync(kFull, cnt, m);
  if (has && hl == 0) {
    uint32_t cL[CM], nL = 0u;
#pragma unroll
    for (int c = 0; c < CM; ++c) {
      cL[c] = static_cast<uint32_t>(cnt >> (8 * c)) & 255u;
      nL += cL[c];
    }
    commit_counts<CM>(d, k, split, feat, bin, nL, cL, bs, nd.n);
    bytes += static_cast<unsigned long long>(nd.len) * (d.mtry + 4ull);
  }
  // stable partition: left rows in order, then right rows in order
  const unsigned sm_mask = SEG == 32 ? kFull : (((1u << (SEG & 31)) - 1u) << (seg * SEG));
  const unsigned bl = __ballot_sync(kFull, gl) & sm_mask, brm = __ballot_sync(kFull, gr) & sm_mask;
  const uint32_t nl = __popc(bl);
  if (gl) rows_out[nd.base + __popc(bl & lanemask_lt())] = e;
  if (gr) rows_out[nd.base + nl + __popc(brm & lanemask_lt())] = e;
  if (split && hl == 0) {
    d.nd_lrows[k] = nl;
    bytes += static_cast<unsigned long long>(nd.len) * 5ull;
  }
}

// ---------------------------------------------------------------- at most 64 rows
struct MidTile {
  uint32_t bins[32 * 33];
  uint32_t key[32];
  uint32_t tot[8];
};

// q_k of the candidates of rows 16 mb + g and 16 mb + 8 + g (this lane's two
// class columns, or q_0 alone for two classes) and their n_L, exact
template <int CM>
__device__ __forceinline__ void mid_block(const uint32_t (&A)[8], uint32_t R0, uint32_t R1, const uint32_t (&B)[4][2],
                                          const uint32_t (&Bw)[4][2], int nb, float n, float c0, float c1,
                                          float (&q0)[2], float (&q1)[2], float (&nL)[2]) {
  float a[4] = {0.0f, 0.0f, 0.0f, 0.0f}, w[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int kb = 0; kb < 4; ++kb)
    if (kb < nb) {
      const uint32_t a0 = le_h2(A[2 * kb], R0), a1 = le_h2(A[2 * kb], R1), a2 = le_h2(A[2 * kb + 1], R0),
                     a3 = le_h2(A[2 * kb + 1], R1);
      mma16816(a, a0, a1, a2, a3, B[kb][0], B[kb][1]);
      if (CM > 2) mma16816(w, a0, a1, a2, a3, Bw[kb][0], Bw[kb][1]);
    }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    nL[r] = CM == 2 ? a[2 * r + 1] : w[2 * r];
    q0[r] = a[2 * r] * n - c0 * nL[r];  // products of integers below 2^24: exact
    q1[r] = CM == 2 ? 0.0f : a[2 * r + 1] * n - c1 * nL[r];
  }
}

template <int CM>
__device__ void mid_rows(const Dev& d, int level, uint32_t k, MidTile& sm, unsigned long long& bytes) {
  const int lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const uint32_t* rows_in = d.rows[level & 1];
  uint32_t* rows_out = d.rows[(level & 1) ^ 1];
  NodeInfo<CM> nd;
  load_node<0, CM>(d, k, level, nd);
  Perm P;
  node_perm(d, k, P);
  const int len = static_cast<int>(nd.len), nb = (len + 15) >> 4;
  __syncwarp();
  if (lane == 0) {
#pragma unroll
    for (int c = 0; c < 8; ++c) sm.tot[c] = c < CM ? nd.cp[c < CM ? c : 0] : 0u;
  }
  uint32_t e[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) e[h] = lane + 32 * h < len ? rows_in[nd.base + lane + 32 * h] : 0u;
  __syncwarp();
  uint32_t B[4][2], Bw[4][2];
#pragma unroll
  for (int kb = 0; kb < 4; ++kb)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      int a[2], w[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const uint32_t ek = __shfl_sync(kFull, e[kb >> 1], 16 * (kb & 1) + 8 * h + 2 * t + u);
        w[u] = static_cast<int>(ent_w<0>(ek));
        a[u] = static_cast<int>(ent_y(ek)) == (CM == 2 ? 0 : g) ? w[u] : 0;
        if (CM == 2 && (g & 1)) a[u] = w[u];
      }
      B[kb][h] = pack_h2(a[0], a[1]);
      Bw[kb][h] = CM > 2 ? pack_h2(w[0], w[1]) : 0u;
    }
  const float n = static_cast<float>(nd.n);
  const float c0 = static_cast<float>(sm.tot[CM == 2 ? 0 : 2 * t]), c1 = static_cast<float>(sm.tot[2 * t + 1]);
  uint32_t seen = 0u;  // best float score so far, as its bits
  unsigned long long bs = 0ull;
  uint32_t bden = 1u, bkey = 0xFFFFFFFFu;
  for (int r0 = 0; r0 < d.mtry; r0 += 32) {
    const int nf = min(32, d.mtry - r0);
    const uint32_t f = lane < nf ? perm_apply(P, static_cast<uint32_t>(r0 + lane)) : 0u;
    if (r0 > 0) __syncwarp();
    sm.key[lane] = (d.tie_break == 1 ? static_cast<uint32_t>(r0 + lane) : f) << 8;
#pragma unroll
    for (int hb = 0; hb < 4; ++hb) {
      if (hb >= nb) break;
      uint32_t b[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int slot = 16 * hb + q;
        const uint32_t r = __shfl_sync(kFull, e[hb >> 1], slot & 31) >> 8;
        b[q] = 0u;
        if (lane < nf && slot < len) b[q] = row_bin(d, r, f);
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) sm.bins[lane * 33 + 8 * hb + q] = b[2 * q] | (b[2 * q + 1] << 16);
    }
    __syncwarp();
    uint32_t fbest = 0u;  // of feature `lane`
    for (int j = 0; j < nf; ++j) {
      const uint32_t* tw = sm.bins + j * 33;
      const uint16_t* th = reinterpret_cast<const uint16_t*>(tw);
      uint32_t A[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) A[i] = i < 2 * nb ? tw[4 * i + t] : 0u;
      // best float score of the feature (non-negative: their bits order as they do)
      float mine = 0.0f;
#pragma unroll
      for (int hb = 0; hb < 2; ++hb) {
        float p[4] = {0.0f, 0.0f, 0.0f, 0.0f}, nl[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          const int mb = 2 * hb + m;
          if (mb < nb) {
            float q0[2], q1[2], x[2];
            mid_block<CM>(A, dup_h(th[16 * mb + g]), dup_h(th[16 * mb + 8 + g]), B, Bw, nb, n, c0, c1, q0, q1, x);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
              p[2 * m + r] = fmaf(q0[r], q0[r], q1[r] * q1[r]);
              nl[2 * m + r] = x[r];
            }
          }
        }
        const float s = CM == 2 ? 2.0f * pick4(p[0], p[1], p[2], p[3], t) : quad_sum_own(p, t);
        const float l = pick4(nl[0], nl[1], nl[2], nl[3], t);
        if (32 * hb + 8 * t + g < len && s > 0.0f) mine = fmaxf(mine, __fdividef(s, l * (n - l)));
      }
      const uint32_t mx = __reduce_max_sync(kFull, __float_as_uint(mine));
      if (lane == j) fbest = mx;
    }
    // the features inside the window of the best score (usually one), exactly
    seen = max(seen, __reduce_max_sync(kFull, fbest));
    for (unsigned in = __ballot_sync(kFull, fbest != 0u && __uint_as_float(fbest) >= screen(__uint_as_float(seen))); in;
         in &= in - 1) {
      const int j = __ffs(in) - 1;
      const uint32_t* tw = sm.bins + j * 33;
      const uint16_t* th = reinterpret_cast<const uint16_t*>(tw);
      uint32_t A[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) A[i] = i < 2 * nb ? tw[4 * i + t] : 0u;
#pragma unroll
      for (int hb = 0; hb < 2; ++hb) {
        unsigned long long p[4] = {0ull, 0ull, 0ull, 0ull};
        float nL[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          const int mb = 2 * hb + m;
          if (mb < nb) {
            float q0[2], q1[2], x[2];
            mid_block<CM>(A, dup_h(th[16 * mb + g]), dup_h(th[16 * mb + 8 + g]), B, Bw, nb, n, c0, c1, q0, q1, x);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
              const long long y0 = static_cast<int32_t>(q0[r]), y1 = static_cast<int32_t>(q1[r]);
              p[2 * m + r] = static_cast<unsigned long long>(y0 * y0 + y1 * y1);
              nL[2 * m + r] = x[r];
            }
          }
        }
        const unsigned long long s = CM == 2 ? 2ull * pick4(p[0], p[1], p[2], p[3], t) : quad_sum_own(p, t);
        const uint32_t nl = f23_to_u32(pick4(nL[0], nL[1], nL[2], nL[3], t));
        if (32 * hb + 8 * t + g < len && s > 0ull) {
          const uint32_t den = nl * (nd.n - nl);
          const uint32_t key = sm.key[j] | th[32 * hb + 8 * t + g];
          const unsigned long long x = s * bden, y = bs * den;  // n <= 64 * 31: below 2^62
          if (x > y || (x == y && key < bkey)) {
            bs = s;
            bden = den;
            bkey = key;
          }
        }
      }
    }
  }
#pragma unroll
  for (int m = 1; m < 32; m <<= 1) {
    const unsigned long long os = __shfl_xor_sync(kFull, bs, m);
    const uint32_t od = __shfl_xor_sync(kFull, bden, m), ok = __shfl_xor_sync(kFull, bkey, m);
    const unsigned long long x = os * bden, y = bs * od;
    if (x > y || (x == y && ok < bkey)) {
      bs = os;
      bden = od;
      bkey = ok;
    }
  }
  const bool split = bs > 0ull;
  uint32_t feat = bkey >> 8;
  if (split && d.tie_break == 1) feat = perm_apply(P, feat);
  const uint32_t bin = bkey & 255u;
  bool gl[2], gr[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const bool v = split && lane + 32 * h < len;
    const uint32_t b = v ? row_bin(d, e[h] >> 8, feat) : 0u;
    gl[h] = v && b <= bin;
    gr[h] = v && !gl[h];
  }
  uint32_t cL[CM], nL = 0u;
#pragma unroll
  for (int c = 0; c < CM; ++c) {
    uint32_t x = 0u;
#pragma unroll
    for (int h = 0; h < 2; ++h) x += (gl[h] && ent_y(e[h]) == static_cast<uint32_t>(c)) ? ent_w<0>(e[h]) : 0u;
    cL[c] = __reduce_add_sync(kFull, x);
    nL += cL[c];
  }
  const unsigned l0 = __ballot_sync(kFull, gl[0]), l1 = __ballot_sync(kFull, gl[1]);
  const unsigned r0 = __ballot_sync(kFull, gr[0]), r1 = __ballot_sync(kFull, gr[1]);
  const uint32_t nl = __popc(l0) + __popc(l1);
  const unsigned lt = lanemask_lt();
  if (gl[0]) rows_out[nd.base + __popc(l0 & lt)] = e[0];
  if (gl[1]) rows_out[nd.base + __popc(l0) + __popc(l1 & lt)] = e[1];
  if (gr[0]) rows_out[nd.base + nl + __popc(r0 & lt)] = e[0];
  if (gr[1]) rows_out[nd.base + nl + __popc(r0) + __popc(r1 & lt)] = e[1];
  if (lane == 0) {
    commit_counts<CM>(d, k, split, feat, bin, nL, cL, bs, nd.n);
    if (split) d.nd_lrows[k] = nl;
    bytes += static_cast<unsigned long long>(nd.len) * (d.mtry + 4ull + (split ? 5ull : 0ull));
  }
}

// All four lists of the level in one launch: the warps take items dealt
// round-robin, the longest first (a mid node; one small, two tiny or four
// micro nodes).
template <int CM>
__global__ void __launch_bounds__(256, 4) k_few_rows(Dev d, int level) {
  union Tile {
    MidTile mid;
    FewTile few;
  };
  __shared__ Tile tiles[8];
  Tile& sm = tiles[threadIdx.x >> 5];
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t nmid = d.nmid[level], nsmall = d.nsmall[level], ntiny = d.ntiny[level], nmicro = d.nmicro[level];
  const uint32_t end32 = nmid + nsmall, end16 = end32 + (ntiny + 1u) / 2u, end8 = end16 + (nmicro + 3u) / 4u;
  unsigned long long bytes = 0;
  for (uint32_t it = gwarp; it < end8; it += nwarps) {
    if (it < nmid) {
      mid_rows<CM>(d, level, d.mid[it], sm.mid, bytes);
    } else if (it < end32) {
      few_rows<CM, 32>(d, level, d.small[it - nmid], sm.few, bytes);
    } else if (it < end16) {
      const uint32_t i = 2u * (it - end32) + (lane >> 4);
      few_rows<CM, 16>(d, level, i < ntiny ? d.small[d.small_cap - 1u - i] : kNoNode, sm.few, bytes);
    } else {
      const uint32_t i = 4u * (it - end16) + (lane >> 3);
      few_rows<CM, 8>(d, level, i < nmicro ? d.micro[i] : kNoNode, sm.few, bytes);
    }
  }
  if (bytes) atomicAdd(&d.counters[0], bytes);
}

template <int CM>
int launch(const Dev& d, int level, int grid, cudaStream_t st) {
  k_few_rows<CM><<<grid, 256, 0, st>>>(d, level);
  return 1;
}

}  // namespace

int launch_few_rows(const Dev& d, int level, int grid, cudaStream_t st) {
  switch (split_variant(d.kind, d.C)) {
    case 0: return launch<2>(d, level, grid, st);
    case 1: return launch<3>(d, level, grid, st);
    case 2: return launch<4>(d, level, grid, st);
    case 3: return launch<5>(d, level, grid, st);
    default: return launch<8>(d, level, grid, st);
  }
}

}  // namespace bgb
