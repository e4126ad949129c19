// boruta_quantise: float features -> uint8 quantile bins, on the GPU.
//
// The method consumes binned features (the histogram forest of the fit), and
// the paper does not say how they are binned; the library's reading is
//   bin(x) = min(B - 1, floor(B * rank(x) / N)),  rank(x) = #{values < x},
// so equal values share a bin.  With r_k = ceil(k N / B) (k = 1..B-1) and T_k
// the r_k-th smallest value of the column, floor(B rank / N) >= k exactly
// when rank >= r_k, i.e. when T_k < x; hence bin(x) = #{k : T_k < x}.
//
// One block per column.
//   N <= 4096: the keys are sorted in shared memory; T_k is read off.
//   larger: three sweeps over the column.  A sample of 4096 keys sizes a
//   monotone map of the 32-bit order-preserving key to at most 16384 buckets
//   (the key's top 12 bits select a base and a shift of the other 20, finer
//   where the sample is dense; the map decides only the work, not the result).
//   Sweep 1 counts the buckets; their prefix sums give every target's bucket
//   and its rank inside it.  Sweep 2 collects the keys of the targets' buckets
//   (about 3% of them), into the output column, which is written last; a warp
//   per target selects by bisection on the key.  Sweep 3 writes the bins: the
//   number of targets in lower buckets, and a comparison with those of the
//   value's own bucket, if any.  Where too many keys fall into the targets'
//   buckets (heavily repeated values), a sweep finds the buckets that hold one
//   distinct key, whose targets are that key; if that does not thin them out
//   either, all targets are found by bisection over the column, from their
//   buckets' least and greatest keys.
// Bound by the three reads (13 bytes a value moved against 5) and the shared
// atomics.  Measured at N = 1e6, p = 500, B = 256: 3.0 ms (32 sweeps with
// a binary search per value before: 81.9 ms); N = 1000, p = 50, B = 64, the
// call with its host work:
// 58 us (272 us before).
#include <cstdint>

#include <cuda_runtime.h>

#include "boruta.h"

namespace {

constexpr int kQThreads = 512;
constexpr int kQTargets = 255;         // B - 1 at most
constexpr uint32_t kQSort = 4096;      // columns of at most this many values are sorted
constexpr uint32_t kQSample = 4096;    // keys that size the buckets
constexpr uint32_t kQBuckets = 16384;  // at most kQSample + 2 * 4096 are used

int qfail(int code, const char* msg);  // below

// order-preserving key of a float (-0 taken as +0); NaN reported by the caller
__device__ __forceinline__ uint32_t fkey(float x) {
  if (x == 0.0f) x = 0.0f;
  const uint32_t u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// number of sorted keys m[0..n) that are < v
__device__ __forceinline__ int count_below(const uint32_t* m, int n, uint32_t v) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (m[mid] < v)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo;
}

// r_k = ceil(k N / B) for target k - 1
__device__ __forceinline__ uint32_t target_rank(int k, uint32_t N, int B) {
  return static_cast<uint32_t>((static_cast<uint64_t>(k + 1) * N + static_cast<uint64_t>(B) - 1) /
                               static_cast<uint64_t>(B));
}

// f(i, key) for every value of the column (16-byte loads where the column is
// so aligned); returns true if this thread met a NaN (f is not called for it)
template <typename F>
__device__ __forceinline__ bool sweep(const float* col, uint32_t N, F&& f) {
  bool nan = false;
  auto one = [&](uint32_t i, float x) {
    if (x != x)
      nan = true;
    else
      f(i, fkey(x));
  };
  uint32_t done = 0;
  if ((reinterpret_cast<uintptr_t>(col) & 15u) == 0u) {
    const uint32_t quads = N / 4u;
    const float4* c4 = reinterpret_cast<const float4*>(col);
    uint32_t i = threadIdx.x;
    for (; i + blockDim.x < quads; i += 2u * blockDim.x) {
      const float4 a = c4[i], b = c4[i + blockDim.x];
      one(4u * i, a.x), one(4u * i + 1u, a.y), one(4u * i + 2u, a.z), one(4u * i + 3u, a.w);
      const uint32_t j = 4u * (i + blockDim.x);
      one(j, b.x), one(j + 1u, b.y), one(j + 2u, b.z), one(j + 3u, b.w);
    }
    if (i < quads) {
      const float4 a = c4[i];
      one(4u * i, a.x), one(4u * i + 1u, a.y), one(4u * i + 2u, a.z), one(4u * i + 3u, a.w);
    }
    done = quads * 4u;
  }
  for (uint32_t i = done + threadIdx.x; i < N; i += blockDim.x) one(i, col[i]);
  return nan;
}

// All targets by bisection on the key, one sweep per halving: every target
// keeps an interval [lo_k, hi_k], at first the least and the greatest key of
// its bucket; the intervals stay ordered in k (the targets are), so the
// midpoints are sorted and one sweep counts for every midpoint the values at
// or below it.  A bucket spans at most 20 bits of the key, and 20 - m where it
// holds many of the values (2^m at least its cell's sample count), so columns of
// close repeated values, which come here, take few sweeps (200 neighbouring
// floats, 1000 columns, B = 64: N = 20000 1.35 ms, 1e5 3.8 ms; from the whole key
// range, 33 sweeps, 3.9 and 12.0 ms).  Result in lo.
__device__ void bisect_column(const float* col, uint32_t N, int B, uint32_t* lo, uint32_t* hi, uint32_t* mid,
                              uint32_t* cnt) {
  const int nt = B - 1;
  for (int pass = 0; pass < 33; ++pass) {  // (an open interval halves: at most 32)
    int open = 0;
    for (int k = threadIdx.x; k < nt; k += blockDim.x) {
      open |= lo[k] < hi[k];
      mid[k] = static_cast<uint32_t>((static_cast<uint64_t>(lo[k]) + hi[k]) >> 1);
    }
    for (int k = threadIdx.x; k <= nt; k += blockDim.x) cnt[k] = 0u;
    if (!__syncthreads_or(open)) break;
    // cnt[c] = values whose key lies above exactly c midpoints
    sweep(col, N, [&](uint32_t, uint32_t key) { atomicAdd(&cnt[count_below(mid, nt, key)], 1u); });
    __syncthreads();
    if (threadIdx.x == 0) {
      // values <= mid_k = those above fewer than k + 1 midpoints (mid is sorted)
      uint32_t run = 0;
      for (int k = 0; k < nt; ++k) {
        run += cnt[k];
        if (lo[k] < hi[k]) {
          if (run >= target_rank(k, N, B))
            hi[k] = mid[k];
          else
            lo[k] = mid[k] + 1u;
        }
      }
      // keep the intervals ordered in k (T_k <= T_k+1)
      for (int k = 1; k < nt; ++k)
        if (lo[k] < lo[k - 1]) lo[k] = lo[k - 1];
      for (int k = nt - 2; k >= 0; --k)
        if (hi[k] > hi[k + 1]) hi[k] = hi[k + 1];
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kQThreads) k_quantise_sort(const float* X, int64_t ldx, uint32_t N, int64_t p, int B,
                                                             uint8_t* Xb, int64_t ldb, uint32_t* bad) {
  __shared__ uint32_t key[kQSort];
  __shared__ uint32_t T[kQTargets];
  const int nt = B - 1;
  uint32_t n2 = 2u;
  while (n2 < N) n2 <<= 1;
  for (int64_t j = blockIdx.x; j < p; j += gridDim.x) {
    const float* col = X + j * ldx;
    bool nan = false;
    for (uint32_t i = threadIdx.x; i < n2; i += blockDim.x) {
      const float x = i < N ? col[i] : 0.0f;
      nan |= x != x;
      key[i] = i < N ? fkey(x) : 0xFFFFFFFFu;
    }
    if (nan) atomicOr(bad, 1u);
    __syncthreads();
    for (uint32_t size = 2u; size <= n2; size <<= 1) {  // bitonic
      for (uint32_t d = size >> 1; d > 0u; d >>= 1) {
        for (uint32_t t = threadIdx.x; t < n2 / 2u; t += blockDim.x) {
          const uint32_t a = 2u * t - (t & (d - 1u)), b = a + d;
          const uint32_t x = key[a], y = key[b];
          if ((x > y) == ((a & size) == 0u)) {
            key[a] = y;
            key[b] = x;
          }
        }
        __syncthreads();
      }
    }
    for (int k = threadIdx.x; k < nt; k += blockDim.x) T[k] = key[target_rank(k, N, B) - 1u];
    __syncthreads();
    uint8_t* out = Xb + j * ldb;
    for (uint32_t i = threadIdx.x; i < N; i += blockDim.x) {
      const float x = col[i];
      out[i] = (x != x) ? 0u : static_cast<uint8_t>(count_below(T, nt, fkey(x)));
    }
    __syncthreads();
  }
}

struct QuantSmem {
  uint32_t cnt[kQBuckets];  // bucket counts; prefix sums; 1 + target of a collected bucket; first target, targets
  uint32_t tab[4096];       // sample counts; base | shift << 16
  uint32_t T[kQTargets], bk[kQTargets], rank[kQTargets];      // target's key, bucket, rank inside it
  uint32_t head[kQTargets], cur[kQTargets], start[kQTargets + 1];  // first target of the same bucket; its list
  uint32_t size[kQTargets], mn[kQTargets], mx[kQTargets];
  uint32_t warp[kQThreads / 32];
  uint32_t used, total;
};

// exclusive scan of v over the block
__device__ uint32_t quant_scan(uint32_t v, uint32_t* warp, uint32_t* total) {
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, d);
    if (lane >= static_cast<uint32_t>(d)) x += y;
  }
  if (lane == 31u) warp[w] = x;
  __syncthreads();
  uint32_t before = 0u, all = 0u;
  for (uint32_t i = 0; i < kQThreads / 32; ++i) {
    const uint32_t t = warp[i];
    before += i < w ? t : 0u;
    all += t;
  }
  __syncthreads();
  *total = all;
  return before + x - v;
}

// Lists of the targets' buckets in scratch: start and size per target (equal
// for targets of one bucket), offsets by the buckets with mn < mx only (or all
// of them, before mn and mx are known); total keys.
__device__ void place_lists(QuantSmem& sm, int nt, bool known) {
  if (threadIdx.x == 0) {
    uint32_t at = 0u;
    for (int k = 0; k < nt; ++k) {
      if (k > 0 && sm.bk[k] == sm.bk[k - 1]) {
        sm.head[k] = sm.head[k - 1];
        sm.start[k] = sm.start[k - 1];
        continue;
      }
      sm.head[k] = static_cast<uint32_t>(k);
      sm.start[k] = at;
      if (!known || sm.mn[k] < sm.mx[k]) at += sm.size[k];
    }
    sm.total = at;
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kQThreads, 2) k_quantise(const float* X, int64_t ldx, uint32_t N, int64_t p, int B,
                                                           uint8_t* Xb, int64_t ldb, uint32_t* bad) {
  extern __shared__ __align__(16) unsigned char raw[];
  QuantSmem& sm = *reinterpret_cast<QuantSmem*>(raw);
  const int nt = B - 1;
  const uint32_t tid = threadIdx.x;
  for (int64_t j = blockIdx.x; j < p; j += gridDim.x) {
    const float* col = X + j * ldx;
    uint8_t* out = Xb + j * ldb;
    // scratch for collected keys: the output column's whole words
    uint32_t* list = reinterpret_cast<uint32_t*>((reinterpret_cast<uintptr_t>(out) + 3u) & ~uintptr_t{3});
    const uint32_t room = (N - 3u) / 4u;
    // ---- the bucket map, from a sample
    for (uint32_t i = tid; i < 4096u; i += kQThreads) sm.tab[i] = 0u;
    for (uint32_t i = tid; i < kQBuckets; i += kQThreads) sm.cnt[i] = 0u;
    __syncthreads();
    for (uint32_t i = tid; i < kQSample; i += kQThreads) {
      const float x = col[static_cast<uint64_t>(i) * N / kQSample];
      if (x == x) atomicAdd(&sm.tab[fkey(x) >> 20], 1u);
    }
    __syncthreads();
    {
      // 2^m sub-buckets for a sample count c: 1 for c <= 1, else 2^m in [c, 2c)
      uint32_t m[4096 / kQThreads], sum = 0u, total;
#pragma unroll
      for (uint32_t q = 0; q < 4096 / kQThreads; ++q) {
        const uint32_t c = sm.tab[tid * (4096 / kQThreads) + q];
        m[q] = c <= 1u ? 0u : 32u - __clz(c - 1u);
        sum += 1u << m[q];
      }
      uint32_t base = quant_scan(sum, sm.warp, &total);  // total <= 4096 + 2 * 4096
#pragma unroll
      for (uint32_t q = 0; q < 4096 / kQThreads; ++q) {
        sm.tab[tid * (4096 / kQThreads) + q] = base | ((20u - m[q]) << 16);
        base += 1u << m[q];
      }
      if (tid == 0) sm.used = total;
    }
    __syncthreads();
    auto bucket = [&](uint32_t key) {
      const uint32_t e = sm.tab[key >> 20];
      return (e & 0xFFFFu) + ((key & 0xFFFFFu) >> (e >> 16));
    };
    // ---- sweep 1: counts, then prefix sums in place
    if (sweep(col, N, [&](uint32_t, uint32_t key) { atomicAdd(&sm.cnt[bucket(key)], 1u); })) atomicOr(bad, 1u);
    __syncthreads();
    {
      constexpr uint32_t kPer = kQBuckets / kQThreads;
      uint32_t sum = 0u, total;
      for (uint32_t q = 0; q < kPer; ++q) sum += sm.cnt[tid * kPer + ((q + tid) & (kPer - 1u))];
      uint32_t run = quant_scan(sum, sm.warp, &total);
      for (uint32_t q = 0; q < kPer; ++q) {
        const uint32_t c = sm.cnt[tid * kPer + q];
        sm.cnt[tid * kPer + q] = run;
        run += c;
      }
    }
    __syncthreads();
    const uint32_t used = sm.used;
    for (int k = tid; k < nt; k += kQThreads) {
      const uint32_t r = target_rank(k, N, B);
      uint32_t lo = 0u, hi = used;  // last bucket whose prefix is below r
      while (lo + 1u < hi) {
        const uint32_t m = (lo + hi) >> 1;
        if (sm.cnt[m] < r)
          lo = m;
        else
          hi = m;
      }
      sm.bk[k] = lo;
      sm.rank[k] = r - sm.cnt[lo];
      sm.size[k] = (lo + 1u < kQBuckets ? sm.cnt[lo + 1u] : N) - sm.cnt[lo];
      sm.mn[k] = 0xFFFFFFFFu;
      sm.mx[k] = 0u;
    }
    __syncthreads();
    place_lists(sm, nt, false);
    // ---- sweep 2: the keys of the targets' buckets
    for (uint32_t i = tid; i < kQBuckets; i += kQThreads) sm.cnt[i] = 0u;
    __syncthreads();
    for (int k = tid; k < nt; k += kQThreads) {
      if (sm.head[k] == static_cast<uint32_t>(k)) sm.cnt[sm.bk[k]] = static_cast<uint32_t>(k) + 1u;
      sm.cur[k] = sm.start[k];
    }
    __syncthreads();
    bool fit = sm.total <= room;
    if (!fit) {  // repeated values: which buckets hold one distinct key
      sweep(col, N, [&](uint32_t, uint32_t key) {
        const uint32_t h = sm.cnt[bucket(key)];
        if (h == 0u) return;
        if (key < *const_cast<volatile uint32_t*>(&sm.mn[h - 1u])) atomicMin(&sm.mn[h - 1u], key);
        if (key > *const_cast<volatile uint32_t*>(&sm.mx[h - 1u])) atomicMax(&sm.mx[h - 1u], key);
      });
      __syncthreads();
      place_lists(sm, nt, true);
      for (int k = tid; k < nt; k += kQThreads) {
        if (sm.head[k] == static_cast<uint32_t>(k) && sm.mn[k] == sm.mx[k]) sm.cnt[sm.bk[k]] = 0u;
        sm.cur[k] = sm.start[k];
      }
      __syncthreads();
      fit = sm.total <= room;
    }
    if (fit) {
      if (sm.total > 0u)
        sweep(col, N, [&](uint32_t, uint32_t key) {
          const uint32_t h = sm.cnt[bucket(key)];
          if (h) list[atomicAdd(&sm.cur[h - 1u], 1u)] = key;
        });
      __syncthreads();
      // a warp per target: the rank-th smallest of its list, by bisection
      for (int k = tid >> 5; k < nt; k += kQThreads / 32) {
        const uint32_t h = sm.head[k], lane = tid & 31u;
        if (sm.mn[h] == sm.mx[h]) {  // (mn > mx where no sweep looked)
          if (lane == 0u) sm.T[k] = sm.mn[h];
          continue;
        }
        const uint32_t n = sm.cur[h] - sm.start[h], r = sm.rank[k];
        const uint32_t* l = list + sm.start[h];
        uint32_t mn = 0xFFFFFFFFu, mx = 0u;
        for (uint32_t i = lane; i < n; i += 32u) {
          const uint32_t v = __ldcg(l + i);
          mn = min(mn, v);
          mx = max(mx, v);
        }
        uint32_t lo = __reduce_min_sync(0xFFFFFFFFu, mn), hi = __reduce_max_sync(0xFFFFFFFFu, mx);
        while (lo < hi) {
          const uint32_t m = lo + ((hi - lo) >> 1);
          uint32_t c = 0u;
          for (uint32_t i = lane; i < n; i += 32u) c += __ldcg(l + i) <= m;
          if (__reduce_add_sync(0xFFFFFFFFu, c) >= r)
            hi = m;
          else
            lo = m + 1u;
        }
        if (lane == 0u) sm.T[k] = lo;
      }
    } else {
      for (int k = tid; k < nt; k += kQThreads) {
        sm.T[k] = sm.mn[sm.head[k]];
        sm.size[k] = sm.mx[sm.head[k]];
      }
      __syncthreads();
      bisect_column(col, N, B, sm.T, sm.size, sm.cur, sm.start);
    }
    __syncthreads();
    // ---- sweep 3: bin = number of targets below the value
    for (uint32_t i = tid; i < kQBuckets; i += kQThreads) {
      const uint32_t first = static_cast<uint32_t>(count_below(sm.bk, nt, i));
      sm.cnt[i] = first | (static_cast<uint32_t>(count_below(sm.bk, nt, i + 1u)) - first) << 16;
    }
    __syncthreads();
    auto bin = [&](uint32_t key) {
      const uint32_t e = sm.cnt[bucket(key)], n = e >> 16;
      const uint32_t first = e & 0xFFFFu;
      return first + (n ? static_cast<uint32_t>(count_below(sm.T + first, static_cast<int>(n), key)) : 0u);
    };
    if (((reinterpret_cast<uintptr_t>(col) & 15u) | (reinterpret_cast<uintptr_t>(out) & 3u)) == 0u) {
      const float4* c4 = reinterpret_cast<const float4*>(col);
      for (uint32_t i = tid; i < N / 4u; i += kQThreads) {
        const float4 a = c4[i];
        reinterpret_cast<uint32_t*>(out)[i] = bin(fkey(a.x)) | bin(fkey(a.y)) << 8 | bin(fkey(a.z)) << 16 |
                                              bin(fkey(a.w)) << 24;
      }
      for (uint32_t i = (N & ~3u) + tid; i < N; i += kQThreads) out[i] = static_cast<uint8_t>(bin(fkey(col[i])));
    } else {
      for (uint32_t i = tid; i < N; i += kQThreads) out[i] = static_cast<uint8_t>(bin(fkey(col[i])));
    }
    __syncthreads();
  }
}

}  // namespace

int boruta_noalloc_fail(int code, const char* msg);  // api.cu: records the message

namespace {
int qfail(int code, const char* msg) { return boruta_noalloc_fail(code, msg); }
}  // namespace

extern "C" int boruta_quantise(const float* X, int64_t ldx, int64_t N, int64_t p, int n_bins, uint8_t* Xb,
                               int64_t ldb, void* stream) {
  if (N < 1 || N >= (1ll << 24) || p < 1 || ldx < N || ldb < N || !X || !Xb)
    return qfail(BORUTA_EINVAL, "boruta_quantise: bad sizes or pointers");
  if (n_bins < 2 || n_bins > 256) return qfail(BORUTA_EINVAL, "boruta_quantise: n_bins outside [2, 256]");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint32_t* bad = nullptr;
  if (cudaMallocAsync(reinterpret_cast<void**>(&bad), sizeof(uint32_t), st) != cudaSuccess) {
    cudaGetLastError();
    return qfail(BORUTA_ENOMEM, "boruta_quantise: scratch allocation failed");
  }
  uint32_t bad_h = 0;
  cudaMemsetAsync(bad, 0, sizeof(uint32_t), st);
  const int grid = static_cast<int>(p < 65535 ? p : 65535);
  cudaError_t e = cudaSuccess;
  if (N <= kQSort) {
    k_quantise_sort<<<grid, kQThreads, 0, st>>>(X, ldx, static_cast<uint32_t>(N), p, n_bins, Xb, ldb, bad);
  } else {
    e = cudaFuncSetAttribute(k_quantise, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(sizeof(QuantSmem)));
    if (e == cudaSuccess)
      k_quantise<<<grid, kQThreads, sizeof(QuantSmem), st>>>(X, ldx, static_cast<uint32_t>(N), p, n_bins, Xb, ldb, bad);
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(&bad_h, bad, sizeof(uint32_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFreeAsync(bad, st);
  if (e != cudaSuccess) return qfail(BORUTA_ECUDA, cudaGetErrorString(e));
  if (bad_h) return qfail(BORUTA_EINVAL, "boruta_quantise: NaN in the input");
  return 0;
}
