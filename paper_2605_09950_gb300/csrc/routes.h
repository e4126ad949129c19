// Which kernels take a call, as rules on its sizes (plain C++: no CUDA).  Each
// line lies where both sides were measured equal.
#pragma once
#include <cstdint>

namespace bgb {

// Alg. 3 by walks.cu (else k_permut).  Packing the trees and filling shared
// memory pays for large forests of deep trees only, and only while a re-walk's
// loss is cheap: its 3 rows a warp leave half the lanes of the loss idle, which
// the FP64 units (divisions and a logarithm per class) cannot hide.
// Importance stage, k_permut -> walks.cu, ms:
//   FP32 terms, 2 / 5 / 8 classes
//     N = 8192, 100 trees, depth 16        0.25 -> 0.38, 0.33 -> 0.43, 0.36 -> 0.47
//     N = 1e5, 10 trees, depth 16          0.35 -> 0.51, 0.44 -> 0.59, 0.45 -> 0.65
//     N = 20000, 100 trees, depth 20       0.86 -> 0.70, 1.10 -> 0.80, 1.22 -> 0.88
//     N = 50000, 100 trees, depth 12       0.88 -> 1.10, 1.25 -> 1.25, 1.44 -> 1.35
//     N = 50000, 100 trees, depth 16       1.40 -> 1.33, 1.97 -> 1.53, 2.27 -> 1.67
//     N = 1e5, 100 trees, depth 20         4.23 -> 2.99, 6.52 -> 3.42, 7.51 -> 3.80
//   FP64 terms: 2 to 25 times the time of k_permut everywhere measured
//     N = 1e5, 100 trees, depth 20         7.38 -> 14.2, 18.9 -> 35.5, 29.3 -> 56.4
//   regression (FP64 / FP32 terms)
//     N = 20000, 100 trees, depth 16       0.65 -> 0.73, 0.63 -> 0.64
//     N = 1e5, 100 trees, depth 16         3.57 -> 3.04, 3.46 -> 2.68
inline bool walks_pay(bool classification, bool fp32, int64_t N, int64_t trees, int depth) {
  if (N < 8192 || depth < 16) return false;
  const int64_t rows = N * trees;
  if (!classification) return rows >= 10000000;
  return fp32 && rows >= (depth < 20 ? 5000000 : 2000000);
}

}  // namespace bgb
