// Which kernels take a call, as rules on its sizes (plain C++: no CUDA).  Each
// line lies where both sides were measured equal.
#pragma once
#include <cstdint>

namespace bgb {

// Alg. 3 by walks.cu (else k_permut).  Packing the trees and filling shared
// memory pays for large forests of deep trees, and only while a re-walk's loss
// is cheap: its 3 rows a warp leave half the lanes of the loss idle, which the
// FP64 units (divisions and a logarithm per class) cannot hide.  The rows of all
// trees that it takes grow by half with every level below 17.
// Importance stage, k_permut -> walks.cu, ms:
//   FP32 terms, 2 / 5 / 8 classes
//     N = 8192, 100 trees, depth 16        0.25 -> 0.38, 0.33 -> 0.43, 0.36 -> 0.47
//     N = 1e5, 10 trees, depth 16          0.35 -> 0.51, 0.44 -> 0.59, 0.45 -> 0.65
//     N = 20000, 100 trees, depth 20       0.86 -> 0.70, 1.10 -> 0.80, 1.22 -> 0.88
//     N = 50000, 100 trees, depth 12       0.88 -> 1.10, 1.25 -> 1.25, 1.44 -> 1.35
//     N = 50000, 100 trees, depth 16       1.40 -> 1.33, 1.97 -> 1.53, 2.27 -> 1.67
//     N = 1e5, 100 trees, depth 20         4.23 -> 2.99, 6.52 -> 3.42, 7.51 -> 3.80
//   times as fast at N x trees (1e6), over 150 random problems: depth 13 0.96 at
//   4.0, 1.04 at 6.1, 1.2 at 12 to 27; depth 15 0.9 at 1.5, 1.04 at 4.4, 1.3 at 10 to
//   31; depth 17 0.95 at 2.7, 1.2 at 4, 1.7 at 10 to 26; depth 19 and 20 0.9 at 1.1, 1.3
//   at 2 to 4, 1.7 at 16 to 53; two classes 0.7 to 1.0 at 1.4 to 20 below depth 15
//   FP64 terms: 2 to 25 times the time of k_permut everywhere measured
//     N = 1e5, 100 trees, depth 20         7.38 -> 14.2, 18.9 -> 35.5, 29.3 -> 56.4
//   regression (FP64 / FP32 terms)
//     N = 20000, 100 trees, depth 16       0.65 -> 0.73, 0.63 -> 0.64
//     N = 1e5, 100 trees, depth 16         3.57 -> 3.04, 3.46 -> 2.68
// classes: 0 for regression
inline bool walks_pay(int classes, bool fp32, int64_t N, int64_t trees, int depth) {
  if (N < 8192 || depth < 12) return false;
  const int64_t rows = N * trees;
  if (classes == 0) return depth >= 16 && rows >= 10000000;
  if (!fp32) return false;
  int64_t need = depth >= 19 ? 1500000 : 2000000;
  for (int l = 17; l > depth; --l) need += need / 2;
  if (classes <= 2 && depth < 15) need *= 2;
  return rows >= need;
}

// Classification nodes above 64 rows in problems of 65,536 rows and more, whose
// nodes of weight 65,536 and up are counted by column gathers in feature bands
// in any case.  column.cu and record.cu then run before the band kernels of
// every level, and the longest node of each is waited for in turn; with few
// (node, column) items, which leave the GPU idle, the bands alone take all the
// nodes of a level together in less time.  Both lines by the columns a node
// samples, the trees and the depth (few rows a node, and many nodes, lie deep);
// below 65,536 rows (and a little above, where few levels hold both) there is no
// second wait, and the rules say yes.
// Split stage, column.cu against the bands alone, times as fast (2, 5 classes,
// depth 12):
//   N = 60000, 30 trees, 10 / 31 columns      2.20, 1.49 / 1.95, 1.61
//   N = 80000, 60 trees, 4 / 10 / 31          1.04, 0.91 / 1.11, 0.93 / 1.20, 1.17
//   N = 1e5, 1 tree, 4 / 63                   1.12, 1.14 / 1.50, 1.48
//   N = 1e5, 30 trees, 10 / 31 / 63           0.97, 0.91 / 0.95, 0.89 / 1.24, 1.10
//   N = 1e5, 200 trees, 4 / 20 / 44           0.85, 0.80 / 1.03, 1.05 / 1.37, 1.22
//   N = 130000, 60 trees, 10 / 31 / 63        0.82, 0.78 / 0.92, 0.86 / 1.22, 1.13
// Over 500 problems of 2 to 8 classes and 32 to 256 bins: from depth 13 on columns
// win with a tenth of the items (column, tree) that they need at depth 9 to 12, up
// to depth 8 only where there are many (N = 75,000 to 120,000, 3000 to 5500 items
// 1.08 to 1.28 times as fast, 400 to 2000 0.81 to 0.99); six and more classes, whose
// histograms hold three and four words a bin, need as many as depth 9 to 12.
inline bool columns_pay(int64_t N, int64_t trees, int64_t mtry, int depth, int classes) {
  if (N < 66000 || trees <= 3) return true;
  const int64_t items = trees * mtry;
  if (depth <= 8) return items >= 2300 && 16 * items >= N - 65536;
  if (N < 82000 || (mtry >= 44 && N < 110000)) return true;
  return (classes >= 6 ? 16 : (depth > 12 ? 200 : 28)) * items >= N - 65536;
}

// record.cu (where column.cu does not take the problem) against the bands alone,
// times as fast, 5 classes:
//   N = 2e5, depth 12, 100 trees, 4 / 10 / 31 / 63 columns  0.87 / 0.89 / 1.07 / 1.24
//   N = 2e5, depth 12, 10 trees                             0.87 / 0.86 / 0.92 / 1.07
//   N = 2e5, depth 20, 100 trees                            0.78 / 0.89 / 1.18 / 1.35
//   N = 1e6, depth 20, 300 trees, 10 / 31 columns           0.87 / 1.15
//   N = 2e5, 2 classes, 14 to 26 columns, 266 to 362 trees, depth 11 to 18  1.02 to 1.12
//   N = 2e5, 6 classes, 33 columns, 132 trees, depth 10     0.88
inline bool records_pay(int64_t N, int64_t trees, int64_t mtry, int depth, int classes) {
  if (N < 65536) return true;
  if (depth <= 9) return false;
  const int64_t items = trees * mtry;
  if (mtry >= 60 || (classes <= 2 && mtry >= 14 && depth >= 11 && items >= 2500)) return true;
  return mtry >= 22 && items >= (depth <= 13 ? 2300 : 900);
}

// Regression over more than 4 bins.  Nodes of 33..1024 rows by regress.cu's
// blocks (else the column gathers): a block reads 32 columns of its node at a
// time and deals them to its warps, so few sampled columns leave it idle; up to
// 1024 rows the gathers' launches go too.  Split stage, k_reg_record against the
// gathers, times as fast (depth 12, 1 / 10 / 100 trees):
//   N = 1000, 4 / 33 columns      1.99 / 1.64 / 1.46    3.17 / 2.47 / 1.84
//   N = 2000, 10 / 16 / 24        1.21 / 1.01 / 0.86    1.47 / 1.14 / 1.01    1.67 / 1.19 / 1.08
//   N = 5000, 33 / 48 / 64        1.33 / 1.04 / 0.79    1.46 / 1.17 / 0.90    1.83 / 1.36 / 0.99
//   N = 20000, 33 / 64 / 133      1.13 / 0.88 / 0.83    1.20 / 1.08 / 1.08    1.48 / 1.27 / 1.29
//   N = 1e5, 33 / 64 / 133        0.92 / 0.89 / 0.91    0.99 / 1.05 / 1.05    1.10 / 1.22 / 1.18
inline bool reg_record_pays(int64_t N, int64_t trees, int64_t mtry) {
  if (N <= 1024 || mtry >= 64 || N <= 128 * mtry) return true;
  return (mtry >= 24 && N * trees <= 50000) || (mtry >= 48 && N * trees <= 200000);
}

// Nodes of at most 32 rows by its warps (else k_split_small): their products take
// 32 columns at a time.  Split stage, times as fast (depth 16, 100 trees, 4 / 16 /
// 24 / 48 columns): N = 2000 0.99 / 1.11 / 1.20 / 1.50, N = 5000 0.87 / 0.97 / 1.09 /
// 1.32, N = 20000 0.85 / 0.93 / 1.00 / 1.14, N = 1e5 0.94 / 0.97 / 1.01 / 1.05; 10
// trees 0.99 to 1.05 below 24 columns, more above.
inline bool reg_rows_pays(int64_t N, int64_t mtry) { return N <= 2048 || mtry >= 24; }

// Regression over at most 3 bins by threebin.cu (else by row, and the column
// gathers' register counts).  Its blocks read records whole, 1024 columns a
// round, and score the sampled ones: worth it while a node samples many of them,
// or while there is so little to do that the launches count.  Split stage, times
// as fast (depth 10):
//   N = 1000, 100 trees, 6 / 24 / 48 columns    1.16 / 2.00 / 3.09 (p = 24)
//   N = 2000, 100 trees, 16 / 40                1.13 / 1.64 (p = 24, 60; iteration)
//   N = 2000, 300 trees, 16 / 40                0.73 / 1.19 (p = 24, 60; iteration)
//   N = 5000, 10 trees, 6 / 24 / 48             1.17 / 1.81 / 2.59 (p = 24)
//   N = 5000, 100 trees, 6 / 24 / 48            0.49 / 0.86 / 1.30 (p = 24)
//   N = 5000, 100 trees, 50 / 100 / 400         1.19 / 2.06 / 5.82 (p = 200)
//   N = 16000, 100 trees, 13 / 50 / 100         0.45 / 0.99 / 1.82 (p = 50)
//   N = 40000, 10 trees, 13 / 50 / 100          0.61 / 0.84 / 1.33 (p = 50)
//   N = 30000, 100 trees, 40 / 66               0.85 / 1.22 (p = 60, 100; iteration)
//   N = 40000, 1 tree, 500 / 1000 of 4000       0.66 / 1.21
// From 16,384 rows on the largest nodes go to the gathers in any case.  Shallow
// trees are few large nodes, a block each, whose time the level waits for, and do
// not reach the small ones (iteration, times as fast, depth 2 / 4 / 6 / 8):
//   N = 4000, 10 trees, 133 / 1333 columns     1.12 / 1.69 / 2.65 / 3.56    0.71 / 1.02 / 4.39 / 7.70
//   N = 8000, 10 trees, 66 / 400               0.78 / 0.97 / 1.31 / 1.65    0.74 / 0.93 / 1.83 / 3.18
//   N = 8000, 100 trees, 66 / 400              1.08 / 1.09 / 1.36 / 1.47    1.51 / 1.70 / 2.87 / 3.73
//   N = 16000, 10 trees, 133 / 400             0.63 / 0.73 / 1.04 / 1.48    0.53 / 0.64 / 1.05 / 1.96
//   N = 16000, 100 trees, 66 / 133             0.89 / 0.84 / 1.04 / 1.23    1.22 / 1.27 / 1.63 / 2.08
//   N = 70000, depth 4 / 6 / 8 / 10, 30 trees, 66 / 133  0.76 / 0.76 / 0.86 / 1.01, 0.88 / 0.96 / 1.15 / 1.50
//   N = 200000, the same                       0.89 / 0.82 / 0.84 / 0.95, 0.94 / 0.92 / 1.03 / 1.22
inline bool three_bins_pay(int64_t N, int64_t trees, int64_t mtry, int64_t columns, int depth) {
  if (8 * mtry < columns || (N >= 16384 && 4 * mtry < columns)) return false;
  const int64_t items = trees * mtry;
  if (depth <= 4) {
    if (N > 8192) {
      if (items < 12000 || trees < (depth <= 2 ? 100 : 30)) return false;
    } else if (N > 4096) {
      if (trees < (depth <= 2 ? 100 : 30)) return false;
    } else if (depth <= 2 && N > 1024 && trees < 30) {
      return false;
    }
  } else if (depth <= 7) {
    const bool many = items >= 4000 && trees >= 30 && 15 * items >= N && (N < 16384 || mtry >= 128);
    if (N > 8192 && !many && !(N < 16384 && trees >= 10 && mtry >= 128)) return false;
  } else if (N >= 16384 && (depth < 10 ? 30 : (depth < 13 ? 100 : 200)) * items < N) {
    return false;
  }
  if (mtry >= 64 || (mtry >= 40 && N <= 5000) || (mtry >= 24 && N <= 1024)) return true;
  return N <= 5000 && N * trees <= (mtry >= 16 ? 200000 : 100000);
}

// Whether a level's lists are written by a kernel of their own (k_classify)
// instead of with its nodes: regression levels of many nodes (at most `nodes`),
// and all of them where k_split_small takes the small ones (not reg_rows).
// There the kernel between k_children and the fork decides which stream's
// kernels reach the SMs first, the larger nodes' or the small ones' (an empty
// kernel in its place measures the same, lists in any order too), and with the
// larger ones first the level ends sooner: N = 10000, p = 50, all columns, 100
// trees, depth 16 17.0 -> 16.3 ms an iteration, N = 5000, 200 columns, 10 trees,
// depth 16 by column gathers and k_split_small 17.4 -> 15.6.  Elsewhere the launch costs more than
// the order gives (classification 1 to 4%, genotypes 2%, small levels 3 us).
inline bool lists_apart(bool regression, bool three_bins, bool reg_rows, uint64_t nodes) {
  return regression && !three_bins && (nodes > 16384 || !reg_rows);
}

}  // namespace bgb
