// Column counts of the augmented matrix (plain C++: no CUDA).
#pragma once
#include <algorithm>
#include <cstdint>

namespace bgb {

// Alg. 1: the live columns are copied until there are at least five shadows.
inline int64_t shadow_count(int64_t p_live) {
  int64_t n = p_live;
  if (n <= 0) return 0;
  while (n < 5) n *= 2;
  return n;
}

// Most columns (live and shadow) that any iteration over p columns can have.
// Below five live columns the count is not monotone (4 + 8 = 12 columns, but
// 5 + 5 = 10), and rejected columns lower the number of live ones.
inline int64_t max_augmented(int64_t p) {
  int64_t most = p + shadow_count(p);
  for (int64_t q = 1; q < std::min<int64_t>(p, 5); ++q) most = std::max(most, q + shadow_count(q));
  return most;
}

}  // namespace bgb
