// When a sort counts the entries before each instead of taking digit passes.
#pragma once

#include <stdint.h>

namespace lgc {

constexpr int64_t kRankWork = 50 << 20;  // comparisons per digit pass spared

// n^2 comparisons against `digits` passes of 8 bits.  A digit pass over so few
// entries is a launch and a chain of look-backs, 8.5 us, and eight with their
// histogram 75; the n^2 comparisons of 64-bit keys and the copy back take 18 us
// at 8,274 entries and 56 at 19,117.  (n * n itself leaves 64 bits past 3.04e9.)
constexpr bool rank_sort_takes(int64_t n, int digits) {
  return n <= 1 || n <= digits * kRankWork / n;
}

}  // namespace lgc
