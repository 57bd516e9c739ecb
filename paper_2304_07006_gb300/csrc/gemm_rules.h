// How the contractions are cut along k: host arithmetic alone, so that it can be tested without a GPU.
#pragma once
#include <stdint.h>

#include <algorithm>

namespace xtc {

// Most ranges of 64 values that the 64-bit sums of an FP64 contraction hold (gemm64_tc.cu).  Digits are at most 2^8 in
// magnitude, so a range adds at most (d + 1) 64 2^16 to diagonal d, the weights of the diagonals are 2^(27 - 9 (d mod 4)),
// and the larger sum, of diagonals 4..7, grows by less than 5.02 * 2^49 a range: 3,200 of them stay below 2^63.
// Rows of one value get there: 8,192 ranges a slice, as it was, let them wrap around.
constexpr int D64_MAX_RANGES = 3200;

// Slices of k of an FP64 contraction.  Few tiles: slices of at least 8 ranges so that the waves of CTAs are full, the
// count with the least (waves x ranges of a slice), a CTA's start and end counted as 6 ranges; with eight waves or
// more the last one matters little.
inline int gemm64_splits(int m_tiles, int n_tiles, int n_ranges, int n_sm) {
  const int64_t tiles = static_cast<int64_t>(m_tiles) * n_tiles;
  int best = 1;
  if (tiles < 8 * static_cast<int64_t>(n_sm)) {
    int64_t best_cost = -1;
    for (int s = 1; s <= std::max(1, std::min(n_ranges / 8, 2 * n_sm)); ++s) {
      const int64_t cost = (tiles * s + n_sm - 1) / n_sm * ((n_ranges + s - 1) / s + 6);
      if (best_cost < 0 || cost < best_cost) {
        best_cost = cost;
        best = s;
      }
    }
  }
  best = std::max(best, (n_ranges + D64_MAX_RANGES - 1) / D64_MAX_RANGES);
  const int per = (n_ranges + best - 1) / best;
  return (n_ranges + per - 1) / per;
}

}  // namespace xtc
