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

// Slices of a step (d) GEMM's K of n ranges, when its tiles leave pairs of SMs idle (10 of 76 pairs at N = 23).  Its sums are
// FP32 chains between FP64 flushes, column c of a thread's `cols` being flushed after the ranges r with r % flush = c: a
// slice that starts at a multiple of the flush interval and runs `cols` ranges past its end holds whole chains of every
// column, and whole periods of the cross-product accumulators (x_period ranges), so that every FP32 sum is the unsliced
// one.  The price is the overlap, `cols` ranges a slice.  The count with the least (waves of tiles on `slots` x (ranges of a
// slice + 30 for its start and end)), at most 16, if that saves 5 %; *flushes receives the flush intervals of a slice.
// Measured, step (d) unsliced -> sliced: N = 23, 3,957 points 154 -> 106 us; two GEMMs of N = 40, 20,000 points 1.45 -> 0.74
// ms; N = 65, 24,001 points (153 pairs of tiles, one more than two waves) 2.69 -> 2.33 ms.
inline int chain_slices(int n, int flush, int x_period, int cols, int tiles, int slots, int* flushes) {
  int best = 1;
  if (flush < cols || flush % cols || cols % x_period) return best;
  int64_t best_cost = static_cast<int64_t>((tiles + slots - 1) / slots) * (n + 30);
  for (int q = (n - 1) / flush; q >= 1; --q) {
    const int z = (n + q * flush - 1) / (q * flush);
    if (z > 16) break;
    if (n - (z - 1) * q * flush <= cols) continue;   // the last slice holds the end of every column's chains
    const int64_t cost =
        (static_cast<int64_t>(tiles) * z + slots - 1) / slots * (std::min(n, q * flush + cols) + 30);
    if (cost < best_cost - best_cost / 20) {
      best_cost = cost;
      best = z;
      *flushes = q;
    }
  }
  return best;
}

}  // namespace xtc
