// Attention on CTA pairs, what needs no GPU: which kernel serves a call, which rows of the cache a block of keys is fetched from.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define PHYAI_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define PHYAI_HOST_DEVICE inline
#endif

namespace phyai {

// the first n columns of 64, a bit each (n below 0 as 0, above 64 as 64)
PHYAI_HOST_DEVICE uint64_t first_columns(int n) { return n <= 0 ? 0 : ~0ull >> (n < 64 ? 64 - n : 0); }

// Block `sb` of the (P + 63) / 64 blocks of a prefix of P keys: 64 rows of the cache from the prefix's row `row` on, of which those
// with a bit in `keys` are the block's keys.  A last block that is not full ends where the prefix ends, so that no row past it is
// read: its first rows are keys of the block before it, or, of a prefix of fewer than 64 keys, what lies before the prefix (row < 0).
struct PrefixBlock {
  int row;
  uint64_t keys;
};
PHYAI_HOST_DEVICE PrefixBlock prefix_block(int P, int sb) {
  const int left = P - sb * 64;
  return left >= 64 ? PrefixBlock{sb * 64, ~0ull} : PrefixBlock{P - 64, ~0ull << (64 - left)};
}

constexpr int MAX_PAIR_RANGES = 4;
constexpr int PAIR_TILE = 128;      // keys per tile of the kernels on pairs

// Key ranges per request: the number of 1 to `most` with the least waves x (fixed cost + tiles of a range).  resident[c]: clusters
// of 2 c CTAs (one range: pairs of the persistent kernel) that the device holds at a time, which decides the waves; <= 0: none, and
// c is no choice (where no c is, the result is 0: the call takes a kernel without clusters).  items: (request, four heads) pairs of
// the call, keys: most keys per request.
inline int choose_pair_ranges(const int (&resident)[MAX_PAIR_RANGES + 1], int items, int keys, int most) {
  int best_c = 0;
  double best = 0;
  for (int c = 1; c <= MAX_PAIR_RANGES && c <= most; ++c) {
    const int n = resident[c];
    if (n <= 0) continue;
    const double cost = (double)((items + n - 1) / n) * ((c > 1 ? 5.5 : 4.0) + (keys + c * PAIR_TILE - 1) / (c * PAIR_TILE));
    if (!best_c || cost < best) best = cost, best_c = c;
  }
  return best_c;
}

// Whether calls of caches of at most `keys` tokens take the kernels on pairs (`pairs` of them resident at a time) or the one-CTA kernel.
// From 256 tokens on always; with less there are at most four 64-key tiles, nothing to split, and the persistent pairs have to win by their
// longer tiles: from half as many items as pairs on, and, where the whole cache is one block of 64 keys, from seven eighths on.  Ten-step
// loops of 19 / 20 / 24 / 28 / 32 / 36 requests (two items each, 74 pairs), one-CTA kernel -> persistent pairs, ms: 60 tokens 10.68 -> 10.89,
// 10.75 -> 10.81, 11.91 -> 12.03, 13.16 -> 13.21, 14.50 -> 14.52, 15.75 -> 15.50; 120: 10.93 -> 11.00, 11.01 -> 10.95, 12.15 -> 12.30, 13.61 -> 13.58,
// 14.91 -> 14.76, 16.04 -> 15.91; 200: 11.32 -> 11.30, 11.40 -> 11.24, 12.66 -> 12.62, 14.08 -> 13.92, 15.48 -> 15.21.
inline bool pairs_pay(int keys, int items, int pairs) { return keys >= 256 || (keys > 64 ? 2 * items >= pairs : 8 * items >= 7 * pairs); }

}  // namespace phyai
