// Which attention kernel on CTA pairs serves a call, from what the host knows of it (no device code).
#pragma once

namespace phyai {

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

}  // namespace phyai
