// Block pairs of the symmetric feature map: the layout of the chunk states that the state kernel writes and the attend
// kernel reads.
//
// The 64 features of a row are cut into 8 runs of 8; the pair (g, h), h <= g, is the 64 products u[8g+i] u[8h+j].
// (q.k)^2 = sum over the pairs of w <Q_gh, K_gh> with w = 1 for g = h and 2 otherwise (the lift is symmetric); the
// blockwise map keeps the pairs inside a feature group.  36, 20 and 12 pairs for 1, 2 and 4 groups: multiples of four,
// so the feature axis falls into slices of 256 rows.  Rows of up to 32 entries have only the first four runs: 10 pairs of
// the full map, and two empty ones.  Inside a pair, row 8 j + i is the product (8g+i, 8h+j).
// Order of the pairs: the pairs 4s and 4s+2, and 4s+1 and 4s+3, share h wherever the counts allow it, because one warp of
// the state kernel builds those two and then fetches the factors of run h once.
#pragma once
#include <stdint.h>

namespace kata {

template <int G, int R = 8> struct PairTable {
  static constexpr int kRuns = R / G;                       // runs of 8 features per group
  static constexpr int kPairs = (G * kRuns * (kRuns + 1) / 2 + 3) / 4 * 4;
  static constexpr int kSlices = kPairs / 4;                // slices of 256 state rows
  static constexpr int kRows = kPairs * 64;
  uint8_t g[kPairs], h[kPairs];
  constexpr PairTable() : g(), h() {
    int couple = 0;                                         // two pairs with the same h
    int single_g[8] = {}, single_h[8] = {}, n_single = 0;
    auto put = [&](int ga, int ha, int gb, int hb) {
      const int p = 4 * (couple / 2) + (couple & 1);
      g[p] = (uint8_t)ga;
      h[p] = (uint8_t)ha;
      g[p + 2] = (uint8_t)gb;
      h[p + 2] = (uint8_t)hb;
      ++couple;
    };
    for (int grp = 0; grp < G; ++grp)
      for (int hh = 0; hh < kRuns; ++hh) {
        const int h0 = grp * kRuns + hh, end = (grp + 1) * kRuns;
        int gg = h0;
        for (; gg + 1 < end; gg += 2) put(gg, h0, gg + 1, h0);
        if (gg < end) {
          single_g[n_single] = gg;
          single_h[n_single] = h0;
          ++n_single;
        }
      }
    for (int i = 0; i + 1 < n_single; i += 2) put(single_g[i], single_h[i], single_g[i + 1], single_h[i + 1]);
    if (2 * couple < kPairs) put(R, R, R + 1 < 8 ? R + 1 : R, R);      // (narrow rows: two pairs of empty runs)
  }
};

}  // namespace kata
