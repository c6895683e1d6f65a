// Size rules of the tensor-core products, plain C++ (no CUDA types), so that they
// can be compiled and checked on any host.
#pragma once

#include <algorithm>
#include <cstdint>

namespace isdf {

// k values from which a tile's sum of a 5- or 6-digit product may not fit 64 bits:
// it is kept in units of 2^-21 with 7 (S - 4) more bits below, at most 2^35 units
// a k value.  2^21 with 5 digits, 2^14 with 6.
constexpr int64_t oz_wide_k(int S) { return int64_t(1) << (28 - 7 * (S - 4)); }

// Tile of a product: 128 rows of A, oz_tile_n(S) rows of B (S levels of them fill
// tensor memory: 5 x 48 twice, 6 x 64, 7 x 48, 8 x 48), steps of 32 k.
constexpr int kOzTileM = 128, kOzTileK = 32;
constexpr int oz_tile_n(int S) { return S == 6 ? 64 : 48; }

// Split-k partials of a product take at most this much scratch: more splits
// than that are neither timed nor chosen.
constexpr int64_t kOzPartialBytes = int64_t(2) << 30;
inline bool oz_splits_fit(int64_t splits, int64_t M, int64_t N) {
  return splits <= 1 || 8.0 * double(splits) * double(M) * double(N) <= double(kOzPartialBytes);
}

// Split-k factor of a product of more than 0.3 ms (shorter ones: 0, they are
// timed).  Waves of CTAs decide, which needs no measurement.  A wave takes its
// share of k at the measured tensor rate and one epilogue, the last one is three
// quarters idle on average, and the partial results are written and read once.
// (Timing the Coulomb matrix of the 2x2x2 diamond cell with every split took
// 0.7 s of its first pass.  1657 x 1657 x 903168, 7 digits, symmetric: 64.9 ms with
// one split, 56.5 with 3, 56.4 with 8, 55.6 with 16, the rule's choice, 54.6 with 32.)
inline int oz_rule_splits(int64_t M, int64_t N, int64_t nkt, int S, bool sym) {
  const int bn = oz_tile_n(S) * (S == 5 ? 2 : 1);
  const int64_t mt = (M + kOzTileM - 1) / kOzTileM, nt = (N + bn - 1) / bn;
  int64_t tiles = mt * nt;
  if (sym) {
    tiles = 0;
    for (int64_t i = 0; i < mt; ++i) tiles += std::min<int64_t>(nt, (i * kOzTileM + kOzTileM - 1) / bn + 1);
  }
  const double step = 2.0 * kOzTileM * bn * kOzTileK * (S * (S + 1) / 2) / (1.7e15 / 152.0);  // one k tile, seconds
  if (!(double(tiles) * double(nkt) * step / 152.0 > 3e-4)) return 0;
  int best = 1;
  double best_t = 1e30;
  for (int c : {1, 2, 4, 8, 16, 32, 64}) {
    if (c > nkt || !oz_splits_fit(c, M, N)) break;
    const double waves = std::max(1.0, double(tiles) * c / 152.0 + 0.75);
    const double t = waves * (double((nkt + c - 1) / c) * step + 4e-6) + (c > 1 ? 16.0 * c * double(M) * double(N) / 6e12 : 0.0);
    if (t < 0.99 * best_t) best_t = t, best = c;
  }
  return best;
}

}  // namespace isdf
