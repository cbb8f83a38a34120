// oz_splits.h -- how the FP64 digit products (k_ozaki.cu) split K.  Host code without CUDA, so that its bounds are
// tested on the CPU.
#pragma once
#include <stdint.h>

#include <algorithm>

namespace lrtei {
namespace oz {

// The most 64-deep pieces of K whose sum of level `level` an int32 holds: a piece adds (level + 1) 64 products of two
// digits of magnitude at most 256.
constexpr int max_pieces(int level) { return (int)(0x7FFFFFFFLL / ((level + 1) * (64LL << 16))); }

// Splits of K (`pieces` of 64) that shorten the last wave of `items` tiles on 152 SMs, each at least 8 pieces and at
// most `most`; a split more costs about `store` pieces (its tile's store and its share of the reduction).
inline int pick_splits(int64_t items, int pieces, double store, int most) {
  int best = 1;
  double cost = 1e30;
  const int least = (pieces + most - 1) / most;
  for (int s = least; s <= std::max(16, least) && (s == least || pieces / s >= 8); ++s) {
    const double c = (double)((items * s + 151) / 152) * ((double)pieces / s + store) * (1.0 + 0.01 * s);
    if (c < cost) {
      cost = c;
      best = s;
    }
  }
  return best;
}

// Splits of a product of `items` tiles.  int32 sums: all eight levels in the skinny product, levels 0 to 5 in the wide
// ones.
inline int product_splits(int64_t items, int pieces, bool skinny) {
  return skinny ? pick_splits(items, pieces, 1.5, max_pieces(7)) : pick_splits(items, pieces, 6.0, max_pieces(5));
}

// Bytes of the split partials of rows [r0, r1) of B_u, the larger of those of G = F_u K and of B_u = G F_u^T, which
// follow one another.  size: columns of the nclass parity classes; cols: of all of them, padded; npair: columns of B_u.
inline double rows_partials(int64_t r0, int64_t r1, int64_t npair, const int* size, int nclass, int64_t cols) {
  const int64_t nr = r1 - r0, tiles_m = (nr + r0 % 128 + 127) / 128, tiles_n = (npair + 127) / 128;
  const bool symmetric = r0 == 0 && r1 == npair;
  int64_t g_items = 0;
  int pieces = 1;
  for (int c = 0; c < nclass; ++c) {
    const int k = (size[c] + 63) / 64 * 64;
    g_items += tiles_m * ((k + 127) / 128);
    pieces = std::max(pieces, k / 64);
  }
  const int sg = product_splits(g_items, pieces, false);
  const int sb = product_splits(symmetric ? tiles_n * (tiles_n + 1) / 2 : tiles_m * tiles_n, (int)(cols / 64), false);
  return std::max(sg > 1 ? 8.0 * sg * nr * cols : 0.0, sb > 1 ? 8.0 * sb * nr * npair : 0.0);
}

}  // namespace oz
}  // namespace lrtei
