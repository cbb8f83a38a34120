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

}  // namespace oz
}  // namespace lrtei
