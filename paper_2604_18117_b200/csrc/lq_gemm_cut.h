// How many CTAs share a tile of the SINT4 GEMM.  Host arithmetic only, apart from the kernel so that a test can compile it by itself.
// Internal: not part of the C ABI.
#pragma once

#include <algorithm>

#include "lq_internal.h"

// CTAs per tile of a launch of few tiles (1, 2, 4 or 8).  A tile's stages are one serial chain, so while SMs are idle they may as well share
// it; a cluster's launch and the exchange cost the rest (us, alone and shared: M = 1, K x N = 1152 x 1152: 7.0 and 4.8 by
// eight; M = 120, 8192 x 1152: 30.8 and 9.8 by eight; M = 256, 4608 x 1152: 18.9 and 10.3 by four).  The hardware places a cluster's CTAs
// next to each other, so fewer fit than there are SMs; a second round of them would cost more than it gives.  Prices, us: a stage 0.44, the
// exchange 1.62 and, in proportion to the rows of a full tile, FULL_US by two, four, eight CTAs.  Eight cost 0.6 more than four (over 1 to
// 15 tiles 0.5 to 1.2, but from 13 stages on they are the faster): at 0.32 more, as four cost than two for as many CTAs, tiles of 8 to 12
// stages went to eight (us by four / by eight, M x K x N = 384 x 872 x 640 6.42 / 7.38, 512 x 872 x 264 6.27 / 6.98, 384 x 1152 x 640
// 6.50 / 7.39, 128 x 864 x 1152 6.21 / 6.71; 128 x 1536 x 640 6.42 / 6.19).  Nor do sums of eight parts round less there (relative error,
// fp32 output, 384 x 1152 x 640: 5.6e-8 by four, 5.9e-8 by eight).
// A stage of a chain is charged 0.08 us beyond its time, because the sum's error grows with the chain: rows of seven to ten stages are so
// shared where alone would be as fast or faster (M = 120, 1152 x 4608: 7.57 by two, 7.50 alone; M = 256: 8.40 and 6.84, the largest
// difference of 504 sizes; 256 x 768 x 1152: 6.40 by four, 5.50 alone), with a relative error of 6.0e-8 instead of 7.4e-8 (M = 128, fp32
// output).  Tiles of six stages are shared up to 60 rows (640 x 1152, by four and alone: M = 1 4.14 and 4.71, M = 60 4.84 and 4.92).
// clusters: of 2, 4 and 8 CTAs, that the device holds at once; asked: option "gemm_split".
inline int pick_split(int M, long long units, int stages, int ctas, const int (&clusters)[3], int asked) {
  constexpr double STAGE_US = 0.44, CHAIN_US = 0.08, FULL_US[3] = {0.76, 0.92, 1.52};
  int best = 1;
  double best_cost = (STAGE_US + CHAIN_US) * stages;
  for (int i = 0, split = 2; i < 3; ++i, split *= 2) {
    if (split > ctas || split > stages || units > std::min(clusters[i], ctas / split)) break;
    if (asked > 0 && split != asked) continue;
    const double exchange = 1.62 + FULL_US[i] * std::min(M, LQ_BM) / LQ_BM;
    const double cost = asked > 0 ? 0 : (STAGE_US + CHAIN_US) * lq_ceil_div(stages, split) + exchange;
    if (cost < best_cost) { best_cost = cost; best = split; }
  }
  return best;
}
