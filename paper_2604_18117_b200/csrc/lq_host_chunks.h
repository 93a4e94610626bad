// Row chunks of a call from host memory.  Host arithmetic only, apart from the call so that a test can compile it by itself.  Internal:
// not part of the C ABI.
#pragma once

#include <algorithm>

#include "lq_internal.h"

// Row chunks of a call from host memory (end[c]: the row behind chunk c, a multiple of the row tile or M): their number.  The first
// chunk's way in and the last one's way out are paid in full, so those are shorter than the others; but while the other direction is
// busy, a copy's start costs 10 to 15 us of its own direction, so there are few.  Below 2048 rows: chunks of at least 256, all alike.
// us, eight chunks alike / as here: M x K x N = 4096 x 1152 x 1152 368 / 329, 8192 x 1152 x 4608 1547 / 1510, 8192 x 4608 x 1152
// 1509 / 1498; 1536 x 1152 x 1152 with six alike 202, with four of these sizes 212.
inline int host_chunks(int M, size_t bytes, int (&end)[LQ_HOST_CHUNKS]) {
  static_assert(LQ_HOST_CHUNKS >= 5, "");
  const bool tapered = M >= 2048, few = bytes < (size_t)32 << 20;
  const int n = tapered ? (few ? 4 : 5) : std::min(LQ_HOST_CHUNKS, std::max(1, M / (2 * LQ_BM)));
  const int inner = few ? 3 : 2, parts = 2 + (n - 2) * inner, alike = lq_round_up(lq_ceil_div(M, n), LQ_BM);   // sizes of the inner chunks and of all, the outer ones' being 1
  int c = 0;
  for (int i = 0; i < n && (c == 0 || end[c - 1] < M); ++i) {
    const int64_t at = i + 1 == n ? parts : 1 + i * inner;
    end[c++] = std::min(M, tapered ? lq_round_up((int)(M * at / parts), LQ_BM) : (i + 1) * alike);
  }
  return c;
}
