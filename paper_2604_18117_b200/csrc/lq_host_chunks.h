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
// Where Y is one and a half to five times X, and both together some tens of megabytes, the way out sets the time and waits for a long
// chunk's way in: eight alike are the better cut there.  us, eight alike / four or five chunks: X and Y of 8.4 and 16.8 MB 402 / 430, 5.9
// and 14.8 354 / 371, 14.6 and 21.3 588 / 609, 3.1 and 10.6 (another host) 305 / 344; beside it: Y = X, 9.4 MB 353 / 326, 16.8 and 21.0 MB
// 555 / 500, 8.4 and 33.6 708 / 698, 9.4 and 37.7 794 / 777.  (3168 drawn sizes on two hosts, of 2048 rows and more: with four or five chunks
// everywhere 297 take more than 3 % longer than with eight, so 95; the hosts differ, and between the bounds 61 give up 2 % or more that
// four or five chunks won there.)
inline int host_chunks(int M, size_t x_bytes, size_t y_bytes, int (&end)[LQ_HOST_CHUNKS]) {
  static_assert(LQ_HOST_CHUNKS >= 5, "");
  const double x = (double)x_bytes, y = (double)y_bytes;
  const bool way_out = y >= 1.4 * x && y <= 5 * x && x + y >= 13e6 && x + y <= (y < 2.1 * x ? 40e6 : 30e6);
  const bool tapered = M >= 2048 && !way_out, few = x + y < 32 * 1048576.0;
  const int n = tapered ? (few ? 4 : 5) : std::min(LQ_HOST_CHUNKS, std::max(1, M / (2 * LQ_BM)));
  // sizes of the inner chunks and of all, the outer ones' being 1
  const int inner = few ? 3 : 2, parts = 2 + (n - 2) * inner, alike = lq_round_up(lq_ceil_div(M, n), LQ_BM);
  int c = 0;
  for (int i = 0; i < n && (c == 0 || end[c - 1] < M); ++i) {
    const int64_t at = i + 1 == n ? parts : 1 + i * inner;
    end[c++] = std::min(M, tapered ? lq_round_up((int)(M * at / parts), LQ_BM) : (i + 1) * alike);
  }
  return c;
}
