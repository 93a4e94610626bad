// How a launch of the MX GEMM is cut: tile width, pairs of CTAs, ring stages, weights that stay in shared memory.  Host arithmetic only,
// apart from the kernel so that a test can compile it by itself.  Internal: not part of the C ABI.
#pragma once

#include <algorithm>

#include "lq_internal.h"

namespace lqmx {

constexpr int MAX_STAGES = 8;
constexpr int STAGE_A_BYTES = LQ_BM * LQ_KSTAGE;   // 16 KB
constexpr int MAX_W = 224;                         // columns of the widest tile
constexpr int SF_BYTES = 512;                      // scale bytes of 128 rows x 4 K blocks
constexpr int STAGE_SF_BYTES = 3 * SF_BYTES;       // SFA, then SFB of up to 256 columns
constexpr int SC_FLOATS = LQ_BM + 2 * MAX_W;       // per tile: sT[128], sL2[W], bias[W]
constexpr int SMEM_BAR_BYTES = 320;
constexpr int FIXED_SMEM = 1024 /*alignment slack*/ + 2 * SC_FLOATS * 4 + SMEM_BAR_BYTES;
constexpr int MAX_SMEM = 227 * 1024;

// What a cut depends on, besides the device and the options.
struct MxShape {
  int M, N, b_wrap;     // b_wrap: K stages of the weights
  int planes;           // digit planes of the activations
  bool branch, acc;     // acc: an integer branch, with an accumulator of its own
  int weight_bits, out_bytes;
};
struct MxCut {
  int width_index, width, tiles_n;   // width: LQ_MX_WIDTHS[width_index]
  int pair, ctas, stages;            // stages: of the operand ring
  int resident, b_slots, smem;       // weights stay in b_slots places of shared memory; dynamic shared memory of the launch
};

// Ring depth that fits beside the fixed part.
inline int ring_stages(int bw) {      // bw: columns of B per CTA
  return std::min(MAX_STAGES, (MAX_SMEM - FIXED_SMEM) / (STAGE_A_BYTES + bw * LQ_KSTAGE + STAGE_SF_BYTES));
}
inline int ring_smem(int bw) {
  return FIXED_SMEM + ring_stages(bw) * (STAGE_A_BYTES + bw * LQ_KSTAGE + STAGE_SF_BYTES);
}
// The same with `slots` stages of B resident (negative: they do not fit).
inline int resident_smem(int bw, int slots, int stages) {
  return FIXED_SMEM + slots * (bw * LQ_KSTAGE + STAGE_SF_BYTES - SF_BYTES) + stages * (STAGE_A_BYTES + SF_BYTES);
}
inline int resident_stages(int bw, int slots) {
  return std::min(MAX_STAGES, (MAX_SMEM - resident_smem(bw, slots, 0)) / (STAGE_A_BYTES + SF_BYTES));
}

// Index (LQ_MX_WIDTHS) of the tile width for a launch.  Model, in clocks: a stage takes the longest of its MMAs (2 W, and 40 where
// one stage's meet the next's), its operands' way from the L2 (70 bytes per clock and SM) and its hand-shakes (350: what a
// stage of 64 columns takes); a tile the longer of its stages and the drain of the tile before; a launch the tiles of the CTA
// with the most, plus the last drain and the filling of the ring.  Measured, M = 8192, K x N = 4608 x 1152, W = 64 / 128 / 192 /
// 224: 58 / 37.9 / 35.3 / 38.0 us; 1152 x 3456: 52.5 / 34.2 / 30.3 / 30.0; 2240 x 2240: 61 / 39.6 / 36.3 / 35.0.
inline int pick_width(const MxShape& s, int ctas, int width_option, bool pair) {
  const int tiles_m = lq_ceil_div(s.M, LQ_BM), stages = s.b_wrap * s.planes + s.branch;
  int best = -1;
  double best_cost = 1e30;
  for (int i = 0; i < LQ_MX_NWIDTHS; ++i) {
    const int w = LQ_MX_WIDTHS[i];
    if (!lq_mx_width_used(w, s.acc)) continue;
    if (width_option > 0 && w != width_option) continue;
    const int c = pair ? 2 : 1, units = ctas / c;
    const long long tiles = (long long)lq_ceil_div(tiles_m, c) * lq_ceil_div(s.N, w);
    const double stage = std::max({2.0 * w + 40.0, 350.0, (STAGE_A_BYTES + w / c * LQ_KSTAGE / 8 * s.weight_bits) / 70.0});
    const double drain = 600.0 + 1200.0 * lq_ceil_div(w, 128);
    const double cost = (double)((tiles + units - 1) / units) * std::max(stages * stage, drain) + drain + 4.0 * stage;
    if (cost < best_cost) { best_cost = cost; best = i; }
  }
  return best;
}

// Whether a pair keeps the weights of its columns in shared memory and goes down them.  That saves their way from the L2 with every tile but the
// first, and costs stages of the ring and the order that keeps the pairs together.
//   A ring of at least half of a tile's stages is left for A.  (x: time with / without; MXFP4 and MXINT4 x 8, M = 2560 to 16384, 5 of 9 stages
//     0.94 - 1.00, 4 of 10 1.00 - 1.12)
//   Tiles of 160 columns or more - 128, where weights are six bits wide and no second accumulator is: else the weights are too little of what a
//     tile loads (128 columns: W8A8 0.93 - 1.08, MXFP4 0.93 - 1.06, MXINT4 with no or an fp16 branch 0.85 - 0.99)
//   A and Y together stay in three quarters of the L2, and no more than 32 columns of tiles: else the pairs, spread over all rows, write
//     back each other's lines (A and Y 110 to 500 MB: 0.88 - 1.2; Y of 70 MB, but 37 columns: 0.95 - 1.11)
//   Ten to 64 blocks of rows, two tiles for every pair, six stages of K, with an integer branch seven: within these it was timed.
// It was fitted to 2265 sizes of ten formats, drawn between K = 700 and 2000, N = 300 and 8192, M = 2305 and 16384: of these 979 are taken, 0.94 on
// average, the slowest 1.02; of 2013 others none is slower than by what two runs differ.  us without / with, M = 8192, 1152 x 3456: MXFP4
// 29.0 / 27.5, W8A8 32.4 / 31.0, MXINT4 x 8 50.0 / 47.7.
inline bool weights_stay(const MxShape& s, int pairs, int width, int tiles_n, int left) {
  const int blocks = lq_ceil_div(s.M, 2 * LQ_BM);
  const double bytes = (double)s.M * ((double)s.b_wrap * LQ_KSTAGE * s.planes + (double)s.N * s.out_bytes);
  return 2 * left >= s.b_wrap && width >= (s.acc || s.weight_bits == 4 ? 160 : 128) && bytes <= 96e6 && tiles_n <= 32 &&
         blocks >= 10 && blocks <= 64 && (long long)blocks * tiles_n >= 2 * pairs && s.b_wrap >= (s.acc ? 7 : 6);
}

// ctas: one per SM, or fewer.  False: no tile width is to be had.
inline bool plan_mx(const MxShape& s, int ctas, int width_option, bool pairs, MxCut& out) {
  const int tiles_m = lq_ceil_div(s.M, LQ_BM);
  // Pairs from 256 rows on; below, a pair's second CTA would have nothing to do.
  const bool pair = tiles_m > 1 && ctas > 1 && pairs;
  const int c = pair ? 2 : 1, wi = pick_width(s, ctas, width_option, pair);
  if (wi < 0) return false;
  out = {};
  out.width_index = wi; out.width = LQ_MX_WIDTHS[wi]; out.pair = pair;
  out.tiles_n = lq_ceil_div(s.N, out.width);
  const int bw = out.width / c;
  const long long tiles = (long long)lq_ceil_div(tiles_m, c) * out.tiles_n;
  out.ctas = c * (int)std::min<long long>(ctas / c, tiles);
  out.stages = ring_stages(bw);
  out.smem = ring_smem(bw);
  out.b_slots = s.b_wrap + s.branch;
  const int left = std::min(resident_stages(bw, out.b_slots), s.b_wrap);   // (the kernel's slots are free in time if the ring has no more stages than K)
  if (pair && weights_stay(s, out.ctas / 2, out.width, out.tiles_n, left)) {
    out.resident = 1;
    out.stages = left;
    out.smem = resident_smem(bw, out.b_slots, left);
  }
  return true;
}

}  // namespace lqmx
