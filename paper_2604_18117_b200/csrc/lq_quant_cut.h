// How a launch of the quantizer kernel is cut: rows per tile, stages of K per chunk, teams of warps, ring slots, shared memory.
// Host arithmetic only (and the shared-memory map, which the kernel uses too), apart from the kernel so that a test can compile it
// by itself.  Internal: not part of the C ABI.
#pragma once

#include <algorithm>

#include "lq_internal.h"

namespace lqcut {

constexpr int QWARPS = 15;             // quantizer warps (at most; teams of RG * SX): 20 warps are the most that leave 96 registers each
constexpr int MAX_SLOTS = 4;           // chunk slots of the branch's operands
constexpr int SETTLE_CHAINS = 9;       // MXFP: chains of the sum that near ties are settled on
constexpr int SETTLE_BYTES = SETTLE_CHAINS * 16 * 32 * 4;   // their partial sums for sixteen rows, where the rings were
constexpr int MAX_XSLOTS = 12;         // chunk slots of X
enum { BR_NONE = 0, BR_INT = 1, BR_F16 = 2, BR_MXFP = 3, BR_MXINT = 4 };

struct QuantCut {
  int groups, stages;   // RG row groups of 8 per tile, SX stages of K per chunk
  int teams;            // teams of RG * SX quantizer warps: they take the chunks in turn
  int ntiles, nchunks;  // tiles of the launch, chunks of a tile
  int slots, xslots;    // chunk slots of the branch's operands and of X
  int refetch;          // integer branch: the X ring is smaller than a tile, which is streamed twice
  int smem;             // dynamic shared memory of the launch
  int drop_x;           // X is the first to leave the L2 (x_leaves_first)
};

// Shared memory, from a 1024-byte aligned base; the same arithmetic on the host (size) and in the kernel.  First the X ring,
// then the slots: a slot holds a chunk's operand slabs (128 bytes of K wide, a_ps and b_ps of them per stage) and scale bytes.
struct QuantSmem {
  int xslot, a_unit, a_ps, b_unit, b_ps;
  int off_b, off_sfa, off_sfb, slot;            // within a slot
  int off_slots, off_l1, off_max, off_sb, off_bar, total;
};
__host__ __device__ inline QuantSmem quant_smem(int br, int tr, int st, int rn, int bplanes, int slots, int xslots) {
  QuantSmem s{};
  const bool mx = br == BR_MXFP || br == BR_MXINT;
  s.xslot = tr * 256 * st;                      // st: stages of K per chunk
  s.a_unit = tr * 128; s.b_unit = rn * bplanes * 128;
  s.a_ps = br == BR_NONE ? 0 : (br == BR_F16 || br == BR_MXINT) ? 2 : 1;
  s.b_ps = br == BR_NONE ? 0 : br == BR_F16 ? 2 : 1;
  s.off_b = st * s.a_ps * s.a_unit;
  s.off_sfa = s.off_b + st * s.b_ps * s.b_unit;
  s.off_sfb = s.off_sfa + (mx ? st * s.a_ps * 512 : 0);
  s.slot = s.off_sfb + (mx ? st * s.b_ps * 512 : 0);
  s.slot = (s.slot + 1023) & ~1023;
  s.off_slots = xslots * s.xslot;
  s.off_l1 = s.off_slots + (br == BR_NONE ? 0 : slots) * s.slot;
  if (br == BR_MXFP && s.off_l1 < SETTLE_BYTES) s.off_l1 = SETTLE_BYTES;
  s.off_max = s.off_l1 + LQ_MAX_RANK * 4;       // sL1; MXFP: settle_tiles' list
  // row maxima of three tiles in rotation, row scales of two
  s.off_sb = s.off_max + 3 * 64 * 4;
  s.off_bar = s.off_sb + 2 * 64 * 4;
  s.total = s.off_bar + 8 * (2 * MAX_XSLOTS + 3 * MAX_SLOTS + 5) + 16;
  // the 128-row MMA reads past the last slab of a shorter tile
  if (br != BR_NONE && s.total < s.off_l1 + 128 * 128) s.total = s.off_l1 + 128 * 128;
  return s;
}

// Cost model in rounds, a round being one chunk for every team: a CTA's tiles times (its rounds,
// twice where a tile is walked twice, plus three for starting and finishing a tile, or one without a branch: no factor, sums or
// re-quantization wait there, and with three M = 22000, K = 1152 took 17.7 / 13.7 us, caches cold / warm, for 16.5 / 13.1).  It prices
// rounds only: not the second stream of X where an integer branch's tile is larger than the ring (140 MB read for 75 at M = 8192, K =
// 4608), nor what overlaps between tiles.  Of cuts with the same rounds the one with the most warps and then the longer chunks (up to four
// stages) is taken, where a slot's operands are small enough (integer branches, MXFP up to rank 64; the others lose up to 5 % by it) and
// K has the eight stages that fill two such chunks (without that limit 44 more of the timed sizes are over 1.5 % slower than by short
// ones).  Exceptions.  An integer branch, whose ring the long chunks shrink: a ring of two chunks (from five row groups on; us, M =
// 17600, rank 128, K = 1280 / 1664, chunks of 1 and of 3 stages: 27.6 and 31.2 / 33.4 and 37.6), and chunks of two stages where K has an
// odd number of them (M = 32768, rank 32, K = 1408, chunks of 1 and of 2 stages: 41.1 and 42.7; above rank 48 and from 1536 on, or from
// 24 stages on, they are the faster ones all the same).  Elsewhere they may even make a tile too large for the ring: M = 32768, K = 1536,
// rank 64, X streamed once by chunks of 1 and twice by chunks of 2: 49.1 and 45.8.
// MXFP: chunks of two of an odd number below twelve where a CTA has one tile, whose first chunk nothing covers (rank 64, M = 8192, K = 1152,
// caches cold: 11.16 by chunks of 1, 11.43 of 2).
// Eight row groups leave room for one team of eight warps with nothing to run beside its waits: a tenth more a round (SINT4 rank 32, M =
// 17600, K = 640 / 896: 16.2 / 19.0 us by 5 groups, 17.4 / 21.6 by 8).  With the widest factors, which every tile fetches anew, their
// fewer tiles make up for it (rank 128, K = 384: 18.5 and 15.8).
// Timed over the sensible cuts of 11616 sizes (22 formats and ranks, K from 256 to 8192, M from 1 to 32768, caches warm and cold): by one
// round for every tile and none of these rules 3830 of them get another cut, which is 6.4 % slower in the mean; 84 get one that is more
// than 1.5 % faster, 9 % at most (26 more than 4 %: factors of up to 32 columns at K above 5000, tiles of 16 or 24 rows instead of 40 or
// 48, and a few instead of seven or eight groups).  All these times are of the kernel before tiles of up to 32 rows had MMAs of 64 rows,
// branch codes one FMA, and the re-quantization two values to an instruction.
//
// Barrier phases have one bit, so a team that waits for a slot must not be able to mistake the phase before last for the last
// one: the chunk that was in the slot before has to be known to have landed (X) or to have been multiplied (operands).
//   operands  MMAs retire in order, and a team waits for the slots of its own chunks, so as many slots as teams are enough
//   X         copies land in any order.  A team has seen its own earlier chunks land, so the ring holds a multiple of the teams
//             and the chunk before was its own - unless the chunk before is known to have landed for another reason: an
//             integer branch's ring holds a whole tile (the teams meet between the two walks, having seen all of it), or the ring is
//             as long as the teams and the operand slots together (the slot that the team waited for last was free, so every
//             chunk up to the one before had been multiplied).
inline bool plan_cut(int br, int M, int nst, int rn, int bplanes, int sms, int force_groups, int force_stages, QuantCut& out) {
  const int walks = br == BR_INT ? 2 : 1, room = 227 * 1024 - 1024;
  const double per_tile = br == BR_NONE ? 1.0 : 3.0;
  double best = 1e30;
  for (int groups = 8; groups >= 1; --groups) {
    if (force_groups > 0 && groups != force_groups) continue;
    for (int stages = 1; stages <= std::min(QWARPS / groups, nst); ++stages) {
      if (force_stages > 0 && stages != force_stages) continue;
      QuantCut c{};
      c.groups = groups; c.stages = stages;
      c.ntiles = lq_ceil_div(M, 8 * groups);
      c.nchunks = lq_ceil_div(nst, stages);
      for (c.teams = std::min(std::min(QWARPS / (groups * stages), c.nchunks), MAX_SLOTS); c.teams >= 1; --c.teams) {
        c.xslots = 0;
        // operand slots first, then as many chunks of X as fit; an integer branch would rather hold a whole tile of X
        const int want = br == BR_INT ? c.nchunks : 2 * c.teams + 2;
        for (int slots = br == BR_NONE ? 1 : MAX_SLOTS; slots >= (br == BR_NONE ? 1 : std::max(2, c.teams)) && c.xslots < want; --slots) {
          const QuantSmem s = quant_smem(br, 8 * groups, stages, rn, bplanes, slots, 0);
          int fit = std::min(MAX_XSLOTS, (room - s.total) / s.xslot);
          const bool whole = br == BR_INT && fit >= c.nchunks, behind = br != BR_NONE && br != BR_INT && fit >= c.teams + slots;
          if (!whole && !behind) fit -= fit % c.teams;
          if (fit > c.xslots && fit >= std::max(2, 2 * c.teams - (whole ? 1 : 0))) { c.xslots = fit; c.slots = slots; }
        }
        if (c.xslots == 0) continue;
        // no more than two tiles of X (whole turns of the teams, for the reason above)
        const int two = br == BR_INT && c.xslots >= c.nchunks ? std::max(2 * c.teams - 1, 2 * c.nchunks) : lq_round_up(2 * c.nchunks, c.teams);
        c.xslots = std::min(c.xslots, std::max(2, two));
        c.refetch = br == BR_INT && c.xslots < c.nchunks;
        c.smem = quant_smem(br, 8 * groups, stages, rn, bplanes, c.slots, c.xslots).total + 1024;
        const int warps = groups * stages * c.teams;
        const double round = 0.4 + 0.6 * warps / QWARPS + (groups == 8 && rn <= 96 ? 0.1 : 0.0);
        const bool shallow = c.xslots < 3 && groups > 4;
        const bool uneven = stages == 2 && nst % 2 != 0 && (br == BR_INT ? nst < 24 && (rn <= 48 || nst < 12) : nst < 12 && c.ntiles <= sms);
        const bool longer = nst >= 8 && stages <= 4 && !uneven && (br == BR_INT ? !shallow : br == BR_MXFP && rn <= 64);
        const double cost = lq_ceil_div(c.ntiles, sms) * (lq_ceil_div(c.nchunks, c.teams) * walks * round + per_tile) + 3.0 -
                            (longer ? 1e-3 * (warps + stages) : 0.0);
        if (cost < best - 1e-9) { best = cost; out = c; }
        break;
      }
    }
  }
  return best < 1e30;
}

// The same under the options (0: free): what a launch cannot have - more warps than there are, more stages than K has, more shared
// memory than there is - becomes the largest that it can, stages first.
inline bool plan_cut_as_asked(int br, int M, int nst, int rn, int bplanes, int sms, int groups, int stages, QuantCut& out) {
  for (int g = std::min(8, groups);; --g) {
    for (int s = std::min(stages, nst);; --s) {
      if (plan_cut(br, M, nst, rn, bplanes, sms, g, s, out)) return true;
      if (s <= 1) break;
    }
    if (g <= 1) break;
  }
  return plan_cut(br, M, nst, rn, bplanes, sms, 0, 0, out);
}

// Whether X is the first to leave the L2 (126 MB), before the codes, which the GEMM comes for next.  The launch cannot know whether somebody reads X
// again - another layer, a residual sum - so it is so only where X and the codes (bytes) are too large to stay all the same, and then it
// costs nobody anything; nor where an integer branch streams X twice itself.  Timed with and without over X and codes of 36 to 240 MB, K
// from 640 to 4608, four formats: quantizer and GEMM alone, two layers in turn on one X, both quantizers first, X just written, X read
// again behind the GEMM.  Rank 32 / 64, K = 1152, N = 1152:
//   X and codes   MXINT4: one layer, two, quantizers first, read again   MXFP4
//     28 MB       0.972  1.010  1.019  1.014                             0.987  1.017  1.028  1.014   not taken (M = 8192)
//     72 MB       0.986  0.986  0.984  0.988                             0.973  0.975  0.973  0.997   not taken (K = 4608: 0.981  0.997  1.005  0.996)
//    125 MB       0.983  0.980  0.984  0.983                             0.986  0.987  0.982  0.982
//    200 MB       0.996  0.982  1.001  0.997                             0.994  1.002  1.003  0.996   not taken (K = 4608: 0.981  0.989  1.008  0.994)
// MXINT8's codes (two planes) are as large as X: both quantizers first lost 1.0 to 1.7 % at K = 4608, one layer won 1 to 2 %; it is left out.
inline bool x_leaves_first(const QuantCut& c, bool two_planes, double x_and_codes) {
  return !c.refetch && !two_planes && x_and_codes > 80e6 && x_and_codes < 160e6;
}

}  // namespace lqcut
