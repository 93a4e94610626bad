// Activation side of the layer, ONE kernel and one pass of X over HBM (Figure 1; Appendix A.2: both branches
// consume quantized X, except the full-precision reference branch of Section 4.2 / Table 2):
//   a1  codes + scales per token and block along K (SINT4: 64, MX formats: 32; Appendix A.3)
//   a2  per-token codes of the low-rank branch (needs the whole row's maximum first)
//   a3  down-projection I1 = qb L1q on the tensor cores (tcgen05): exact int32 (integer branches), fp16 x fp16 -> fp32
//       (fp16 reference branch), block-scaled (MX branches: the operand IS the main codes and their scale bytes)
//   a4  the rank-r row, re-quantized (per token, or per block of 32 along the rank)
//
// Shape of the kernel (persistent, one CTA per SM, warp-specialised, 20 warps): tiles of TR = 8 RG rows, walked in chunks
// of TR rows x SX stages of 128 values.
//   warp 3      TMA producer of X: a box is TR rows x 64 values; a ring of up to twelve chunks is always in flight, across
//               tiles too
//   warps 5-19  quantizer: teams of RG x SX warps take the chunks in turn; in a chunk each warp has one piece, 8 rows x one
//               stage.  A lane owns 16 neighbouring values of two rows, two 16-byte vectors of X each: they share a block and its
//               scale, a block of 32 is two lanes, its maximum one shuffle, and a lane's codes are one 16-byte store, to global and
//               to shared memory.  (With a vector of each half of the stage to a lane, four lanes to a block, every scale was worked
//               out twice as often and stores were of 8 bytes; us, timed in turn, M = 8192, K = 1152 / 4608, X cold: SINT4 13.8 / 37.4 ->
//               13.4 / 36.2, MXINT4 x 8 13.5 / 37.6 -> 12.9 / 34.2, MXFP4 11.1 / 28.4 -> 11.1 / 28.6; X in the L2: 12.1 / 35.0 -> 11.5 /
//               32.6, 12.5 / 37.7 -> 11.4 / 34.2.)  Loads and stores move whole rows of a box.  (A first version loaded X into registers
//               from global memory, half rows per instruction: the tag stage of the L1 was what bounded it, at 40 lookups a piece, and
//               its unrolled ring cost a microsecond of instruction misses.)  The branch's operand goes to shared memory in the layout
//               the MMA reads (K-major, 128-byte swizzle).  More warps (28 at 64 registers) were no faster, twelve were
//               10-30 % slower
//   warp 4      TMA producer of the first factor's slabs, one per stage, and their scale bytes.  (The MMA warp fetched them at
//               first, after the chunk it had just issued: the slabs were late, 24 against 30 us at K = 4608)
//   warp 2      owns tensor memory, issues the MMAs of a chunk once its slabs are complete.  The MMA is 128 rows high, or 64 (mma_64_rows); the rows
//               beyond TR read whatever follows in shared memory and their results are never looked at (rows are
//               independent, and the tensor cores are idle here otherwise)
//   warps 0-1   a4: lane = row; the rank-r row is read from tensor memory under the next tile's quantization (two
//               accumulator sets alternate)
// An integer branch needs the row's maximum before its first code: the tile is walked twice, the first time for the main
// codes and the maximum, the second time for the branch codes - from the ring when it holds the whole tile, else
// streamed again from the L2.
//
// Exactness contract: codes and scales equal the definition evaluated in IEEE binary32 with
// round-to-nearest-even and true division.  The kernel is division free:
//   scale     fp16(a / 7) == fp16(a * fl32(1/7)) for every finite fp16 a (checked exhaustively on the host),
//             because a/7 never comes closer than 2^-15 (relative) to an fp16 midpoint.
//   SINT4     x and s are 11-bit numbers, so x / s is either exactly k + 1/2 or at least 2^-14 away from it.  The product
//             with a reciprocal that is an ulp or two off is within 2^-19 of the quotient; adding 192 rounds it to a multiple of 2^-16,
//             which restores exact ties and moves nothing else across one; a second addition then rounds to the integer, ties to even.
//   branch    x / sb is within 2^-23 of qm x / max, which is either exactly k + 1/2 or at least 2^-19 away from it (11-bit numbers, qm of 5
//             or 7 bits); so one FMA with 1.5 * 2^23 and a reciprocal good to 2^-21 rounds like the quotient everywhere but on such
//             ties.  As qm is prime they are at x = +-max / 2, for which the reciprocal is taken on the side that gives the quotient's code
//             (BranchScale), or the maximum's significand is a multiple of qm: such rows go by the correctly rounded
//             quotient, from the reciprocal by one FMA correction step.
//   MX        x * 2^-e is exact, and the fp16 pipe does it two values at a time: one fma with 1.5 * 2^10 rounds x * 2^-e to
//             the nearest even integer without an intermediate rounding; blocks so small that 2^-e is no fp16 number
//             are scaled up (exactly) first, a rare branch.  MXFP8e4: products below 2^-14 may lose bits, far below half of e4m3's
//             smallest step 2^-9.
#include <cuda_fp16.h>
#include <math.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "lq_device.cuh"
#include "lq_quant_cut.h"

namespace {

using namespace lqdev;
using namespace lqcut;

constexpr int FIRST_QWARP = 5;         // warps 0-1 a4, 2 MMA, 3 X, 4 first factor
constexpr int NTHREADS = (FIRST_QWARP + QWARPS) * 32;
constexpr float MAGIC = 12582912.0f;   // 1.5 * 2^23: adding it rounds to an integer (ties to even)
// MXFP: MXFP8e4 activation codes for an MXFP4 weight; MXINT8: MXINT8 activation codes for an MXINT4 weight, stored as
// two E4M3 digit planes (code = 16 hi + lo); MXFP6: MXFP6e2 activation codes, stored as the E4M3 bytes of the same values
enum { MAIN_SINT4 = 0, MAIN_MXINT4 = 1, MAIN_MXFP = 2, MAIN_MXINT8 = 3, MAIN_MXFP6 = 4 };

struct QuantParams : QuantCut {
  int M, K, Kpad, Mpad;
  int nst;              // Kpad / 128 stages of K
  uint8_t* qx8;         // [Mpad][Kpad] (MXINT8: [Mpad][2 Kpad], the hi digits' plane then the lo digits')
  float* sx;            // [Gpad][Mpad]
  uint8_t* sfa;         // MX: E8M0 scale bytes [Mpad/128][Kpad/128][512] (MXINT8: [Mpad/128][2 Kpad/128][512], by plane)
  int8_t* qb;           // [Mpad][Kpad] or null (not stored)
  float* sXb;           // [Mpad]
  const float* sL1;     // [LQ_MAX_RANK]
  const uint8_t* l1c;   // MXFP: the first factor's elements, [rn][Kpad] (the MMA reads them through tmL1)
  uint32_t* near;       // MXFP: [Mpad], bit b: block b of the row's intermediate is near a tie
  uint32_t* near_which; // MXFP: [Mpad][4], where so: its elements
  const uint8_t* sfl1;  // MX branches: E8M0 bytes of the first factor's block scales, [Kpad/128][512]
  uint8_t* sft;         // MX branches: E8M0 bytes of the rank-r intermediate's block scales, [Mpad/128][512 or 1024]
  uint8_t* tq;          // [Mpad][tq_stride]
  float* sT;            // [Mpad]
  int r, rn;            // rank, rank rounded up to 16 (columns of the MMA)
  int bplanes;          // digit planes of the first factor, side by side in the MMA's columns (2: MXINT8 factors, else 1)
  int tq_stride;        // bytes per row of tq: LQ_RCONT, or 2 LQ_RCONT when each digit plane of the intermediate has a container
  int nacc, sets;       // accumulators a tile's stages alternate over (floating-point branches: shorter chains of fp32 sums),
                        // sets of them (2: the next tile's MMAs run under a4)
  int tmem_cols;        // power of two
  float dev;            // MXFP: how far a sum of the tensor core is taken to be from the one in settle_tiles' order, over its block's maximum
  float unit;           // MX branches: the intermediate over the tensor core's sums (a power of two, 1 but for tiny first factors)
  float qm, rqm;        // largest branch activation code, 1 over it
  float near_tie;       // half an ulp of qm / 2
  int32_t* status;
  const uint8_t* X;     // [M][2 K], where a CTA's first tile is fetched ahead, else null
};

// Position in a ring of n slots and the parity its barriers have there.
struct Ring {
  int at;
  uint32_t par;
  __device__ __forceinline__ void step(int by, int n) {
    for (at += by; at >= n; at -= n) par ^= 1;
  }
};

__device__ __forceinline__ __half2 as_half2(uint32_t v) { return *reinterpret_cast<const __half2*>(&v); }
__device__ __forceinline__ uint32_t as_u32(__half2 v) { return *reinterpret_cast<const uint32_t*>(&v); }
__device__ __forceinline__ float2 splat(float v) { return make_float2(v, v); }
__device__ __forceinline__ float pow2f_n(int e) { return __uint_as_float((uint32_t)(e + 127) << 23); }   // -126 <= e <= 127

// two floats -> two E4M3 bytes (hi: first operand, lo: second)
__device__ __forceinline__ uint32_t f32x2_to_e4m3x2(float hi, float lo) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
  return (uint32_t)r;
}
__device__ __forceinline__ uint32_t f16x4_to_e4m3x4(__half2 a, __half2 b) {
  uint32_t w;
  asm("{\n\t.reg .b16 lo, hi;\n\tcvt.rn.satfinite.e4m3x2.f16x2 lo, %1;\n\tcvt.rn.satfinite.e4m3x2.f16x2 hi, %2;\n\t"
      "mov.b32 %0, {lo, hi};\n\t}" : "=r"(w) : "r"(as_u32(a)), "r"(as_u32(b)));
  return w;
}

// largest magnitude of eight halves (one 16-byte vector), exact in fp16
__device__ __forceinline__ __half absmax8(const uint4& a) {
  const __half2 m = __hmax2(__hmax2(__habs2(as_half2(a.x)), __habs2(as_half2(a.y))), __hmax2(__habs2(as_half2(a.z)), __habs2(as_half2(a.w))));
  return __hmax(__low2half(m), __high2half(m));
}

// Block exponents and factors 2^-e of two rows at once, from the fp16 bit patterns of their block maxima (the low half: the
// first row).  e = E' - TOP, E' the maximum's binary exponent, one more where its mantissa is beyond 0x400 - UP.  The
// exponent fields stay where they are in the halves: two integer instructions give both factors.  Where a factor would
// not be a normal fp16 number - a maximum below 2^-7 or less, an all-zero block - `ok` is false.
template <int TOP, int UP>
struct PairScale {
  uint32_t inv;          // the factors' bit patterns
  uint32_t bytes;        // E8M0 bytes: first row in bits 0-7, second in bits 16-23
  bool ok;
  __device__ __forceinline__ explicit PairScale(uint32_t bm) {
    const uint32_t m = (bm + (uint32_t)(UP * 0x10001)) & 0x7C007C00u;
    inv = (uint32_t)((30 + TOP) << 10) * 0x10001u - m;
    bytes = (m >> 10) + (uint32_t)(112 - TOP) * 0x10001u;
    ok = (m & 0xFFFFu) >= (TOP << 10) && m >= ((uint32_t)TOP << 26);
  }
};
// The same factor for one row and any exponent (1 for the all-zero block's -127).  Where 2^-e is out of fp16's range the
// values are scaled up, exactly, and e follows.
__device__ __forceinline__ __half2 half_scale(uint4& v, int e) {
  if (e > -127) {
    const __half2 up = __float2half2_rn(4096.f);
    for (; e < -15; e += 12) {
      v.x = as_u32(__hmul2(as_half2(v.x), up)); v.y = as_u32(__hmul2(as_half2(v.y), up));
      v.z = as_u32(__hmul2(as_half2(v.z), up)); v.w = as_u32(__hmul2(as_half2(v.w), up));
    }
  }
  return __half2half2(__ushort_as_half((unsigned short)((15 - (e == -127 ? 0 : e)) << 10)));
}

// MXFP8e4 / MXFP6e2 of eight values that share a block (Appendix A.3 "MX Formats"; conversion of the OCP specification
// the paper cites): the block's exponent is e = floor(log2 a) - emax for the block maximum a (emax = 8: e4m3's largest
// binade, 2: e2m3's), -127 for an all-zero block; the elements are x / 2^e - exact - rounded to the element format by
// the hardware conversion (nearest even, magnitudes above the largest normal clamped).  Every e2m3 value is an e4m3
// value, so both formats are stored, and multiplied, as e4m3 bytes: the 6-bit path rounds to e2m3 first and widens
// the result (e2m3 -> f16 -> e4m3, both exact).
template <bool SIX>
__device__ __forceinline__ int mxfp_exponent(float a) {
  const int e = (int)(__float_as_uint(a) >> 23) - 127 - (SIX ? 2 : 8);
  return (a > 0.f && e >= -126) ? e : -127;
}
__device__ __forceinline__ uint32_t f32x2_to_e4m3x2_via_e2m3(float hi, float lo) {
  uint16_t r6, r8;
  uint32_t h2;
  asm("cvt.rn.satfinite.e2m3x2.f32 %0, %1, %2;" : "=h"(r6) : "f"(hi), "f"(lo));
  asm("cvt.rn.f16x2.e2m3x2 %0, %1;" : "=r"(h2) : "h"(r6));
  asm("cvt.rn.satfinite.e4m3x2.f16x2 %0, %1;" : "=h"(r8) : "r"(h2));
  return (uint32_t)r8;
}
template <bool SIX>
__device__ __forceinline__ uint32_t mxfp_pair(float hi, float lo) {
  return SIX ? f32x2_to_e4m3x2_via_e2m3(hi, lo) : f32x2_to_e4m3x2(hi, lo);
}
__device__ __forceinline__ uint2 mxfp6_codes8(const uint4& v, int e) {
  const float inv = e == -127 ? 0.f : pow2f_n(-e);
  const float2 a = __half22float2(as_half2(v.x)), b = __half22float2(as_half2(v.y)), c = __half22float2(as_half2(v.z)),
               d = __half22float2(as_half2(v.w));
  return make_uint2(f32x2_to_e4m3x2_via_e2m3(a.y * inv, a.x * inv) | (f32x2_to_e4m3x2_via_e2m3(b.y * inv, b.x * inv) << 16),
                    f32x2_to_e4m3x2_via_e2m3(c.y * inv, c.x * inv) | (f32x2_to_e4m3x2_via_e2m3(d.y * inv, d.x * inv) << 16));
}
__device__ __forceinline__ uint2 mxfp8_codes8(const uint4& v, __half2 inv) {
  auto q = [&](uint32_t h) { return __hmul2(as_half2(h), inv); };
  return make_uint2(f16x4_to_e4m3x4(q(v.x), q(v.y)), f16x4_to_e4m3x4(q(v.z), q(v.w)));
}

// MXINT4 (Appendix A.3): 2^e with e the smallest integer such that 7 * 2^e >= a: a = 1.f * 2^E, e = E - 2 if 1.f <= 1.75
// else E - 1; -127 for an all-zero block.  Codes rint_even(x / 2^e) as E4M3 bytes.
__device__ __forceinline__ int mxint4_exponent(float a) {
  const uint32_t ab = __float_as_uint(a);
  return a > 0.f ? (int)(ab >> 23) - 127 - (((ab & 0x7FFFFFu) <= 0x600000u) ? 2 : 1) : -127;
}
__device__ __forceinline__ uint2 mxint4_codes8(const uint4& v, __half2 inv) {
  const __half2 magic = __float2half2_rn(1536.f);
  auto q = [&](uint32_t h) { return __hsub2(__hfma2(as_half2(h), inv, magic), magic); };
  return make_uint2(f16x4_to_e4m3x4(q(v.x), q(v.y)), f16x4_to_e4m3x4(q(v.z), q(v.w)));
}

// MXINT8 (signed 8-bit codes, blocks of 32, power-of-two scale): the block's exponent is the smallest e with
// 127 * 2^e >= a for the block maximum a = 1.f * 2^E: e = E - 6 if 1.f <= 127/64, else E - 5; at least -127, and -127
// for an all-zero block.
__device__ __forceinline__ int mxint8_exponent(float a) {
  const uint32_t ab = __float_as_uint(a);
  const int e = (int)(ab >> 23) - 127 - (((ab & 0x7FFFFFu) <= 0x7E0000u) ? 6 : 5);
  return a > 0.f ? max(e, -127) : -127;
}
// The code c = rint_even(x / 2^e) of eight values as two digits, c = 16 hi + lo, lo in [-8, 7], hi in [-8, 8], both exact
// E4M3 values: hi = rint((c + 1/4) / 16), every step exact in fp16 (|c| <= 127).
__device__ __forceinline__ void mxint8_codes8(const uint4& v, __half2 inv, uint2& hi, uint2& lo) {
  const __half2 magic = __float2half2_rn(1536.f), sixteenth = __float2half2_rn(0.0625f), bias = __float2half2_rn(0.015625f),
                m16 = __float2half2_rn(-16.f);
  __half2 h[4], l[4];
  const uint32_t x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __half2 c = __hsub2(__hfma2(as_half2(x[i]), inv, magic), magic);
    h[i] = __hsub2(__hadd2(__hfma2(c, sixteenth, bias), magic), magic);
    l[i] = __hfma2(h[i], m16, c);
  }
  hi = make_uint2(f16x4_to_e4m3x4(h[0], h[1]), f16x4_to_e4m3x4(h[2], h[3]));
  lo = make_uint2(f16x4_to_e4m3x4(l[0], l[1]), f16x4_to_e4m3x4(l[2], l[3]));
}
// Two fp32 values (of the rank-r intermediate) under their block's exponent, the same digits.
__device__ __forceinline__ void mxint8_digits(float2 x, float inv, float2& hi, float2& lo) {
  const float2 up = splat(MAGIC), down = splat(-MAGIC);
  const float2 c = __fadd2_rn(__ffma2_rn(x, splat(inv), up), down);
  hi = __fadd2_rn(__fadd2_rn(__ffma2_rn(c, splat(0.0625f), splat(0.015625f)), up), down);
  lo = __ffma2_rn(hi, splat(-16.f), c);
}

// Two rows' vectors whose block maxima are out of PairScale's range (MXFP6e2: any): kept out of the main loop's instructions.
// The E8M0 bytes come as PairScale has them.
struct RareCodes {
  uint2 wa, wb, da, db;
  uint32_t bytes;
};
template <int MAIN>
__device__ __noinline__ RareCodes rare_codes(uint4 a, uint4 b, __half2 bm) {
  const float m0 = __low2float(bm), m1 = __high2float(bm);
  RareCodes r;
  r.da = r.db = make_uint2(0, 0);
  int e0, e1;
  if constexpr (MAIN == MAIN_MXFP6) {
    e0 = mxfp_exponent<true>(m0); e1 = mxfp_exponent<true>(m1);
    r.wa = mxfp6_codes8(a, e0); r.wb = mxfp6_codes8(b, e1);
  } else if constexpr (MAIN == MAIN_MXFP) {
    e0 = mxfp_exponent<false>(m0); e1 = mxfp_exponent<false>(m1);
    const __half2 i0 = half_scale(a, e0), i1 = half_scale(b, e1);
    r.wa = mxfp8_codes8(a, i0); r.wb = mxfp8_codes8(b, i1);
  } else if constexpr (MAIN == MAIN_MXINT4) {
    e0 = mxint4_exponent(m0); e1 = mxint4_exponent(m1);
    const __half2 i0 = half_scale(a, e0), i1 = half_scale(b, e1);
    r.wa = mxint4_codes8(a, i0); r.wb = mxint4_codes8(b, i1);
  } else {
    e0 = mxint8_exponent(m0); e1 = mxint8_exponent(m1);
    const __half2 i0 = half_scale(a, e0), i1 = half_scale(b, e1);
    mxint8_codes8(a, i0, r.wa, r.da); mxint8_codes8(b, i1, r.wb, r.db);
  }
  r.bytes = (uint32_t)(e0 + 127) | ((uint32_t)(e1 + 127) << 16);
  return r;
}

// SINT4 (Appendix A.3): fp16 scales a / 7 (at least 2^-24) of two rows from their group maxima; the reciprocals may be an
// ulp off (see the top).  Codes rint_even(x / s) clamped to [-7, 7]; only a subnormal scale can leave the quotient above 7.5.
struct Sint4Scale {
  float s[2], inv[2];
  bool coarse;
  __device__ __forceinline__ explicit Sint4Scale(__half2 a) {
    const float2 f = __half22float2(a);
    const __half2 s16 = __floats2half2_rn(__fmul_rn(f.x, 0.142857149243354797f), __fmul_rn(f.y, 0.142857149243354797f));   // fl32(1/7)
    const uint32_t bits = __vmaxu2(as_u32(s16), 0x00010001u);           // floor 2^-24
    const float2 g = __half22float2(as_half2(bits));
    s[0] = g.x; s[1] = g.y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv[0]) : "f"(g.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv[1]) : "f"(g.y));
    coarse = (bits & 0xFFFFu) < 0x0400u || bits < 0x04000000u;
  }
};
__device__ __forceinline__ uint4 vec16(const uint2 (&v)[2]) { return make_uint4(v[0].x, v[0].y, v[1].x, v[1].y); }
__device__ __forceinline__ uint2 sint4_codes8(const uint4& v, float rcp, bool coarse) {
  const float2 x[4] = {__half22float2(as_half2(v.x)), __half22float2(as_half2(v.y)), __half22float2(as_half2(v.z)), __half22float2(as_half2(v.w))};
  const float2 inv = splat(rcp), c0 = splat(192.f), c1 = splat(MAGIC - 192.f), c2 = splat(-MAGIC);
  float2 q[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) q[i] = __fadd2_rn(__fadd2_rn(__ffma2_rn(x[i], inv, c0), c1), c2);
  if (coarse) {
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = make_float2(fminf(fmaxf(q[i].x, -7.f), 7.f), fminf(fmaxf(q[i].y, -7.f), 7.f));
  }
  return make_uint2(f32x2_to_e4m3x2(q[0].y, q[0].x) | (f32x2_to_e4m3x2(q[1].y, q[1].x) << 16),
                    f32x2_to_e4m3x2(q[2].y, q[2].x) | (f32x2_to_e4m3x2(q[3].y, q[3].x) << 16));
}

// Scale of a row's branch codes (its maximum over qm, 1 for a row of zeros) and the reciprocal that codes are formed with (see the top).  All of
// a tile's warps wait for it between its two walks, so it is worked out without a division: the maximum over a constant is the correctly
// rounded quotient after one correction step (checked for every fp16 maximum on the host), and where codes do not need the quotient an
// approximate reciprocal will do.
struct BranchScale {
  float sb, inv;
  bool exact;            // this row's codes need the quotient: ties elsewhere, or a maximum that is no number
  // rqm: fl32(1 / qm); near: half an ulp of qm / 2
  __device__ __forceinline__ BranchScale(uint32_t max_bits, float qm, float rqm, float near) {
    const float rm = __half2float(__ushort_as_half((unsigned short)max_bits));
    const float q0 = __fmul_rn(rm, rqm), q1 = __fmaf_rn(__fmaf_rn(q0, -qm, rm), rqm, q0);
    sb = rm == 0.f ? 1.f : max_bits >= 0x7C00u ? rm : q1;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(sb));
    const float a = (float)((max_bits & 0x3FFu) | (max_bits < 0x400u ? 0u : 0x400u));       // significand of the maximum
    exact = max_bits >= 0x7C00u || (a != 0.f && __fmul_rn(rintf(__fmul_rn(a, rqm)), qm) == a);
    // The code of max / 2 is rint(fl32(max / 2 / sb)).  The quotient is within 2^-23 of qm / 2, which is half of an odd number plus one:
    // ties go up, and what is no more than half an ulp below is a tie.  (max / 2 - sb qm / 2 is exact, half of the division's remainder.)
    const bool up = __fmaf_rn(sb, -0.5f * qm, 0.5f * rm) >= -near * sb;
    if ((__fmaf_rn(0.5f * rm, inv, -0.5f * qm) >= 0.f) != up) inv = __uint_as_float(__float_as_uint(inv) + (up ? 4u : -4u));
  }
};
// Branch codes of eight values: the low byte of the code + MAGIC is the code.
__device__ __forceinline__ uint2 low_bytes8(const float2 (&q)[4]) {
  uint32_t t[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) { t[2 * i] = __float_as_uint(q[i].x); t[2 * i + 1] = __float_as_uint(q[i].y); }
  return make_uint2(__byte_perm(__byte_perm(t[0], t[1], 0x0040), __byte_perm(t[2], t[3], 0x0040), 0x5410),
                    __byte_perm(__byte_perm(t[4], t[5], 0x0040), __byte_perm(t[6], t[7], 0x0040), 0x5410));
}
__device__ __forceinline__ uint2 branch_codes8(const uint4& v, float inv) {
  const float2 x[4] = {__half22float2(as_half2(v.x)), __half22float2(as_half2(v.y)), __half22float2(as_half2(v.z)), __half22float2(as_half2(v.w))};
  const float2 y = splat(inv), magic = splat(MAGIC);
  float2 q[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) q[i] = __ffma2_rn(x[i], y, magic);
  return low_bytes8(q);
}
// The same by the quotient, inv = fl32(1 / sb): q0 = fl32(x inv) is within one ulp of x / sb, r = x - sb q0 is exact in an FMA, and
// fl32(q0 + r inv) is then the correctly rounded quotient (Markstein's correction step); |x| / sb <= qm (1 + 2^-23), so it never
// leaves [-qm, qm].
__device__ __forceinline__ uint2 branch_codes8_exact(const uint4& v, float sb, float inv) {
  const float2 x[4] = {__half22float2(as_half2(v.x)), __half22float2(as_half2(v.y)), __half22float2(as_half2(v.z)), __half22float2(as_half2(v.w))};
  const float2 y = splat(inv), ns = splat(-sb), magic = splat(MAGIC);
  float2 q[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 q0 = __fmul2_rn(x[i], y);
    q[i] = __fadd2_rn(__ffma2_rn(__ffma2_rn(q0, ns, x[i]), y, q0), magic);
  }
  return low_bytes8(q);
}

// Near ties of the MXFP intermediate T = deq(Q(X)) deq(Q2(L1)).  Floating-point elements round in steps of up to a fourteenth of the
// block's maximum, so a sum that lands on the other side of a tie shows in Y.  Blocks of T that are too close to call on the
// tensor core's sum - the block's exponent, an element of the largest binade - are settled on the sum in one fixed order
// instead: a partial sum of 32 products per block of K on mma.sync, fp32 additions of the scaled partial sums in nine
// interleaved chains (box g of 64 values belongs to chain g mod 9, its second block first), the chains added in order.  What
// is settled is decided for each element by itself, so a row's codes do not depend on the rows around it.
// "Too close" is measured, not a bound: the tensor core's sum differs from the other by less than 2^-22.2 of the block's
// maximum in 999 of 1000 elements at K = 1152, 2^-20.6 at K = 4608 with one-sided inputs.  An element beyond that keeps the code of the
// tensor core's sum, which is as near to the exact one.
template <bool SIX>
struct TieTest {
  float k, limit;
  __device__ __forceinline__ TieTest(float inv, float dev) : k(inv * (SIX ? 2.f : 0.03125f)), limit(0.5f - dev * k) {}
  // elements of the largest binade (steps of 32 in e4m3, 1/2 in e2m3) whose distance to the nearest code is within the deviation of
  // half a step
  __device__ __forceinline__ bool operator()(float x) const {
    const float u = fabsf(x) * k;
    return u > 7.5f && fabsf(u - __fadd_rn(__fadd_rn(u, MAGIC), -MAGIC)) > limit;
  }
  // whether one of them is that close to half a step of the largest binade, in whichever binade it is
  __device__ __forceinline__ bool any(const float (&x)[32]) const {
    float far[2] = {0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float2 u = __fmul2_rn(make_float2(x[2 * i], x[2 * i + 1]), splat(k));
      const float2 d = __ffma2_rn(__fadd2_rn(__fadd2_rn(u, splat(MAGIC)), splat(-MAGIC)), splat(-1.f), u);
      far[0] = fmaxf(far[0], fabsf(d.x)); far[1] = fmaxf(far[1], fabsf(d.y));
    }
    return fmaxf(far[0], far[1]) > limit;
  }
};
__device__ __forceinline__ void mma_e4m3_16832(float (&c)[4], const uint2& a0, const uint2& a1, const uint2& b) {
  asm("mma.sync.aligned.m16n8k32.row.col.f32.e4m3.e4m3.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0.x), "r"(a1.x), "r"(a0.y), "r"(a1.y), "r"(b.x), "r"(b.y));
}
__device__ __forceinline__ float e8m0(uint32_t byte) { return __uint_as_float((byte & 0xFFu) << 23); }
__device__ __forceinline__ size_t sf_row(int m) { return 16 * (m & 31) + 4 * ((m & 127) >> 5); }

// Settled are the elements that are near a tie, or with the exponent in doubt all of the block's: a few of a CTA one after the other,
// more by tiles.  Both sum in the same order, so which of the two it is shows in the time only.  A launch of 8192 rows and rank 64
// meets an element every few times at K = 1152 and most times at K = 4608; us at K = 4608 without / with one: 27.0 / 26.7 - it is gone
// in the launch's end - against 31.8 by tiles.  An element takes about 0.4 us, a round by tiles 1.6 us at K = 1152 and 4.7 us at K =
// 4608, hence the line between them.  One value per row, where most blocks are exact ties: 18.6 and 48 us by tiles, 610 and
// 815 element by element.
constexpr int SETTLE_ROWS = 16, SETTLE_ENTRIES = 18;
__device__ __forceinline__ int settle_few(int K) { return 2 + K / 512; }   // 18 at most: never all of a block's 32
struct SettleList {
  int entries, elements;           // near blocks and elements that the CTA met
  union {
    int4 entry[SETTLE_ENTRIES];    // (row, block, elements, exponent)
    struct {
      int n[4];                    // rows of a round, by block
      int row[4][SETTLE_ROWS];
    };
  };
};
static_assert(sizeof(SettleList) <= LQ_MAX_RANK * 4, "the list lies where other branches keep sL1");

// One element after the other (all threads of the CTA, after its last tile).  Eight blocks of K per MMA: row i of A and column i of B
// hold block i, so the products wanted are on the diagonal, and loads are contiguous.
// (What this kernel has written itself is read through the L2, here and below.)
template <bool SIX>
__device__ __forceinline__ void settle_elements(const QuantParams& p, float* part, const SettleList& list) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3, blocks = p.Kpad / 32, n = list.entries;
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const int4 what = list.entry[i];
    const int m = what.x, b = what.y;
    const uint8_t* qx = p.qx8 + (size_t)m * p.Kpad;
    const uint8_t* sfx = p.sfa + (size_t)(m >> 7) * (p.Kpad >> 7) * 512 + sf_row(m);
    float mine = 0.f;
#pragma unroll 1
    for (uint32_t todo = (uint32_t)what.z; todo != 0; todo &= todo - 1) {
      const int j = __ffs(todo) - 1, col = 32 * b + j;
      if (col >= p.r) break;
      const uint8_t *l1 = p.l1c + (size_t)col * p.Kpad, *sfl = p.sfl1 + sf_row(col);
#pragma unroll 1
      for (int b0 = 8 * warp; b0 < blocks; b0 += 8 * (NTHREADS / 32)) {
        const int k = b0 + gid;                                  // (blocks is a multiple of 4)
        uint2 a = make_uint2(0, 0), w = a;
        float sc = 0.f;
        if (k < blocks) {
          a = __ldcg(reinterpret_cast<const uint2*>(qx + 32 * k + 8 * tig));
          w = __ldg(reinterpret_cast<const uint2*>(l1 + 32 * k + 8 * tig));
          sc = e8m0(__ldcg(sfx + (k >> 2) * 512 + (k & 3))) * e8m0(__ldg(sfl + (k >> 2) * 512 + (k & 3)));
        }
        float c[4] = {0.f, 0.f, 0.f, 0.f};
        mma_e4m3_16832(c, a, make_uint2(0, 0), w);
        if (tig == (gid >> 1) && k < blocks) part[k] = ((gid & 1) ? c[1] : c[0]) * sc;
      }
      __syncthreads();
      if (warp == 0) {
        float chain = 0.f, v = 0.f;
        if (lane < SETTLE_CHAINS)
          for (int k = 2 * lane; k < blocks; k += 2 * SETTLE_CHAINS) chain = __fadd_rn(part[k], __fadd_rn(part[k + 1], chain));
        for (int c = 0; c < SETTLE_CHAINS; ++c) v = __fadd_rn(v, __shfl_sync(0xffffffffu, chain, c));
        if (lane == j) mine = v;
      }
      __syncthreads();
    }
    if (warp == 0) {
      const float inv = what.w == -127 ? 0.f : pow2f_n(-what.w) * p.unit;
      if (((uint32_t)what.z >> lane) & 1) p.tq[(size_t)m * p.tq_stride + 32 * b + lane] = (uint8_t)mxfp_pair<SIX>(0.f, mine * inv);
    }
  }
}

// By tiles: all near blocks of the CTA in rounds of up to sixteen rows for each block of the rank: warp 9 h + c sums chain c of sixteen
// of the 32 elements, then a warp adds a row's chains and quantizes them as a4 does.  What bounds it is the tag stage of the L1:
// eight rows or columns to a load.
template <bool SIX>
__device__ __forceinline__ void settle_tiles(const QuantParams& p, float* part, SettleList& list) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3, TR = 8 * p.groups;
  const int half = warp / SETTLE_CHAINS, chain = warp - half * SETTLE_CHAINS, boxes = p.Kpad / 64;
  const int rows = (p.ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x * TR;   // of this CTA
#pragma unroll 1
  for (int r0 = 0; r0 < rows; r0 += NTHREADS) {
    const int at_row = r0 + (int)threadIdx.x, m = ((int)blockIdx.x + at_row / TR * (int)gridDim.x) * TR + at_row % TR;
    uint32_t pending = at_row < rows && m < p.M ? __ldcg(p.near + m) : 0;
#pragma unroll 1
    while (__syncthreads_or(pending != 0)) {
      if (threadIdx.x < 4) list.n[threadIdx.x] = 0;
      __syncthreads();
      for (uint32_t todo = pending; todo != 0; todo &= todo - 1) {
        const int b = __ffs(todo) - 1, n = atomicAdd(&list.n[b], 1);
        if (n < SETTLE_ROWS) { list.row[b][n] = m; pending &= ~(1u << b); }
      }
      __syncthreads();
#pragma unroll 1
      for (int b = 0; 32 * b < p.rn; ++b) {
        const int n = min(list.n[b], SETTLE_ROWS);
        if (n == 0) continue;
        if (half < 2) {
          // rows gid and gid + 8 of the round (beyond its end: the first one again), columns 16 half + 8 t + gid of the block
          const int m0 = list.row[b][gid < n ? gid : 0], m1 = list.row[b][gid + 8 < n ? gid + 8 : 0];
          const uint8_t* x0 = p.qx8 + (size_t)m0 * p.Kpad + 8 * tig;
          const uint8_t* x1 = p.qx8 + (size_t)m1 * p.Kpad + 8 * tig;
          const uint8_t* s0 = p.sfa + (size_t)(m0 >> 7) * (p.Kpad >> 7) * 512 + sf_row(m0);
          const uint8_t* s1 = p.sfa + (size_t)(m1 >> 7) * (p.Kpad >> 7) * 512 + sf_row(m1);
          const int c0 = 32 * b + 16 * half;                     // (the rank rounded up to 16 may end in the middle of the block)
          const bool live = c0 < p.rn;
          const uint8_t* w = p.l1c + (size_t)(c0 + gid) * p.Kpad + 8 * tig;
          const uint8_t* sl = p.sfl1 + sf_row(c0 + 2 * tig);
          float acc[2][4] = {};
          if (live) {
#pragma unroll 1
            for (int g = chain; g < boxes; g += SETTLE_CHAINS) {
              const int at = (g >> 1) * 512 + 2 * (g & 1);       // the box's two scale bytes
              const uint32_t e0 = __ldcg(reinterpret_cast<const uint16_t*>(s0 + at)), e1 = n > 8 ? __ldcg(reinterpret_cast<const uint16_t*>(s1 + at)) : 0;
              uint2 a0[2], a1[2], wt[2][2];
              uint32_t el[2][2];
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                a0[h] = __ldcg(reinterpret_cast<const uint2*>(x0 + 64 * g + 32 * h));
                a1[h] = n > 8 ? __ldcg(reinterpret_cast<const uint2*>(x1 + 64 * g + 32 * h)) : make_uint2(0, 0);
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                  wt[t][h] = __ldg(reinterpret_cast<const uint2*>(w + (size_t)(8 * t) * p.Kpad + 64 * g + 32 * h));
                  el[t][h] = __ldg(reinterpret_cast<const uint16_t*>(sl + at + 128 * t + 16 * h));   // columns 2 tig + h
                }
              }
#pragma unroll
              for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int h = 1; h >= 0; --h) {
                  float f[4] = {0.f, 0.f, 0.f, 0.f};
                  mma_e4m3_16832(f, a0[h], a1[h], wt[t][h]);
                  const float r0 = e8m0(e0 >> (8 * h)), r1 = e8m0(e1 >> (8 * h)), ca = e8m0(el[t][0] >> (8 * h)), cb = e8m0(el[t][1] >> (8 * h));
                  acc[t][0] = __fadd_rn(f[0] * (r0 * ca), acc[t][0]); acc[t][1] = __fadd_rn(f[1] * (r0 * cb), acc[t][1]);
                  acc[t][2] = __fadd_rn(f[2] * (r1 * ca), acc[t][2]); acc[t][3] = __fadd_rn(f[3] * (r1 * cb), acc[t][3]);
                }
            }
          }
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            float* to = part + (chain * SETTLE_ROWS + gid) * 32 + 16 * half + 8 * t + 2 * tig;
            to[0] = acc[t][0]; to[1] = acc[t][1];
            to[8 * 32] = acc[t][2]; to[8 * 32 + 1] = acc[t][3];
          }
        }
        __syncthreads();
        if (warp < n) {
          const int mr = list.row[b][warp];
          float v = 0.f;
          for (int c = 0; c < SETTLE_CHAINS; ++c) v = __fadd_rn(v, part[(c * SETTLE_ROWS + warp) * 32 + lane]);
          float amax = fabsf(v);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
          const uint32_t which = __ldcg(p.near_which + 4 * (size_t)mr + b);
          uint8_t* const sf = p.sft + (size_t)(mr >> 7) * 512 + sf_row(mr) + b;
          const int e = which == 0xFFFFFFFFu ? mxfp_exponent<SIX>(amax * p.unit) : (int)__ldcg(sf) - 127;
          const float inv = e == -127 ? 0.f : pow2f_n(-e) * p.unit;
          __syncwarp();
          if ((which >> lane) & 1) p.tq[(size_t)mr * p.tq_stride + 32 * b + lane] = (uint8_t)mxfp_pair<SIX>(0.f, v * inv);
          if (lane == 0) *sf = (uint8_t)(e + 127);
        }
        __syncthreads();
      }
    }
  }
}

// A stage's MMAs under one election, predicated instead of branched around.  (Against an `if` of one lane around them, us, M = 8192,
// K = 1152 / 4608: MXFP rank 64 10.5 / 29.1 -> 10.2 / 28.4, SINT4 rank 32 12.4 / 37.3 -> 12.2 / 36.8; M = 256, K = 1152: 6.9 -> 6.6.)
template <int KIND>
__device__ __forceinline__ void issue_four(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  if constexpr (KIND == TC_I8) {
    asm volatile(
        "{\n\t.reg .pred P, T, A;\n\t"
        "elect.sync _|P, 0xffffffff;\n\t"
        "setp.ne.b32 A, %10, 0;\n\t"
        "setp.eq.b32 T, 0, 0;\n\t"
        "@P tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %5, %9, A;\n\t"
        "@P tcgen05.mma.cta_group::1.kind::i8 [%0], %2, %6, %9, T;\n\t"
        "@P tcgen05.mma.cta_group::1.kind::i8 [%0], %3, %7, %9, T;\n\t"
        "@P tcgen05.mma.cta_group::1.kind::i8 [%0], %4, %8, %9, T;\n\t}"
        ::"r"(d), "l"(a), "l"(a + 2), "l"(a + 4), "l"(a + 6), "l"(b), "l"(b + 2), "l"(b + 4), "l"(b + 6), "r"(idesc), "r"(accumulate)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred P, T, A;\n\t"
        "elect.sync _|P, 0xffffffff;\n\t"
        "setp.ne.b32 A, %10, 0;\n\t"
        "setp.eq.b32 T, 0, 0;\n\t"
        "@P tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %5, %9, A;\n\t"
        "@P tcgen05.mma.cta_group::1.kind::f16 [%0], %2, %6, %9, T;\n\t"
        "@P tcgen05.mma.cta_group::1.kind::f16 [%0], %3, %7, %9, T;\n\t"
        "@P tcgen05.mma.cta_group::1.kind::f16 [%0], %4, %8, %9, T;\n\t}"
        ::"r"(d), "l"(a), "l"(a + 2), "l"(a + 4), "l"(a + 6), "l"(b), "l"(b + 2), "l"(b + 4), "l"(b + 6), "r"(idesc), "r"(accumulate)
        : "memory");
  }
}
//   block-scaled: scale bytes of the activations' plane and, where asked for, of the first factor, then the MMAs
__device__ __forceinline__ void issue_four_mx(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate, uint64_t sfa, uint64_t sfb,
                                              uint32_t copy_b, uint32_t tsfa, uint32_t tsfb) {
  asm volatile(
      "{\n\t.reg .pred P, Q, T, A;\n\t"
      "elect.sync _|P, 0xffffffff;\n\t"
      "setp.ne.and.b32 Q, %18, 0, P;\n\t"
      "setp.ne.b32 A, %13, 0;\n\t"
      "setp.eq.b32 T, 0, 0;\n\t"
      "@P tcgen05.cp.cta_group::1.32x128b.warpx4 [%14], %16;\n\t"
      "@Q tcgen05.cp.cta_group::1.32x128b.warpx4 [%15], %17;\n\t"
      "@P tcgen05.mma.cta_group::1.kind::mxf8f6f4.block_scale [%0], %1, %5, %9, [%14], [%15], A;\n\t"
      "@P tcgen05.mma.cta_group::1.kind::mxf8f6f4.block_scale [%0], %2, %6, %10, [%14], [%15], T;\n\t"
      "@P tcgen05.mma.cta_group::1.kind::mxf8f6f4.block_scale [%0], %3, %7, %11, [%14], [%15], T;\n\t"
      "@P tcgen05.mma.cta_group::1.kind::mxf8f6f4.block_scale [%0], %4, %8, %12, [%14], [%15], T;\n\t}"
      ::"r"(d), "l"(a), "l"(a + 2), "l"(a + 4), "l"(a + 6), "l"(b), "l"(b + 2), "l"(b + 4), "l"(b + 6), "r"(idesc), "r"(idesc | idesc_mx_ids(1)),
      "r"(idesc | idesc_mx_ids(2)), "r"(idesc | idesc_mx_ids(3)), "r"(accumulate), "r"(tsfa), "r"(tsfb), "l"(sfa), "l"(sfb), "r"(copy_b)
      : "memory");
}

// What bounds a narrow MMA is its A operand's way from shared memory, so tiles of up to 32 rows use MMAs of 64 (block-scaled ones have no fewer than
// 128).  Their rows lie in tensor memory sixteen to a quarter of the lanes, and the two warps of a4 reach the first two quarters.  us
// with 128 rows / 64, X in the L2: W16A16 rank 24, M x K = 1365 x 2312 8.6 / 7.5, 1 x 4608 12.0 / 10.4, 120 x 1152 5.1 / 4.7; W8A8 rank
// 32 9.1 / 8.7, 11.1 / 10.3, 5.9 / 5.7; rank 128 12.1 / 11.8, 15.0 / 14.6, 8.0 / 7.8.
__device__ __forceinline__ constexpr bool mma_64_rows(int br, int groups) { return (br == BR_INT || br == BR_F16) && groups <= 4; }

template <int MAIN, int BR>
__global__ void __launch_bounds__(NTHREADS, 1)
lq_quant_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmL1,
                const __grid_constant__ QuantParams p) {
  constexpr bool SINT = MAIN == MAIN_SINT4;
  constexpr bool MXB = BR == BR_MXFP || BR == BR_MXINT;      // the branch multiplies the main codes under their scale bytes
  extern __shared__ uint8_t qsm_raw[];
  const uint32_t base = (smem_u32(qsm_raw) + 1023u) & ~1023u;
  uint8_t* smem = qsm_raw + (base - smem_u32(qsm_raw));
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const int lane = threadIdx.x & 31;
  const int RG = p.groups, spc = p.stages, TR = 8 * RG, nq = RG * spc;       // spc: stages of K per chunk, nq: warps of a team
  const QuantSmem sm = quant_smem(BR, TR, spc, p.rn, p.bplanes, p.slots, p.xslots);
  auto bar_afull = [&](int s) { return base + (uint32_t)sm.off_bar + 8u * (uint32_t)s; };
  auto bar_bfull = [&](int s) { return bar_afull(MAX_SLOTS + s); };
  auto bar_empty = [&](int s) { return bar_afull(2 * MAX_SLOTS + s); };
  auto bar_tfull = [&](int b) { return bar_afull(3 * MAX_SLOTS + b); };
  auto bar_tempty = [&](int b) { return bar_afull(3 * MAX_SLOTS + 2 + b); };
  const uint32_t bar_sync = bar_afull(3 * MAX_SLOTS + 4);
  auto bar_xfull = [&](int s) { return bar_afull(3 * MAX_SLOTS + 5 + s); };
  auto bar_xempty = [&](int s) { return bar_afull(3 * MAX_SLOTS + 5 + MAX_XSLOTS + s); };
  int* rowmax = reinterpret_cast<int*>(smem + sm.off_max);                   // [3][64] fp16 bit patterns
  float* row_sb = reinterpret_cast<float*>(smem + sm.off_sb);                // [2][64]
  float* sl1 = reinterpret_cast<float*>(smem + sm.off_l1);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + sm.off_bar + 8 * (3 * MAX_SLOTS + 5 + 2 * MAX_XSLOTS));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.xslots; ++s) { mbar_init(bar_xfull(s), 1); mbar_init(bar_xempty(s), (uint32_t)nq); }
    if constexpr (BR != BR_NONE) {
      for (int s = 0; s < p.slots; ++s) { mbar_init(bar_afull(s), (uint32_t)nq); mbar_init(bar_bfull(s), 1); mbar_init(bar_empty(s), 1); }
      for (int b = 0; b < 2; ++b) { mbar_init(bar_tfull(b), 1); mbar_init(bar_tempty(b), 2); }
      mbar_init(bar_sync, (uint32_t)(nq * p.teams));
    }
    *abort_flag = 0;
    mbar_init_fence();
  }
  if (BR == BR_MXFP && threadIdx.x == 0) {
    SettleList* settle = reinterpret_cast<SettleList*>(smem + sm.off_l1);
    settle->entries = settle->elements = 0;
  }
  if constexpr (BR == BR_INT) {
    if (threadIdx.x < 3 * 64) rowmax[threadIdx.x] = 0;
    if (threadIdx.x >= 256 && threadIdx.x < 256 + LQ_MAX_RANK) sl1[threadIdx.x - 256] = p.sL1[threadIdx.x - 256];
  }
  if (BR != BR_NONE && warp == 2) tmem_alloc(smem_u32(tmem_slot), (uint32_t)p.tmem_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // The tensor-memory columns are taken before a dependent kernel may start and want them.
  grid_launch_dependents();

  // While the kernel before still runs, as much of this CTA's first tile as the X ring holds comes to the L2 (what that kernel writes of
  // it, it writes there).  All CTAs of a launch ask for their X at once, so the first chunk was there after 1.3 to 2.1 us instead of 0.8;
  // M = 8192, K = 1152 behind a GEMM, from the dependency wait to the end, us: SINT4 11.0 -> 9.8, MXINT4 10.2 -> 8.9, MXFP4 7.7 -> 6.5;
  // two linears of 1365 rows 34.0 -> 32.3.  (By the X producer's warp, whose loads then queue behind it: 10.6 -> 11.9 where X is in the L2 already.)
  auto fetch_ahead = [&]() {
    if (p.X != nullptr)
      for (int m = blockIdx.x * TR + lane; m < min(p.M, ((int)blockIdx.x + 1) * TR); m += 32)
        bulk_prefetch(p.X + (size_t)m * (2 * p.K), (uint32_t)min(2 * p.K, p.xslots * spc * 256));
  };
  const int qw = warp - FIRST_QWARP;
  if (warp == 3) {
    // ------------------------------------------------------------------ TMA producer: X
    const uint64_t policy = p.drop_x ? l2_evict_first() : l2_evict_normal();       // (x_leaves_first; behind the wait it cost MXFP 0.2 us a launch)
    grid_dependency_wait();
    int xs = 0;
    uint32_t par = 1, issued = 0;
    bool ok = true;
    const int walks = BR == BR_INT && p.refetch ? 2 : 1;
    for (int tile = blockIdx.x; tile < p.ntiles && ok; tile += gridDim.x)
      for (int w = 0; w < walks && ok; ++w)
        for (int c = 0; c < p.nchunks; ++c) {
          ok = mbar_wait_warp(bar_xempty(xs), par, abort_flag, p.status, LQ_STAGE_PRODUCER);
          if (!ok) break;
          if (elect_one()) {
            const int nb = 2 * min(spc, p.nst - c * spc);
            mbar_expect_tx(bar_xfull(xs), (uint32_t)(nb * TR * 128));
            for (int b = 0; b < nb; ++b)
              tma_load_2d_hint(base + (uint32_t)(xs * sm.xslot + b * TR * 128), &tmX, (2 * c * spc + b) * 128, tile * TR, bar_xfull(xs), policy);
          }
          __syncwarp();
          ++issued;
          if (++xs == p.xslots) { xs = 0; par ^= 1; }
        }
    if (!ok && lane == 0)      // aborting: the copies in flight get a bounded time to land
      for (uint32_t i = min(issued, (uint32_t)p.xslots); i > 0; --i) {
        if (--xs < 0) { xs = p.xslots - 1; par ^= 1; }
        mbar_settle(bar_xfull(xs), par ^ 1);
      }
  } else if (BR != BR_NONE && warp == 4) {
    // ------------------------------------------------------------------ TMA producer: the first factor (weights: no earlier
    // kernel has to be waited for)
    int slot = 0;
    uint32_t par = 1, issued = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < p.ntiles && ok; tile += gridDim.x)
      for (int c = 0; c < p.nchunks; ++c) {
        ok = mbar_wait_warp(bar_empty(slot), par, abort_flag, p.status, LQ_STAGE_PRODUCER);
        if (!ok) break;
        const int st0 = c * spc, ns = min(spc, p.nst - st0);
        const uint32_t dst = base + (uint32_t)(sm.off_slots + slot * sm.slot), full = bar_bfull(slot);
        if (elect_one()) {
          mbar_expect_tx(full, (uint32_t)(ns * sm.b_ps * (sm.b_unit + (MXB ? 512 : 0))));
          for (int s = 0; s < ns; ++s)
            for (int u = 0; u < sm.b_ps; ++u) {
              const int i = s * sm.b_ps + u;                     // fp16: a stage's 256 bytes of K in two slabs
              tma_load_2d(dst + sm.off_b + i * sm.b_unit, &tmL1, (BR == BR_F16 ? 2 * (st0 + s) + u : st0 + s) * 128, 0, full);
              if constexpr (MXB) bulk_load(dst + sm.off_sfb + i * 512, p.sfl1 + (size_t)(st0 + s) * 512, 512, full);
            }
        }
        __syncwarp();
        ++issued;
        if (++slot == p.slots) { slot = 0; par ^= 1; }
      }
    if (!ok && lane == 0)      // aborting: the copies in flight get a bounded time to land
      for (uint32_t i = min(issued, (uint32_t)p.slots); i > 0; --i) {
        if (--slot < 0) { slot = p.slots - 1; par ^= 1; }
        mbar_settle(bar_bfull(slot), par ^ 1);
      }
  } else if (BR != BR_NONE && warp == 2) {
    // ------------------------------------------------------------------ MMA issuer
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    const int cols = p.rn * p.bplanes;
    const uint32_t shape = idesc_shape(cols) - (mma_64_rows(BR, RG) ? (uint32_t)(64 >> 4) << 24 : 0u), tsf = tmem + (uint32_t)(p.sets * p.nacc * cols);
    bool ok = true;
    uint32_t tc = 0, par = 0;
    int slot = 0;
    for (int tile = blockIdx.x; tile < p.ntiles && ok; tile += gridDim.x, ++tc) {
      const uint32_t set = tmem + (uint32_t)((tc & (p.sets - 1)) * p.nacc * cols);
      ok = mbar_wait_warp(bar_tempty(tc & 1), ((tc >> 1) & 1) ^ 1, abort_flag, p.status, LQ_STAGE_MMA);
      for (int c = 0; c < p.nchunks && ok; ++c) {
        const int ns = min(spc, p.nst - c * spc);
        ok = mbar_wait_warp(bar_bfull(slot), par, abort_flag, p.status, LQ_STAGE_MMA) &&
             mbar_wait_warp(bar_afull(slot), par, abort_flag, p.status, LQ_STAGE_MMA);
        if (!ok) break;
        tc_fence_after();
        const uint32_t at = base + (uint32_t)(sm.off_slots + slot * sm.slot);
#pragma unroll 1
        for (int s = 0; s < ns; ++s) {
          const int gs = c * spc + s;                            // stage of K: the accumulators take turns
          const uint32_t d = set + (uint32_t)((gs & (p.nacc - 1)) * cols), more = gs >= p.nacc;
          const uint32_t a = at + s * sm.a_ps * sm.a_unit, bw = at + sm.off_b + s * sm.b_ps * sm.b_unit;
          if constexpr (BR == BR_INT) {
            issue_four<TC_I8>(d, make_smem_desc(a), make_smem_desc(bw), IDESC_I8 | shape, more);
          } else if constexpr (BR == BR_F16) {
            issue_four<TC_F16>(d, make_smem_desc(a), make_smem_desc(bw), IDESC_F16 | shape, more);
            issue_four<TC_F16>(d, make_smem_desc(a + sm.a_unit), make_smem_desc(bw + sm.b_unit), IDESC_F16 | shape, 1u);
          } else {
            // scale bytes into tensor memory (one slot: the tensor pipe executes these copies and MMAs in issue order), the
            // activations' digit planes one after the other
            constexpr int ap = BR == BR_MXINT ? 2 : 1;
            const uint64_t sfb = make_smem_desc_plain(at + sm.off_sfb + s * 512, 16, 128);
#pragma unroll
            for (int u = 0; u < ap; ++u)
              issue_four_mx(d, make_smem_desc(a + u * sm.a_unit), make_smem_desc(bw), idesc_mx(cols, 0), more | (uint32_t)u,
                            make_smem_desc_plain(at + sm.off_sfa + (s * ap + u) * 512, 16, 128), sfb, (uint32_t)(u == 0), tsf + 4 * u, tsf + 8);
          }
        }
        if (elect_one()) {
          tc_commit(bar_empty(slot));
          if (c + 1 == p.nchunks) tc_commit(bar_tfull(tc & 1));
        }
        __syncwarp();
        if (++slot == p.slots) { slot = 0; par ^= 1; }
      }
    }
  } else if (BR != BR_NONE && warp < 2) {
    // ------------------------------------------------------------------ a4: lane = row of the tile, straight from tensor memory
    // One warp's chain of instructions at the end of a launch, a microsecond or two long: 32 columns at a time, two values to an
    // instruction, a rank of up to 32 read once.  (Sixteen at a time, one by one, the scaled sums worked out for the maximum and again
    // for the codes: us, M = 1 / 8192, K = 1152, X in the L2, SINT4 rank 32 6.5 / 11.1 -> 5.9 / 10.7, MXFP8 rank 64 6.2 / 9.3 -> 5.5 /
    // 8.5, MXFP4 rank 128 7.7 / 11.6 -> 6.6 / 10.3, MXINT8 rank 64 7.5 / 11.2 -> 6.9 / 10.5.)
    if (warp == 0) fetch_ahead();
    grid_dependency_wait();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0) + ((uint32_t)(32 * warp) << 16);
    const bool low = mma_64_rows(BR, RG);                // sixteen rows to a warp
    const int nacc = min(p.nacc, p.nst), row0 = (low ? 16 : 32) * warp, row = low && lane >= 16 ? TR : row0 + lane;
    uint32_t tc = 0;
    SettleList* const settle = reinterpret_cast<SettleList*>(smem + sm.off_l1);
    for (int tile = blockIdx.x; tile < p.ntiles; tile += gridDim.x, ++tc) {
      const int m = tile * TR + row;
      const bool valid = row < TR && m < p.M;
      const uint32_t set = tmem + (uint32_t)((tc & (p.sets - 1)) * p.nacc * p.rn * p.bplanes);
      if (!mbar_wait_warp(bar_tfull(tc & 1), (tc >> 1) & 1, abort_flag, p.status, LQ_STAGE_DRAIN)) break;
      tc_fence_after();
      uint8_t* const tqr = p.tq + (size_t)m * p.tq_stride;
      if (row0 < TR) {
        // 32 columns of the row from `col` on (zeros beyond the rank): the sum over the accumulators (and the first factor's digit planes)
        auto fetch = [&](int col, float (&t)[32]) {
          const bool both = col + 16 < p.rn;
          auto load = [&](int a, uint32_t (&v)[2][16]) {
            const uint32_t at = set + (uint32_t)(a * p.rn + col);
            tmem_ld_32x16(at, v[0]);
            if (both) tmem_ld_32x16(at + 16, v[1]);
            tmem_ld_wait();
          };
          uint32_t v[2][16];
          load(0, v);
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const uint32_t w = j < 16 || both ? v[j >> 4][j & 15] : 0u;
            t[j] = BR == BR_INT ? __int2float_rn((int)w) : __uint_as_float(w);
          }
          if constexpr (BR != BR_INT) {
#pragma unroll 1
            for (int a = 1; a < nacc * p.bplanes; ++a) {
              load(a, v);
#pragma unroll
              for (int j = 0; j < 32; ++j)
                if (j < 16 || both) t[j] += __uint_as_float(v[j >> 4][j & 15]);
            }
          }
        };
        auto pair = [](const float (&t)[32], int i) { return make_float2(t[2 * i], t[2 * i + 1]); };
        auto largest = [](const float (&t)[32]) {                // of the magnitudes
          float m[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int j = 0; j < 32; ++j) m[j & 3] = fmaxf(m[j & 3], fabsf(t[j]));
          return fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
        };
        float t[32];
        if constexpr (BR == BR_INT) {
          const float sr = row_sb[(tc & 1) * 64 + row];
          auto scaled = [&](int c) {                           // t = fl32(fl32(I1) fl32(sXb sL1)); rows beyond the tile hold anything
            fetch(c, t);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float4 s = *reinterpret_cast<const float4*>(__builtin_assume_aligned(sl1 + c + 4 * i, 16));
              const float2 u = __fmul2_rn(pair(t, 2 * i), __fmul2_rn(splat(sr), make_float2(s.x, s.y)));
              const float2 w = __fmul2_rn(pair(t, 2 * i + 1), __fmul2_rn(splat(sr), make_float2(s.z, s.w)));
              t[4 * i] = u.x; t[4 * i + 1] = u.y; t[4 * i + 2] = w.x; t[4 * i + 3] = w.y;
            }
          };
          float amax = 0.f;
#pragma unroll 1
          for (int c = 0; c < p.rn; c += 32) {
            scaled(c);
            amax = fmaxf(amax, largest(t));
          }
          const float st = amax == 0.f ? 1.f : __fdiv_rn(amax, p.qm);
          if (valid) p.sT[SINT ? lq_row_slot(m) : m] = st;
          // The correctly rounded quotient t / st as in branch_codes8_exact.  A power of two keeps its steps in binary32's normal range; the quotient
          // stays what it is (what underflows is far below half a code).
          const float k = st < 1e-20f ? 0x1p64f : st > 1e20f ? 0x1p-64f : 1.f;
          const float2 ns = splat(-st * k), y = splat(__frcp_rn(st * k));
          const bool coarse = st < 0x1p-126f;                  // a subnormal scale: amax / st may be up to half again as large as qm
#pragma unroll 1
          for (int c = 0; c < p.rn; c += 32) {
            if (p.rn > 32) scaled(c);                          // (up to 32 columns are still there)
            uint32_t w[8];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float2 x = __fmul2_rn(pair(t, i), splat(k)), q0 = __fmul2_rn(x, y);
              float2 q = __ffma2_rn(__ffma2_rn(q0, ns, x), y, q0);
              if (coarse) q = make_float2(fminf(fmaxf(q.x, -p.qm), p.qm), fminf(fmaxf(q.y, -p.qm), p.qm));
              q = __fadd2_rn(q, splat(MAGIC));
              const uint32_t two = __byte_perm(__float_as_uint(q.x), __float_as_uint(q.y), 0x0040);
              w[i >> 1] = (i & 1) == 0 ? two : __byte_perm(w[i >> 1], two, 0x5410);
            }
            // (a rank of 16 more than a multiple of 32: zeros up to there, where the up-projection's K ends)
            if (valid) {
              *reinterpret_cast<uint4*>(tqr + c) = make_uint4(w[0], w[1], w[2], w[3]);
              *reinterpret_cast<uint4*>(tqr + c + 16) = c + 16 < p.rn ? make_uint4(w[4], w[5], w[6], w[7]) : make_uint4(0, 0, 0, 0);
            }
          }
        } else if constexpr (BR == BR_F16) {
          if (valid) p.sT[SINT ? lq_row_slot(m) : m] = 1.f;
#pragma unroll 1
          for (int c = 0; c < p.rn; c += 32) {
            fetch(c, t);
            uint32_t w[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) w[j] = as_u32(__floats2half2_rn(t[2 * j], t[2 * j + 1]));
            if (valid) {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (j < 2 || c + 16 < p.rn) *reinterpret_cast<uint4*>(tqr + 2 * c + 16 * j) = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
            }
          }
        } else {
          // blocks of 32 along the rank
          constexpr bool FPB = BR == BR_MXFP, SIX = MAIN == MAIN_MXFP6;
          // MXINT with one container for both planes (rank <= 64): lo digits 64 bytes after the hi digits, scale slots c and
          // 2 + c of one chunk; a container per plane: 128 bytes on, slot c of the next chunk
          const bool sep = p.tq_stride != LQ_RCONT;
          uint8_t* const sf = p.sft + (size_t)(m >> 7) * (!FPB && sep ? 1024 : 512) + 16 * (m & 31) + 4 * ((m & 127) >> 5);
          [[maybe_unused]] uint32_t near = 0;                    // MXFP: the row's blocks to be settled at the end
#pragma unroll 1
          for (int b = 0; 32 * b < p.rn; ++b) {
            fetch(32 * b, t);
            const float amax = largest(t);
            const int e = FPB ? mxfp_exponent<SIX>(amax * p.unit) : mxint8_exponent(amax * p.unit);
            const float inv = e == -127 ? 0.f : pow2f_n(-e) * p.unit;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              uint32_t w[4], d[4];
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const float2 x0 = pair(t, 8 * h + 2 * j), x1 = pair(t, 8 * h + 2 * j + 1);
                if constexpr (!FPB) {
                  float2 hi0, lo0, hi1, lo1;
                  mxint8_digits(x0, inv, hi0, lo0);
                  mxint8_digits(x1, inv, hi1, lo1);
                  w[j] = f32x2_to_e4m3x2(hi0.y, hi0.x) | (f32x2_to_e4m3x2(hi1.y, hi1.x) << 16);
                  d[j] = f32x2_to_e4m3x2(lo0.y, lo0.x) | (f32x2_to_e4m3x2(lo1.y, lo1.x) << 16);
                } else {
                  const float2 y0 = __fmul2_rn(x0, splat(inv)), y1 = __fmul2_rn(x1, splat(inv));
                  w[j] = mxfp_pair<SIX>(y0.y, y0.x) | (mxfp_pair<SIX>(y1.y, y1.x) << 16);
                  d[j] = 0;
                }
              }
              if (valid) {
                *reinterpret_cast<uint4*>(tqr + 32 * b + 16 * h) = make_uint4(w[0], w[1], w[2], w[3]);
                if (!FPB) *reinterpret_cast<uint4*>(tqr + (sep ? 128 : 64) + 32 * b + 16 * h) = make_uint4(d[0], d[1], d[2], d[3]);
              }
            }
            if (valid) {
              sf[b] = (uint8_t)(e + 127 + (FPB ? 0 : 4));
              if (!FPB) sf[(sep ? 512 : 2) + b] = (uint8_t)(e + 127);
            }
            if constexpr (FPB) {
              const float dev = amax * p.dev;
              const TieTest<SIX> tie(inv, dev);
              const bool edge = ((__float_as_uint(amax + dev) ^ __float_as_uint(amax - dev)) >> 23) != 0;
              // (any binade at first: few lanes go on to ask which elements)
              if ((edge || tie.any(t)) && valid) {
                uint32_t which = 0;
#pragma unroll
                for (int j = 0; j < 32; ++j) which |= tie(t[j]) ? 1u << j : 0u;
                if (edge) which = 0xFFFFFFFFu;
                if (which != 0) {
                  near |= 1u << b;
                  p.near_which[4 * (size_t)m + b] = which;
                  atomicAdd(&settle->elements, __popc(which));
                  const int n = atomicAdd(&settle->entries, 1);
                  if (n < SETTLE_ENTRIES) settle->entry[n] = make_int4(m, b, (int)which, e);
                }
              }
            }
          }
          if (FPB && valid) p.near[m] = near;
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_tempty(tc & 1));
    }
  } else if (BR == BR_NONE && warp == 0) {
    fetch_ahead();
  } else if (warp >= FIRST_QWARP && qw < nq * p.teams) {
    // ------------------------------------------------------------------ quantizer
    // This lane: 16 neighbouring values (a piece pair pp of a box) of rows ra and ra + 2 of the tile.  They share a block, so its scale
    // is worked out once, and their codes are one 16-byte vector of a row.  The two rows that eight lanes in a row read or write
    // together differ in bits 0 and 2: even pieces of X and the four pieces of an operand slab's half fall in different banks.
    const int team = qw / nq, rg = (qw - team * nq) % RG, sx = (qw - team * nq) / RG, pp = lane & 3, box = (lane >> 3) & 1;
    const int ra = 8 * rg + (((lane >> 2) & 1) * 5 ^ (lane >> 4));
    const uint32_t sw = (uint32_t)(ra & 7);
    // X: the pair's first piece (the second is at the address with bit 4 flipped), a box is TR rows of 128 bytes
    const uint32_t xo = base + (uint32_t)(sx * TR * 256 + box * TR * 128 + ra * 128);
    const uint32_t xo_a = xo + (((2 * pp) ^ sw) << 4), xo_b = xo + 256 + (((2 * pp) ^ sw ^ 2) << 4);
    // this lane's 16 codes in an operand slab (rows of 128 bytes, 16-byte pieces exchanged by row mod 8)
    const uint32_t ao = base + (uint32_t)(sm.off_slots + sx * sm.a_ps * sm.a_unit + ra * 128);
    const uint32_t ao_a = ao + (((4 * box + pp) ^ sw) << 4), ao_b = ao + 256 + (((4 * box + pp) ^ sw ^ 2) << 4);
    const int sr = ra + 2 * box;                                                        // the row whose scale bytes (maximum, scale) this lane has where
    const bool first = pp == 0;                                                         // it is its box's first
    const uint32_t so = base + (uint32_t)(sm.off_slots + sm.off_sfa + sx * sm.a_ps * 512 + 16 * (sr & 31) + 4 * (sr >> 5));
    const size_t qs = MAIN == MAIN_MXINT8 ? (size_t)2 * p.Kpad : (size_t)p.Kpad;        // bytes per row of qx8
    grid_dependency_wait();        // from here on the activation record is written
    Ring xr{0, 0u}, er{0, 1u};     // X slot and operand slot of the current tile's (walk's) first chunk
    uint32_t tc = 0, buf = 0;
    int c0 = team;                 // this team's first chunk of the tile: chunks go round the teams without regard to tiles
    bool ok = true;
    for (int tile = blockIdx.x; tile < p.ntiles && ok; tile += gridDim.x, ++tc) {
      const int ma = tile * TR + ra, ms = tile * TR + sr;
      const bool va = ma < p.M, vb = ma + 2 < p.M, vs = first && ms < p.M;
      uint8_t* const qa = p.qx8 + (size_t)ma * qs + sx * 128 + 64 * box + 16 * pp;
      uint8_t* const sfr = SINT ? nullptr : p.sfa + ((size_t)(ms >> 7) * (qs >> 7) + sx) * 512 + 16 * (ms & 31) + 4 * ((ms & 127) >> 5);
      float sb_a = 1.f, sb_b = 1.f, inv_a = 1.f, inv_b = 1.f;     // integer branch: scales of rows ra, ra + 2
      bool exact = false;                                        // (of any of the warp's rows)
      __half2 hm = __float2half2_rn(0.f);                        // maxima of rows ra, ra + 2
      // One walk over the tile.  MAINP: main codes and scales; BRP: the branch's operand; FREE: the X slots are handed back.
      auto walk = [&](auto MAINP, auto BRP, const bool free_x) {
        Ring x = xr, e = er;
        x.step(c0, p.xslots);
        e.step(c0, p.slots);
        for (int c = c0, st = c0 * spc + sx; c < p.nchunks; c += p.teams, st += p.teams * spc) {
          const bool live = st < p.nst;
          if (!mbar_wait_warp(bar_xfull(x.at), x.par, abort_flag, p.status, LQ_STAGE_QUANT)) return false;
          uint4 a[2], b[2];
          if (live) {
            const uint32_t at = (uint32_t)(x.at * sm.xslot);
            a[0] = lds_v4(xo_a + at); b[0] = lds_v4(xo_b + at);
            a[1] = lds_v4((xo_a + at) ^ 16); b[1] = lds_v4((xo_b + at) ^ 16);
          }
          uint2 wa[2], wb[2], da[2], db[2];                      // main codes of the two rows (MXINT8: hi digits; d: lo digits)
          uint32_t four = 0;                                     // the stage's scale bytes of row sr (a box's first lane has them)
          if constexpr (decltype(MAINP)::value) {
            if (live) {
              __half2 bm = __halves2half2(__hmax(absmax8(a[0]), absmax8(a[1])), __hmax(absmax8(b[0]), absmax8(b[1])));
              bm = __hmax2(bm, __shfl_xor_sync(0xffffffffu, bm, 1));
              if constexpr (SINT) bm = __hmax2(bm, __shfl_xor_sync(0xffffffffu, bm, 2));
              if constexpr (BR == BR_INT) hm = __hmax2(hm, bm);
              if constexpr (SINT) {
                const Sint4Scale sc(bm);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  wa[h] = sint4_codes8(a[h], sc.inv[0], sc.coarse); wb[h] = sint4_codes8(b[h], sc.inv[1], sc.coarse);
                }
                // (of a padding group, too)
                if (pp < 2 && ma + 2 * pp < p.M) p.sx[(size_t)(2 * st + box) * p.Mpad + lq_row_slot(ma + 2 * pp)] = pp ? sc.s[1] : sc.s[0];
              } else {
                constexpr int TOP = MAIN == MAIN_MXINT4 ? 2 : MAIN == MAIN_MXINT8 ? 6 : 8;
                constexpr int UP = MAIN == MAIN_MXINT4 ? 0xFF : MAIN == MAIN_MXINT8 ? 0x0F : 0;
                const PairScale<TOP, UP> ps(as_u32(bm));
                uint32_t own = ps.bytes;                         // this block's bytes: row ra's and, 16 bits on, row ra + 2's
                if (MAIN != MAIN_MXFP6 && ps.ok) {
                  const __half2 i0 = as_half2(__byte_perm(ps.inv, 0, 0x1010)), i1 = as_half2(__byte_perm(ps.inv, 0, 0x3232));
#pragma unroll
                  for (int h = 0; h < 2; ++h) {
                    if constexpr (MAIN == MAIN_MXFP) { wa[h] = mxfp8_codes8(a[h], i0); wb[h] = mxfp8_codes8(b[h], i1); }
                    else if constexpr (MAIN == MAIN_MXINT4) { wa[h] = mxint4_codes8(a[h], i0); wb[h] = mxint4_codes8(b[h], i1); }
                    else if constexpr (MAIN == MAIN_MXINT8) { mxint8_codes8(a[h], i0, wa[h], da[h]); mxint8_codes8(b[h], i1, wb[h], db[h]); }
                  }
                } else {
#pragma unroll
                  for (int h = 0; h < 2; ++h) {
                    const RareCodes rc = rare_codes<MAIN>(a[h], b[h], bm);
                    wa[h] = rc.wa; wb[h] = rc.wb; da[h] = rc.da; db[h] = rc.db;
                    own = rc.bytes;
                  }
                }
                // a row's four bytes are with four lanes: the box's two blocks, then the boxes; box 0 collects row ra's, box 1 row ra + 2's
                const uint32_t next = __shfl_xor_sync(0xffffffffu, own, 2);
                const uint32_t both = __byte_perm(pp & 2 ? next : own, pp & 2 ? own : next, 0x6240);
                const uint32_t other = __shfl_xor_sync(0xffffffffu, both, 8);
                four = box ? __byte_perm(other, both, 0x7632) : __byte_perm(both, other, 0x5410);
                if (vs) {
                  uint8_t* sf = sfr + (size_t)c * spc * 512;     // (the hi digits weigh 16 times as much)
                  *reinterpret_cast<uint32_t*>(sf) = MAIN == MAIN_MXINT8 ? four + 0x04040404u : four;
                  if (MAIN == MAIN_MXINT8) *reinterpret_cast<uint32_t*>(sf + (size_t)p.nst * 512) = four;
                }
              }
              uint8_t* const q = qa + c * spc * 128;
              if (va) {
                *reinterpret_cast<uint4*>(q) = vec16(wa);
                if (MAIN == MAIN_MXINT8) *reinterpret_cast<uint4*>(q + p.Kpad) = vec16(da);
              }
              if (vb) {
                *reinterpret_cast<uint4*>(q + 2 * qs) = vec16(wb);
                if (MAIN == MAIN_MXINT8) *reinterpret_cast<uint4*>(q + 2 * qs + p.Kpad) = vec16(db);
              }
            }
          }
          if constexpr (decltype(BRP)::value) {
            [[maybe_unused]] uint2 ca[2], cb[2];
            if constexpr (BR == BR_INT) {
              if (live && !exact) {
#pragma unroll
                for (int h = 0; h < 2; ++h) { ca[h] = branch_codes8(a[h], inv_a); cb[h] = branch_codes8(b[h], inv_b); }
              } else if (live) {
#pragma unroll
                for (int h = 0; h < 2; ++h) { ca[h] = branch_codes8_exact(a[h], sb_a, inv_a); cb[h] = branch_codes8_exact(b[h], sb_b, inv_b); }
              }
            }
            if (!mbar_wait_warp(bar_empty(e.at), e.par, abort_flag, p.status, LQ_STAGE_QUANT)) return false;
            const uint32_t at = (uint32_t)(e.at * sm.slot);
            if (live) {
              if constexpr (BR == BR_INT) {
                sts_v4(ao_a + at, vec16(ca));
                sts_v4(ao_b + at, vec16(cb));
                if (p.qb != nullptr) {
                  int8_t* o = p.qb + (qa - p.qx8) + c * spc * 128;
                  if (va) *reinterpret_cast<uint4*>(o) = vec16(ca);
                  if (vb) *reinterpret_cast<uint4*>(o + 2 * qs) = vec16(cb);
                }
              } else if constexpr (BR == BR_F16) {               // a slab per box: 64 halves, laid out as in the X ring
                const uint32_t to = (uint32_t)sm.off_slots + at;
                sts_v4(xo_a + to, a[0]); sts_v4((xo_a + to) ^ 16, a[1]);
                sts_v4(xo_b + to, b[0]); sts_v4((xo_b + to) ^ 16, b[1]);
              } else {
                sts_v4(ao_a + at, vec16(wa));
                sts_v4(ao_b + at, vec16(wb));
                if constexpr (BR == BR_MXINT) {
                  sts_v4(ao_a + at + sm.a_unit, vec16(da));
                  sts_v4(ao_b + at + sm.a_unit, vec16(db));
                }
              }
              if (MXB && first) {
                sts_u32(so + at, BR == BR_MXINT ? four + 0x04040404u : four);
                if (BR == BR_MXINT) sts_u32(so + at + 512, four);
              }
            }
            fence_proxy_async();
          }
          // The X slot goes back only here: by now the stores above have been issued, and they needed every value that was
          // loaded from it.  (An arrival right after the loads can overtake them: a load may still sit in its queue when the
          // slot is refilled.)
          __syncwarp();
          if (lane == 0) {
            if (decltype(BRP)::value) mbar_arrive(bar_afull(e.at));
            if (free_x) mbar_arrive(bar_xempty(x.at));
          }
          x.step(p.teams, p.xslots);
          e.step(p.teams, p.slots);
        }
        if (free_x) xr.step(p.nchunks, p.xslots);                // (kept slots are walked again)
        if (decltype(BRP)::value) er.step(p.nchunks, p.slots);
        return true;
      };
      using Yes = std::true_type;
      using No = std::false_type;
      if constexpr (BR == BR_INT) {
        ok = walk(Yes(), No(), p.refetch != 0);
        if (!ok) break;
        // ---- the rows' maxima and scales: non-negative halves order like their bit patterns
        if constexpr (!SINT) hm = __hmax2(hm, __shfl_xor_sync(0xffffffffu, hm, 2));
        hm = __hmax2(hm, __shfl_xor_sync(0xffffffffu, hm, 8));
        int* mx = rowmax + buf * 64;
        if (first) atomicMax(&mx[sr], (int)__half_as_ushort(box ? __high2half(hm) : __low2half(hm)));
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_sync);
        ok = mbar_wait_warp(bar_sync, tc & 1, abort_flag, p.status, LQ_STAGE_QUANT);
        if (!ok) break;
        // eight lanes have the same two rows: one half works out row ra's scale, the other row ra + 2's
        const BranchScale mine((uint32_t)mx[sr], p.qm, p.rqm, p.near_tie);
        {
          exact = __any_sync(0xffffffffu, mine.exact);
          const float own = exact ? __frcp_rn(mine.sb) : mine.inv;
          const float sb = __shfl_xor_sync(0xffffffffu, mine.sb, 8), inv = __shfl_xor_sync(0xffffffffu, own, 8);
          sb_a = box ? sb : mine.sb; sb_b = box ? mine.sb : sb;
          inv_a = box ? inv : own; inv_b = box ? own : inv;
        }
        const uint32_t after = buf == 0 ? 2 : buf - 1;           // two tiles on: every warp is past its last use
        if (team == 0 && sx == 0 && first) rowmax[after * 64 + sr] = 0;
        buf = buf == 2 ? 0 : buf + 1;
        if (team == 0 && sx == 0) {                              // a4 reads the scale: its previous tile of this parity must be done
          ok = mbar_wait_warp(bar_tempty(tc & 1), ((tc >> 1) & 1) ^ 1, abort_flag, p.status, LQ_STAGE_QUANT);
          if (!ok) break;
          if (first) row_sb[(tc & 1) * 64 + sr] = mine.sb;
          if (vs) p.sXb[ms] = mine.sb;
        }
        ok = walk(No(), Yes(), true);
      } else {
        ok = walk(Yes(), std::integral_constant<bool, BR != BR_NONE>(), true);
      }
      c0 = (c0 + p.teams - p.nchunks % p.teams) % p.teams;
    }
  }

  tc_fence_before();
  __syncthreads();
  if constexpr (BR == BR_MXFP) {
    SettleList& list = *reinterpret_cast<SettleList*>(smem + sm.off_l1);
    float* part = reinterpret_cast<float*>(smem);
    if (list.elements != 0 && !*abort_flag) {
      if (list.elements <= settle_few(p.K)) settle_elements<MAIN == MAIN_MXFP6>(p, part, list);
      else settle_tiles<MAIN == MAIN_MXFP6>(p, part, list);
    }
  }
  if (BR != BR_NONE && warp == 2) {
    tc_fence_after();
    tmem_dealloc(__shfl_sync(0xffffffffu, *tmem_slot, 0), (uint32_t)p.tmem_cols);
  }
}

// The launch's cut.  Working it out takes the calling thread 0.5 to 1.5 us of a launch's 4 to 5, which back-to-back calls of a few rows
// wait for, so each thread keeps the last ones by everything that they depend on (a call of one row, K = 1152: 4.3 -> 3.8 us).
bool cut_of(int br, int M, int nst, int rn, int bplanes, int sms, QuantCut& out) {
  struct Kept { int key[8]; QuantCut cut; };
  static thread_local Kept kept[16];                             // (a key's M is not 0)
  const int key[8] = {br, M, nst, rn, bplanes, sms, g_lq_quant_warps, g_lq_quant_ctas};
  Kept& k = kept[((uint32_t)M * 0x9E3779B1u ^ (uint32_t)nst * 0x85EBCA6Bu ^ (uint32_t)(rn + br) * 0xC2B2AE35u) >> 28];
  if (!std::equal(key, key + 8, k.key)) {
    QuantCut c{};
    if (!plan_cut_as_asked(br, M, nst, rn, bplanes, sms, key[6], key[7], c)) return false;
    std::copy(key, key + 8, k.key);
    k.cut = c;
  }
  out = k.cut;
  return true;
}

template <int MAIN, int BR>
cudaError_t launch_quant(const void* X, const CUtensorMap& tm, QuantParams& p, int sms, cudaStream_t st) {
  static std::atomic<bool> attr_set[64];   // (set by several threads at once it does no harm)
  int dev = 0;
  cudaGetDevice(&dev);
  if (!attr_set[dev & 63]) {
    const cudaError_t e = cudaFuncSetAttribute(lq_quant_kernel<MAIN, BR>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return e;
    attr_set[dev & 63] = true;
  }
  if (!cut_of(BR, p.M, p.nst, p.rn, p.bplanes, sms, p)) return cudaErrorInvalidConfiguration;
  p.drop_x = x_leaves_first(p, MAIN == MAIN_MXINT8, (double)p.M * (2.0 * p.K + p.Kpad));
  // From 1 MB of X on: less comes in one trip anyway.
  p.X = (size_t)p.M * p.K * 2 >= (1u << 20) ? static_cast<const uint8_t*>(X) : nullptr;
  // Floating-point branches: a tile's stages alternate over up to four accumulators, which are added in fp32 at the end
  // (each costs a4 a trip to tensor memory per 32 columns: not more than 128 columns of them).  Tensor memory holds two
  // such sets - one where every CTA has a single tile - and the scale bytes' columns.
  const int cols = p.rn * p.bplanes, extra = BR == BR_MXFP || BR == BR_MXINT ? 16 : 0;
  p.sets = p.ntiles <= sms ? 1 : 2;
  p.nacc = BR == BR_INT ? 1 : BR == BR_F16 || cols <= 32 ? 4 : cols <= 64 ? 2 : 1;
  p.tmem_cols = 32;
  while (p.tmem_cols < p.sets * p.nacc * cols + extra) p.tmem_cols *= 2;
  // what the chains of fp32 sums and the bits of the products make of that deviation
  p.dev *= (0.3f + (float)p.K / (1000.f * p.nacc)) * 0x1p-22f;
  CUtensorMap tmX;
  if (lq_make_tmap_bytes(&tmX, const_cast<void*>(X), (uint64_t)p.M, (uint64_t)p.K * 2, (uint32_t)(8 * p.groups)) != LQ_OK)
    return cudaErrorInvalidValue;
  const cudaError_t e = lq_launch(lq_quant_kernel<MAIN, BR>, std::min(p.ntiles, sms), NTHREADS, (size_t)p.smem, st, tmX, tm, p);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

lq_status lq_launch_quantize(const lq_layer* L, const void* X, int M, lq_act* A, cudaStream_t st) {
  if (cudaSetDevice(A->device) != cudaSuccess) return LQ_ERR_CUDA;
  if (A->main_kind != LQ_KIND_E4M3) return LQ_ERR_UNSUPPORTED;
  const int abits = lq_branch_abits(L->cfg.branch);
  QuantParams p;
  p.M = M; p.K = L->K; p.Kpad = L->Kpad; p.Mpad = A->Mpad;
  p.nst = L->Kpad / LQ_KSTAGE;
  p.qx8 = A->d_qx8; p.sx = A->d_sx; p.sfa = A->d_sfa;
  p.qb = g_lq_store_qb ? A->d_qb : nullptr;
  p.sXb = A->d_sXb; p.sL1 = L->d_sL1; p.l1c = L->d_L1c; p.sfl1 = L->d_sfl1;
  p.sft = A->d_sft; p.tq = A->d_tq; p.sT = A->d_sT; 
  // (an MXFP row has neither a scale nor branch codes of its own)
  p.near = reinterpret_cast<uint32_t*>(A->d_sT); p.near_which = reinterpret_cast<uint32_t*>(A->d_qb);
  p.r = L->r; p.rn = lq_l1_rows(L);
  p.bplanes = lq_l1_planes(L);
  p.tq_stride = A->tq_stride;
  p.dev = L->cfg.branch == LQ_BRANCH_MXFP8 ? 1.f : L->cfg.branch == LQ_BRANCH_MXFP6 ? 0.5f : 0.2f;
  p.unit = ldexpf(1.f, -L->l1_shift);
  p.qm = abits > 0 ? (float)((1 << (abits - 1)) - 1) : 0.f;
  p.rqm = 1.f / p.qm;
  p.near_tie = abits > 0 ? ldexpf(1.f, abits - 27) : 0.f;
  p.status = lq_device_status_ptr(A->device);
  if (!p.status) return LQ_ERR_CUDA;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, A->device) != cudaSuccess) return LQ_ERR_CUDA;
  cudaError_t e;
  if (L->mxfp && L->cfg.act_fmt == LQ_ACT_MXFP6)
    e = L->r > 0 ? launch_quant<MAIN_MXFP6, BR_MXFP>(X, L->tmL1, p, sms, st) : launch_quant<MAIN_MXFP6, BR_NONE>(X, L->tmL1, p, sms, st);
  else if (L->mxfp) e = L->r > 0 ? launch_quant<MAIN_MXFP, BR_MXFP>(X, L->tmL1, p, sms, st) : launch_quant<MAIN_MXFP, BR_NONE>(X, L->tmL1, p, sms, st);
  else if (L->a8) e = L->r > 0 ? launch_quant<MAIN_MXINT8, BR_MXINT>(X, L->tmL1, p, sms, st) : launch_quant<MAIN_MXINT8, BR_NONE>(X, L->tmL1, p, sms, st);
  else if (L->mx)
    e = L->f16_branch ? launch_quant<MAIN_MXINT4, BR_F16>(X, L->tmL1, p, sms, st)
                      : L->integer_branch ? launch_quant<MAIN_MXINT4, BR_INT>(X, L->tmL1, p, sms, st)
                                          : launch_quant<MAIN_MXINT4, BR_NONE>(X, L->tmL1, p, sms, st);
  else
    e = L->f16_branch ? launch_quant<MAIN_SINT4, BR_F16>(X, L->tmL1, p, sms, st)
                      : L->integer_branch ? launch_quant<MAIN_SINT4, BR_INT>(X, L->tmL1, p, sms, st)
                                          : launch_quant<MAIN_SINT4, BR_NONE>(X, L->tmL1, p, sms, st);
  return lq_note_cuda(e) == cudaSuccess ? LQ_OK : LQ_ERR_CUDA;
}
