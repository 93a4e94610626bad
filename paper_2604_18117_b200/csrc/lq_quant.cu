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
//   warps 4-19  quantizer: in a chunk each warp has one piece, 8 rows x one stage.  Eight lanes own 64 values of a row, a
//               16-byte vector each, and every lane has vectors of two rows: a block of 32 is four lanes, its maximum two
//               shuffles, and loads, stores and shared-memory accesses all move whole rows of a box.  (A first version
//               loaded X into registers from global memory, half rows per instruction: the tag stage of the L1 was
//               what bounded it, at 40 lookups a piece, and its unrolled ring cost a microsecond of instruction misses.)
//               The branch's operand goes to shared memory in the layout the MMA reads (K-major, 128-byte swizzle)
//   warp 2      owns tensor memory; fetches the first factor's slabs, one per stage, and issues the MMAs of a
//               chunk once its slabs are complete.  The MMA is 128 rows high; the rows beyond TR read whatever follows in
//               shared memory and their results are never looked at (rows are independent, and the tensor cores are
//               idle here otherwise)
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
//             x * fl32(1/s) is within 2^-20 of the quotient; adding 192 rounds it to a multiple of 2^-16, which restores
//             exact ties and moves nothing else across one; a second addition then rounds to the integer, ties to even.
//   branch    x / sb from the correctly rounded reciprocal by one FMA correction step, which yields the correctly
//             rounded binary32 quotient; 1.5 * 2^23 rounds it to the nearest even integer.
//   MX        x * 2^-e is exact, and the fp16 pipe does it two values at a time: one fma with 1.5 * 2^10 rounds x * 2^-e to
//             the nearest even integer without an intermediate rounding; blocks so small that 2^-e is no fp16 number
//             are scaled up (exactly) first, a rare branch.  MXFP8e4: products below 2^-14 may lose bits, far below half of e4m3's
//             smallest step 2^-9.
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "lq_device.cuh"

namespace {

using namespace lqdev;

constexpr int QWARPS = 16;             // quantizer warps (at most; RG * SX of them have work)
constexpr int FIRST_QWARP = 4;         // warps 0-1 a4, 2 MMA and first factor, 3 X
constexpr int NTHREADS = (FIRST_QWARP + QWARPS) * 32;
constexpr int MAX_SLOTS = 4;           // chunk slots of the branch's operands
constexpr int MAX_XSLOTS = 12;         // chunk slots of X
constexpr float MAGIC = 12582912.0f;   // 1.5 * 2^23: adding it rounds to an integer (ties to even)
enum { BR_NONE = 0, BR_INT = 1, BR_F16 = 2, BR_MXFP = 3, BR_MXINT = 4 };
// MXFP: MXFP8e4 activation codes for an MXFP4 weight; MXINT8: MXINT8 activation codes for an MXINT4 weight, stored as
// two E4M3 digit planes (code = 16 hi + lo)
enum { MAIN_SINT4 = 0, MAIN_MXINT4 = 1, MAIN_MXFP = 2, MAIN_MXINT8 = 3 };

struct QuantParams {
  int M, K, Kpad, Mpad;
  int G;                // SINT4: groups of 64 that hold data
  int nst;              // Kpad / 128 stages of K
  int groups, stages;   // RG row groups of 8 per tile, SX stages of K per chunk
  int ntiles, nchunks;  // tiles of the launch, chunks of a tile
  int slots, xslots;    // chunk slots of the branch's operands and of X
  int refetch;          // integer branch: the X ring is smaller than a tile, which is streamed twice
  uint8_t* qx8;         // [Mpad][Kpad] (MXINT8: [Mpad][2 Kpad], the hi digits' plane then the lo digits')
  float* sx;            // [Gpad][Mpad]
  uint8_t* sfa;         // MX: E8M0 scale bytes [Mpad/128][Kpad/128][512] (MXINT8: [Mpad/128][2 Kpad/128][512], by plane)
  int8_t* qb;           // [Mpad][Kpad] or null (not stored)
  float* sXb;           // [Mpad]
  const float* sL1;     // [LQ_MAX_RANK]
  const uint8_t* sfl1;  // MX branches: E8M0 bytes of the first factor's block scales, [planes][Kpad/128][512]
  uint8_t* sft;         // MX branches: E8M0 bytes of the rank-r intermediate's block scales, [Mpad/128][512 or 1024]
  uint8_t* tq;          // [Mpad][tq_stride]
  float* sT;            // [Mpad]
  int r, rn;            // rank, rank rounded up to 16 (columns of the MMA)
  int bplanes;          // MXINT: digit planes of the first factor (2: 8-bit codes, 1: 4-bit codes)
  int tq_stride;        // bytes per row of tq: LQ_RCONT, or 2 LQ_RCONT when each digit plane of the intermediate has a container
  int nacc;             // accumulators a tile's stages alternate over (floating-point branches: shorter chains of fp32 sums)
  int tmem_cols;        // power of two
  int smem;             // dynamic shared memory of the launch
  int act6;             // MXFP: the activations (X and the rank-r intermediate) are MXFP6e2 instead of MXFP8e4
  float qm;             // largest branch activation code
  int32_t* status;
};

// Shared memory, from a 1024-byte aligned base; the same arithmetic on the host (size) and in the kernel.  First the X ring;
// then the slots: a slot holds a
// chunk: its operand slabs (128 bytes of K wide, a_ps and b_ps of them per stage) and scale bytes.
struct QuantSmem {
  int xslot, a_unit, a_ps, b_unit, b_ps;
  int off_b, off_sfa, off_sfb, slot;            // within a slot
  int off_slots, off_l1, off_max, off_sb, off_bar, total;
};
__host__ __device__ inline QuantSmem quant_smem(int br, int tr, int st, int rn, int bplanes, int slots, int xslots) {
  QuantSmem s{};
  const bool mx = br == BR_MXFP || br == BR_MXINT;
  s.xslot = tr * 256 * st;                      // st: stages of K per chunk
  s.a_unit = tr * 128; s.b_unit = rn * 128;
  s.a_ps = br == BR_NONE ? 0 : (br == BR_F16 || br == BR_MXINT) ? 2 : 1;
  s.b_ps = br == BR_NONE ? 0 : br == BR_F16 ? 2 : br == BR_MXINT ? bplanes : 1;
  s.off_b = st * s.a_ps * s.a_unit;
  s.off_sfa = s.off_b + st * s.b_ps * s.b_unit;
  s.off_sfb = s.off_sfa + (mx ? st * s.a_ps * 512 : 0);
  s.slot = s.off_sfb + (mx ? st * s.b_ps * 512 : 0);
  s.slot = (s.slot + 1023) & ~1023;
  s.off_slots = xslots * s.xslot;
  s.off_l1 = s.off_slots + (br == BR_NONE ? 0 : slots) * s.slot;
  s.off_max = s.off_l1 + LQ_MAX_RANK * 4;       // row maxima of three tiles in rotation, row scales of two
  s.off_sb = s.off_max + 3 * 64 * 4;
  s.off_bar = s.off_sb + 2 * 64 * 4;
  s.total = s.off_bar + 128;
  // the 128-row MMA reads past the last slab of a shorter tile
  if (br != BR_NONE && s.total < s.off_l1 + 128 * 128) s.total = s.off_l1 + 128 * 128;
  return s;
}

__device__ __forceinline__ __half2 as_half2(uint32_t v) { return *reinterpret_cast<const __half2*>(&v); }
__device__ __forceinline__ uint32_t as_u32(__half2 v) { return *reinterpret_cast<const uint32_t*>(&v); }
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

// 2^-e as an fp16 factor (1 for the all-zero block's -127).  Where that is out of fp16's range - the block's maximum is
// below 2^-7 or less - the values are scaled up, exactly, and e follows.
__device__ __forceinline__ __half2 half_scale(uint4& v, int e) {
  if (e < -15 && e > -127) {
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
__device__ __forceinline__ int mxfp8_exponent(float a, bool six = false) {
  const int e = (int)(__float_as_uint(a) >> 23) - 127 - (six ? 2 : 8);
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
__device__ __forceinline__ uint32_t mxfp_pair(float hi, float lo, bool six) {
  return six ? f32x2_to_e4m3x2_via_e2m3(hi, lo) : f32x2_to_e4m3x2(hi, lo);
}
__device__ __forceinline__ uint2 mxfp_codes8(uint4 v, int e, bool six) {
  uint2 w;
  if (six) {
    const float inv = e == -127 ? 0.f : pow2f_n(-e);
    const float2 a = __half22float2(as_half2(v.x)), b = __half22float2(as_half2(v.y)), c = __half22float2(as_half2(v.z)),
                 d = __half22float2(as_half2(v.w));
    w.x = f32x2_to_e4m3x2_via_e2m3(a.y * inv, a.x * inv) | (f32x2_to_e4m3x2_via_e2m3(b.y * inv, b.x * inv) << 16);
    w.y = f32x2_to_e4m3x2_via_e2m3(c.y * inv, c.x * inv) | (f32x2_to_e4m3x2_via_e2m3(d.y * inv, d.x * inv) << 16);
    return w;
  }
  const __half2 inv = half_scale(v, e);  // e in [-32, 7]
  auto q = [&](uint32_t h) { return __hmul2(as_half2(h), inv); };
  w.x = f16x4_to_e4m3x4(q(v.x), q(v.y));
  w.y = f16x4_to_e4m3x4(q(v.z), q(v.w));
  return w;
}

// MXINT4 (Appendix A.3): 2^e with e the smallest integer such that 7 * 2^e >= a: a = 1.f * 2^E, e = E - 2 if 1.f <= 1.75
// else E - 1; -127 for an all-zero block.  Codes rint_even(x / 2^e) as E4M3 bytes.
__device__ __forceinline__ int mxint4_exponent(float a) {
  const uint32_t ab = __float_as_uint(a);
  return a > 0.f ? (int)(ab >> 23) - 127 - (((ab & 0x7FFFFFu) <= 0x600000u) ? 2 : 1) : -127;
}
__device__ __forceinline__ uint2 mxint4_codes8(uint4 v, int e) {
  const __half2 magic = __float2half2_rn(1536.f), inv = half_scale(v, e);   // e in [-26, 14]
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
__device__ __forceinline__ void mxint8_codes8(uint4 v, int e, uint2& hi, uint2& lo) {
  const __half2 inv = half_scale(v, e);  // e in [-30, 10]
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
// One fp32 value (the rank-r intermediate) under its block's exponent, the same digits.
__device__ __forceinline__ void mxint8_digits(float x, float inv, float& hi, float& lo) {
  const float c = __fadd_rn(__fmaf_rn(x, inv, MAGIC), -MAGIC);
  hi = floorf(__fmul_rn(__fadd_rn(c, 8.f), 0.0625f));
  lo = __fmaf_rn(hi, -16.f, c);
}

// SINT4 (Appendix A.3): fp16 scale a / 7 (at least 2^-24), codes rint_even(x / s) clamped to [-7, 7]; only a subnormal
// scale can leave the quotient above 7.5.
struct Sint4Scale {
  float s, inv;
  bool coarse;
};
__device__ __forceinline__ Sint4Scale sint4_scale(float a) {
  Sint4Scale m;
  __half s16 = __float2half_rn(__fmul_rn(a, 0.142857149243354797f));   // fl32(1/7)
  const unsigned short bits = __half_as_ushort(s16);
  if (bits == 0) s16 = __ushort_as_half((unsigned short)1);             // floor 2^-24
  m.s = __half2float(s16);
  m.inv = __frcp_rn(m.s);
  m.coarse = bits < 0x0400;
  return m;
}
__device__ __forceinline__ float2 splat(float v) { return make_float2(v, v); }
__device__ __forceinline__ uint2 sint4_codes8(const uint4& v, const Sint4Scale& m) {
  const float2 x[4] = {__half22float2(as_half2(v.x)), __half22float2(as_half2(v.y)), __half22float2(as_half2(v.z)), __half22float2(as_half2(v.w))};
  const float2 inv = splat(m.inv), c0 = splat(192.f), c1 = splat(MAGIC - 192.f), c2 = splat(-MAGIC);
  float2 q[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) q[i] = __fadd2_rn(__fadd2_rn(__ffma2_rn(x[i], inv, c0), c1), c2);
  if (m.coarse) {
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = make_float2(fminf(fmaxf(q[i].x, -7.f), 7.f), fminf(fmaxf(q[i].y, -7.f), 7.f));
  }
  return make_uint2(f32x2_to_e4m3x2(q[0].y, q[0].x) | (f32x2_to_e4m3x2(q[1].y, q[1].x) << 16),
                    f32x2_to_e4m3x2(q[2].y, q[2].x) | (f32x2_to_e4m3x2(q[3].y, q[3].x) << 16));
}

// Branch codes of eight values under the row's scale sb, invb = fl32(1/sb): q0 = fl32(x invb) is within one ulp of x / sb,
// r = x - sb q0 is exact in an FMA, and fl32(q0 + r invb) is then the correctly rounded quotient (Markstein's correction
// step); |x| / sb <= qm (1 + 2^-23), so it never leaves [-qm, qm].  The low byte of (code + MAGIC)'s bit pattern is the code.
__device__ __forceinline__ uint2 branch_codes8(const uint4& v, float sb, float invb) {
  const float2 x[4] = {__half22float2(as_half2(v.x)), __half22float2(as_half2(v.y)), __half22float2(as_half2(v.z)), __half22float2(as_half2(v.w))};
  const float2 y = splat(invb), ns = splat(-sb), magic = splat(MAGIC);
  uint32_t t[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 q0 = __fmul2_rn(x[i], y);
    const float2 q1 = __fadd2_rn(__ffma2_rn(__ffma2_rn(q0, ns, x[i]), y, q0), magic);
    t[2 * i] = __float_as_uint(q1.x); t[2 * i + 1] = __float_as_uint(q1.y);
  }
  uint2 b;
  b.x = __byte_perm(__byte_perm(t[0], t[1], 0x0040), __byte_perm(t[2], t[3], 0x0040), 0x5410);
  b.y = __byte_perm(__byte_perm(t[4], t[5], 0x0040), __byte_perm(t[6], t[7], 0x0040), 0x5410);
  return b;
}

template <int MAIN, int BR>
__global__ void __launch_bounds__(NTHREADS, 1)
lq_quant_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmL1, const QuantParams p) {
  constexpr bool SINT = MAIN == MAIN_SINT4;
  constexpr bool MXB = BR == BR_MXFP || BR == BR_MXINT;      // the branch multiplies the main codes under their scale bytes
  extern __shared__ uint8_t qsm_raw[];
  const uint32_t base = (smem_u32(qsm_raw) + 1023u) & ~1023u;
  uint8_t* smem = qsm_raw + (base - smem_u32(qsm_raw));
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const int lane = threadIdx.x & 31;
  const int RG = p.groups, spc = p.stages, TR = 8 * RG, nq = RG * spc;       // spc: stages of K per chunk
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
      mbar_init(bar_sync, (uint32_t)nq);
    }
    *abort_flag = 0;
    mbar_init_fence();
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

  const int qw = warp - FIRST_QWARP;
  if (warp == 3) {
    // ------------------------------------------------------------------ TMA producer: X
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
              tma_load_2d(base + (uint32_t)(xs * sm.xslot + b * TR * 128), &tmX, (2 * c * spc + b) * 128, tile * TR, bar_xfull(xs));
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
  } else if (BR != BR_NONE && warp == 2) {
    // ------------------------------------------------------------------ first factor and MMA issuer
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    const uint32_t shape = idesc_shape(p.rn), tsf = tmem + (uint32_t)(2 * p.nacc * p.rn);
    const int total = ((p.ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x) * p.nchunks;   // chunks of this CTA
    // the slabs of chunk number n (chunk `c` of its tile) into their slot: weights, so no earlier kernel is waited for
    auto fetch_b = [&](int slot, int c) {
      const int st0 = c * spc, ns = min(spc, p.nst - st0);
      const uint32_t dst = base + (uint32_t)(sm.off_slots + slot * sm.slot), full = bar_bfull(slot);
      if (elect_one()) {
        mbar_expect_tx(full, (uint32_t)(ns * sm.b_ps * (sm.b_unit + (MXB ? 512 : 0))));
        for (int s = 0; s < ns; ++s)
          for (int u = 0; u < sm.b_ps; ++u) {
            const int i = s * sm.b_ps + u;
            // fp16: a stage's 256 bytes of K in two slabs; digit planes: rn rows further down
            tma_load_2d(dst + sm.off_b + i * sm.b_unit, &tmL1, BR == BR_F16 ? (2 * (st0 + s) + u) * 128 : (st0 + s) * 128,
                        BR == BR_F16 ? 0 : u * p.rn, full);
            if constexpr (MXB) bulk_load(dst + sm.off_sfb + i * 512, p.sfl1 + (size_t)(u * p.nst + st0 + s) * 512, 512, full);
          }
      }
      __syncwarp();
    };
    int fetched = 0, fslot = 0, fchunk = 0;
    uint32_t fpar = 1;
    bool ok = true;
    // keeps the slabs of up to slots - 1 chunks ahead of the MMAs in flight; a slot's previous MMAs were issued a chunk ago
    auto fetch_upto = [&](int n) {
      for (; ok && fetched < n; ++fetched) {
        ok = mbar_wait_warp(bar_empty(fslot), fpar, abort_flag, p.status, LQ_STAGE_MMA);
        if (!ok) break;
        fetch_b(fslot, fchunk);
        if (++fslot == p.slots) { fslot = 0; fpar ^= 1; }
        if (++fchunk == p.nchunks) fchunk = 0;
      }
    };
    fetch_upto(min(p.slots, total));
    uint32_t tc = 0, par = 0;
    int slot = 0, done = 0;
    for (int tile = blockIdx.x; tile < p.ntiles && ok; tile += gridDim.x, ++tc) {
      const uint32_t set = tmem + (uint32_t)((tc & 1) * p.nacc * p.rn);
      ok = mbar_wait_warp(bar_tempty(tc & 1), ((tc >> 1) & 1) ^ 1, abort_flag, p.status, LQ_STAGE_MMA);
      for (int c = 0; c < p.nchunks && ok; ++c) {
        const int ns = min(spc, p.nst - c * spc);
        ok = mbar_wait_warp(bar_bfull(slot), par, abort_flag, p.status, LQ_STAGE_MMA) &&
             mbar_wait_warp(bar_afull(slot), par, abort_flag, p.status, LQ_STAGE_MMA);
        if (!ok) break;
        tc_fence_after();
        const uint32_t at = base + (uint32_t)(sm.off_slots + slot * sm.slot);
        if (elect_one()) {
          for (int s = 0; s < ns; ++s) {
            const int gs = c * spc + s;                          // stage of K: the accumulators take turns
            const uint32_t d = set + (uint32_t)((gs & (p.nacc - 1)) * p.rn), more = gs >= p.nacc;
            const uint32_t a = at + s * sm.a_ps * sm.a_unit, bw = at + sm.off_b + s * sm.b_ps * sm.b_unit;
            if constexpr (BR == BR_INT) {
              const uint64_t ad = make_smem_desc(a), bd = make_smem_desc(bw);
#pragma unroll
              for (int j = 0; j < 4; ++j) tc_mma<TC_I8>(d, ad + 2 * j, bd + 2 * j, IDESC_I8 | shape, more | (uint32_t)j);
            } else if constexpr (BR == BR_F16) {
#pragma unroll
              for (int j = 0; j < 8; ++j)
                tc_mma<TC_F16>(d, make_smem_desc(a + (j >> 2) * sm.a_unit) + 2 * (j & 3), make_smem_desc(bw + (j >> 2) * sm.b_unit) + 2 * (j & 3),
                               IDESC_F16 | shape, more | (uint32_t)j);
            } else {
              // scale bytes into tensor memory (one slot: the tensor pipe executes these copies and MMAs in issue order),
              // then every pair of digit planes
              const int ap = BR == BR_MXINT ? 2 : 1, bp = BR == BR_MXINT ? p.bplanes : 1;
              for (int u = 0; u < ap; ++u) tc_cp_sf(tsf + 4 * u, make_smem_desc_plain(at + sm.off_sfa + (s * ap + u) * 512, 16, 128));
              for (int u = 0; u < bp; ++u) tc_cp_sf(tsf + 8 + 4 * u, make_smem_desc_plain(at + sm.off_sfb + (s * bp + u) * 512, 16, 128));
              for (int ua = 0; ua < ap; ++ua)
                for (int ub = 0; ub < bp; ++ub) {
                  const uint64_t ad = make_smem_desc(a + ua * sm.a_unit), bd = make_smem_desc(bw + ub * sm.b_unit);
#pragma unroll
                  for (int j = 0; j < 4; ++j)
                    tc_mma_mx(d, ad + 2 * j, bd + 2 * j, idesc_mx(p.rn, j), tsf + 4 * ua, tsf + 8 + 4 * ub, more | (uint32_t)(j | ua | ub));
                }
            }
          }
          tc_commit(bar_empty(slot));
          if (c + 1 == p.nchunks) tc_commit(bar_tfull(tc & 1));
        }
        __syncwarp();
        if (++slot == p.slots) { slot = 0; par ^= 1; }
        ++done;
        fetch_upto(min(done + p.slots - 1, total));
      }
    }
    if (!ok && lane == 0) {    // aborting: the copies in flight get a bounded time to land
      for (int i = min(fetched, p.slots); i > 0; --i) {
        if (--fslot < 0) { fslot = p.slots - 1; fpar ^= 1; }
        mbar_settle(bar_bfull(fslot), fpar ^ 1);
      }
    }
  } else if (BR != BR_NONE && warp < 2) {
    // ------------------------------------------------------------------ a4: lane = row of the tile, straight from tensor memory
    grid_dependency_wait();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0) + ((uint32_t)(32 * warp) << 16);
    const int nacc = min(p.nacc, p.nst), row = 32 * warp + lane;
    uint32_t tc = 0;
    for (int tile = blockIdx.x; tile < p.ntiles; tile += gridDim.x, ++tc) {
      const int m = tile * TR + row;
      const bool valid = row < TR && m < p.M;
      const uint32_t set = tmem + (uint32_t)((tc & 1) * p.nacc * p.rn);
      if (!mbar_wait_warp(bar_tfull(tc & 1), (tc >> 1) & 1, abort_flag, p.status, LQ_STAGE_DRAIN)) break;
      tc_fence_after();
      uint8_t* const tqr = p.tq + (size_t)m * p.tq_stride;
      if (32 * warp < TR) {
        // 32 columns of the row from `col` on (zeros beyond the accumulator): the accumulators' sum
        auto fetch = [&](int col, float (&t)[32]) {
          const bool wide = col + 16 < p.rn;
          for (int a = 0; a < nacc; ++a) {
            uint32_t v[32];
            tmem_ld_32x16(set + (uint32_t)(a * p.rn + col), reinterpret_cast<uint32_t(&)[16]>(v[0]));
            if (wide) tmem_ld_32x16(set + (uint32_t)(a * p.rn + col + 16), reinterpret_cast<uint32_t(&)[16]>(v[16]));
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              const float x = j >= 16 && !wide ? 0.f : BR == BR_INT ? __int2float_rn((int)v[j]) : __uint_as_float(v[j]);
              t[j] = a == 0 ? x : t[j] + x;
            }
          }
        };
        float t[32];
        if constexpr (BR == BR_INT) {
          const float sr = row_sb[(tc & 1) * 64 + row];
          auto scaled = [&](int c) {                           // t = fl32(fl32(I1) fl32(sXb sL1))
            fetch(c, t);
#pragma unroll
            for (int j = 0; j < 32; ++j) t[j] = valid ? __fmul_rn(t[j], __fmul_rn(sr, sl1[c + j])) : 0.f;   // rows beyond the tile hold anything
          };
          float amax = 0.f;
          for (int c = 0; c < p.rn; c += 32) {
            scaled(c);
#pragma unroll
            for (int j = 0; j < 32; ++j) amax = fmaxf(amax, fabsf(t[j]));
          }
          const float st = amax == 0.f ? 1.f : __fdiv_rn(amax, p.qm), y = __frcp_rn(st);
          const bool plain = st > 1e-27f && st < 1e27f;        // no step of the corrected quotient can leave binary32's normal range
          if (valid) p.sT[m] = st;
          for (int c = 0; c < p.rn; c += 32) {                 // whole blocks of 32: zeros where the up-projection's K is padded
            if (p.rn > 32) scaled(c);
            uint32_t w[8];
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              float q;
              if (plain) {
                const float q0 = __fmul_rn(t[j], y);
                q = __fmaf_rn(__fmaf_rn(-q0, st, t[j]), y, q0);
              } else {
                q = __fdiv_rn(t[j], st);
              }
              const uint32_t code = __float_as_uint(__fadd_rn(fminf(fmaxf(q, -p.qm), p.qm), MAGIC)) & 0xFFu;
              w[j >> 2] = (j & 3) == 0 ? code : w[j >> 2] | (code << (8 * (j & 3)));
            }
            if (valid) {
              *reinterpret_cast<uint4*>(tqr + c) = make_uint4(w[0], w[1], w[2], w[3]);
              *reinterpret_cast<uint4*>(tqr + c + 16) = make_uint4(w[4], w[5], w[6], w[7]);
            }
          }
        } else if constexpr (BR == BR_F16) {
          if (valid) p.sT[m] = 1.f;
          for (int c = 0; c < p.rn; c += 32) {
            fetch(c, t);
            uint32_t w[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) w[j] = as_u32(__floats2half2_rn(t[2 * j], t[2 * j + 1]));
            if (valid) {
#pragma unroll
              for (int j = 0; j < 4; ++j) *reinterpret_cast<uint4*>(tqr + 2 * c + 16 * j) = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
            }
          }
        } else {
          // blocks of 32 along the rank.  MXINT with one container for both planes (rank <= 64): lo digits 64 bytes after the
          // hi digits, scale slots c and 2 + c of one chunk; a container per plane: 128 bytes on, slot c of the next chunk
          const bool sep = p.tq_stride != LQ_RCONT;
          uint8_t* const sf = p.sft + (size_t)(m >> 7) * (BR == BR_MXINT && sep ? 1024 : 512) + 16 * (m & 31) + 4 * ((m & 127) >> 5);
          for (int b = 0; 32 * b < p.rn; ++b) {
            fetch(32 * b, t);
            float amax = 0.f;
#pragma unroll
            for (int j = 0; j < 32; ++j) amax = fmaxf(amax, fabsf(t[j]));
            const int e = BR == BR_MXINT ? mxint8_exponent(amax) : mxfp8_exponent(amax, p.act6 != 0);
            const float inv = e == -127 ? 0.f : pow2f_n(-e);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              uint32_t w[4], d[4];
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                if constexpr (BR == BR_MXINT) {
                  float hi[4], lo[4];
#pragma unroll
                  for (int i = 0; i < 4; ++i) mxint8_digits(t[16 * h + 4 * j + i], inv, hi[i], lo[i]);
                  w[j] = f32x2_to_e4m3x2(hi[1], hi[0]) | (f32x2_to_e4m3x2(hi[3], hi[2]) << 16);
                  d[j] = f32x2_to_e4m3x2(lo[1], lo[0]) | (f32x2_to_e4m3x2(lo[3], lo[2]) << 16);
                } else {
                  const bool six = p.act6 != 0;
                  w[j] = mxfp_pair(t[16 * h + 4 * j + 1] * inv, t[16 * h + 4 * j] * inv, six) | (mxfp_pair(t[16 * h + 4 * j + 3] * inv, t[16 * h + 4 * j + 2] * inv, six) << 16);
                  d[j] = 0;
                }
              }
              if (valid) {
                *reinterpret_cast<uint4*>(tqr + 32 * b + 16 * h) = make_uint4(w[0], w[1], w[2], w[3]);
                if (BR == BR_MXINT) *reinterpret_cast<uint4*>(tqr + (sep ? 128 : 64) + 32 * b + 16 * h) = make_uint4(d[0], d[1], d[2], d[3]);
              }
            }
            if (valid) {
              sf[b] = (uint8_t)(e + 127 + (BR == BR_MXINT ? 4 : 0));
              if (BR == BR_MXINT) sf[(sep ? 512 : 2) + b] = (uint8_t)(e + 127);
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_tempty(tc & 1));
    }
  } else if (warp >= FIRST_QWARP && qw < nq) {
    // ------------------------------------------------------------------ quantizer
    // This lane: 16-byte vector lc of rows ra and ra + 2 of the tile, of both 64-value boxes of a stage.  The four rows of
    // one access have both values of bit 2, so that the 64-byte halves they write to an operand slab do not meet in the
    // same banks.
    const int rg = qw % RG, sx = qw / RG, lr = lane >> 3, lc = lane & 7;
    const int ra = 8 * rg + (lr & 1) + 2 * (lr & 2);
    const uint32_t sw = (uint32_t)(ra & 7), hstep = (uint32_t)(TR * 128);               // from a box to the next
    const uint32_t xo = base + (uint32_t)(sx * TR * 256 + ra * 128);                    // row ra of this warp's first box
    const uint32_t xo_a = xo + ((lc ^ sw) << 4), xo_b = xo + 256 + ((lc ^ sw ^ 2) << 4);
    // this lane's eight codes in an operand slab (rows of 128 bytes, 16-byte pieces exchanged by row mod 8); the second box's
    // are at the address with bit 6 flipped
    const uint32_t ao = base + (uint32_t)(sm.off_slots + sx * sm.a_ps * sm.a_unit + ra * 128 + 8 * (lc & 1));
    const uint32_t ao_a = ao + (((lc >> 1) ^ sw) << 4), ao_b = ao + 256 + (((lc >> 1) ^ sw ^ 2) << 4);
    const int sr = ra + 2 * (lc & 1);                                                   // lanes 0 and 1 of a row store its scale bytes
    const uint32_t so = base + (uint32_t)(sm.off_slots + sm.off_sfa + sx * sm.a_ps * 512 + 16 * (sr & 31) + 4 * (sr >> 5));
    const size_t qs = MAIN == MAIN_MXINT8 ? (size_t)2 * p.Kpad : (size_t)p.Kpad;        // bytes per row of qx8
    grid_dependency_wait();        // from here on the activation record is written
    int xs = 0, slot = 0;
    uint32_t xpar = 0, epar = 1, tc = 0, buf = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < p.ntiles && ok; tile += gridDim.x, ++tc) {
      const int ma = tile * TR + ra, ms = tile * TR + sr;
      const bool va = ma < p.M, vb = ma + 2 < p.M, vs = lc < 2 && ms < p.M;
      uint8_t* const qa = p.qx8 + (size_t)ma * qs + sx * 128 + 8 * lc;
      uint8_t* const sfr = SINT ? nullptr : p.sfa + ((size_t)(ms >> 7) * (qs >> 7) + sx) * 512 + 16 * (ms & 31) + 4 * ((ms & 127) >> 5);
      float sb_a = 1.f, sb_b = 1.f, inv_a = 1.f, inv_b = 1.f;
      __half2 hm = __float2half2_rn(0.f);                        // maxima of rows ra, ra + 2
      // One walk over the tile.  MAINP: main codes and scales; BRP: the branch's operand; FREE: the X slots are handed back.
      auto walk = [&](auto MAINP, auto BRP, const bool free_x) {
        for (int c = 0, st = sx; c < p.nchunks; ++c, st += spc) {
          const bool live = st < p.nst;
          if (!mbar_wait_warp(bar_xfull(xs), xpar, abort_flag, p.status, LQ_STAGE_QUANT)) return false;
          uint4 a[2], b[2];
          if (live) {
            const uint32_t at = (uint32_t)(xs * sm.xslot);
            a[0] = lds_v4(xo_a + at); b[0] = lds_v4(xo_b + at);
            a[1] = lds_v4(xo_a + at + hstep); b[1] = lds_v4(xo_b + at + hstep);
          }
          uint2 wa[2], wb[2], da[2], db[2];                      // main codes of the two rows (MXINT8: hi digits; d: lo digits)
          uint32_t four = 0;                                     // the stage's scale bytes of row sr (lanes 0 and 1 of a row)
          if constexpr (decltype(MAINP)::value) {
            if (live) {
              [[maybe_unused]] uint32_t own = 0;
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                __half2 bm = __halves2half2(absmax8(a[h]), absmax8(b[h]));
                bm = __hmax2(bm, __shfl_xor_sync(0xffffffffu, bm, 1));
                bm = __hmax2(bm, __shfl_xor_sync(0xffffffffu, bm, 2));
                if constexpr (SINT) bm = __hmax2(bm, __shfl_xor_sync(0xffffffffu, bm, 4));
                if constexpr (BR == BR_INT) hm = __hmax2(hm, bm);
                const float m0 = __low2float(bm), m1 = __high2float(bm);
                if constexpr (SINT) {
                  const Sint4Scale s0 = sint4_scale(m0), s1 = sint4_scale(m1);
                  wa[h] = sint4_codes8(a[h], s0); wb[h] = sint4_codes8(b[h], s1);
                  const int g = 2 * st + h;
                  if (vs && g < p.G) p.sx[(size_t)g * p.Mpad + ms] = lc ? s1.s : s0.s;
                } else {
                  int e0, e1;
                  if constexpr (MAIN == MAIN_MXINT4) {
                    e0 = mxint4_exponent(m0); e1 = mxint4_exponent(m1);
                    wa[h] = mxint4_codes8(a[h], e0); wb[h] = mxint4_codes8(b[h], e1);
                  } else if constexpr (MAIN == MAIN_MXFP) {
                    const bool six = p.act6 != 0;
                    e0 = mxfp8_exponent(m0, six); e1 = mxfp8_exponent(m1, six);
                    wa[h] = mxfp_codes8(a[h], e0, six); wb[h] = mxfp_codes8(b[h], e1, six);
                  } else {
                    e0 = mxint8_exponent(m0); e1 = mxint8_exponent(m1);
                    mxint8_codes8(a[h], e0, wa[h], da[h]); mxint8_codes8(b[h], e1, wb[h], db[h]);
                  }
                  own |= ((uint32_t)(e0 + 127) | ((uint32_t)(e1 + 127) << 16)) << (8 * h);
                }
              }
              if constexpr (!SINT) {
                // a row's four bytes are with two lanes, a block pair apart: lane 0 collects row ra's, lane 1 row ra + 2's
                const uint32_t other = __shfl_xor_sync(0xffffffffu, own, 4);
                four = __byte_perm(own, other, lc ? 0x7362 : 0x5140);
                if (vs) {
                  uint8_t* sf = sfr + (size_t)c * spc * 512;     // (the hi digits weigh 16 times as much)
                  *reinterpret_cast<uint32_t*>(sf) = MAIN == MAIN_MXINT8 ? four + 0x04040404u : four;
                  if (MAIN == MAIN_MXINT8) *reinterpret_cast<uint32_t*>(sf + (size_t)p.nst * 512) = four;
                }
              }
              uint8_t* const q = qa + c * spc * 128;
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                if (va) {
                  *reinterpret_cast<uint2*>(q + 64 * h) = wa[h];
                  if (MAIN == MAIN_MXINT8) *reinterpret_cast<uint2*>(q + p.Kpad + 64 * h) = da[h];
                }
                if (vb) {
                  *reinterpret_cast<uint2*>(q + 2 * qs + 64 * h) = wb[h];
                  if (MAIN == MAIN_MXINT8) *reinterpret_cast<uint2*>(q + 2 * qs + p.Kpad + 64 * h) = db[h];
                }
              }
            }
          }
          if constexpr (decltype(BRP)::value) {
            [[maybe_unused]] uint2 ca[2], cb[2];
            if constexpr (BR == BR_INT) {
              if (live) {
#pragma unroll
                for (int h = 0; h < 2; ++h) { ca[h] = branch_codes8(a[h], sb_a, inv_a); cb[h] = branch_codes8(b[h], sb_b, inv_b); }
              }
            }
            if (!mbar_wait_warp(bar_empty(slot), epar, abort_flag, p.status, LQ_STAGE_QUANT)) return false;
            const uint32_t at = (uint32_t)(slot * sm.slot);
            if (live) {
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                if constexpr (BR == BR_INT) {
                  sts_v2((ao_a + at) ^ (64 * h), ca[h]);
                  sts_v2((ao_b + at) ^ (64 * h), cb[h]);
                  if (p.qb != nullptr) {
                    int8_t* o = p.qb + (qa - p.qx8) + c * spc * 128 + 64 * h;
                    if (va) *reinterpret_cast<uint2*>(o) = ca[h];
                    if (vb) *reinterpret_cast<uint2*>(o + 2 * qs) = cb[h];
                  }
                } else if constexpr (BR == BR_F16) {             // a slab per box: 64 halves, laid out as in the X ring
                  sts_v4(xo_a + sm.off_slots + at + h * hstep, a[h]);
                  sts_v4(xo_b + sm.off_slots + at + h * hstep, b[h]);
                } else {
                  sts_v2((ao_a + at) ^ (64 * h), wa[h]);
                  sts_v2((ao_b + at) ^ (64 * h), wb[h]);
                  if constexpr (BR == BR_MXINT) {
                    sts_v2(((ao_a + at) ^ (64 * h)) + sm.a_unit, da[h]);
                    sts_v2(((ao_b + at) ^ (64 * h)) + sm.a_unit, db[h]);
                  }
                }
              }
              if (MXB && lc < 2) {
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
            if (decltype(BRP)::value) mbar_arrive(bar_afull(slot));
            if (free_x) mbar_arrive(bar_xempty(xs));
          }
          if (++xs == p.xslots) { xs = 0; xpar ^= 1; }
          if (decltype(BRP)::value && ++slot == p.slots) { slot = 0; epar ^= 1; }
        }
        return true;
      };
      using Yes = std::true_type;
      using No = std::false_type;
      if constexpr (BR == BR_INT) {
        const int xs0 = xs;
        const uint32_t xpar0 = xpar;
        ok = walk(Yes(), No(), p.refetch != 0);
        if (!ok) break;
        if (!p.refetch) { xs = xs0; xpar = xpar0; }              // the second walk reads the same slots
        // ---- the rows' maxima and scales: non-negative halves order like their bit patterns
        hm = __hmax2(hm, __shfl_xor_sync(0xffffffffu, hm, 4));
        int* mx = rowmax + buf * 64;
        if (lc < 2) atomicMax(&mx[sr], (int)__half_as_ushort(lc ? __high2half(hm) : __low2half(hm)));
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_sync);
        ok = mbar_wait_warp(bar_sync, tc & 1, abort_flag, p.status, LQ_STAGE_QUANT);
        if (!ok) break;
        const float rm_a = __half2float(__ushort_as_half((unsigned short)mx[ra]));
        const float rm_b = __half2float(__ushort_as_half((unsigned short)mx[ra + 2]));
        const uint32_t after = buf == 0 ? 2 : buf - 1;           // two tiles on: every warp is past its last use
        if (sx == 0 && lc < 2) rowmax[after * 64 + sr] = 0;
        buf = buf == 2 ? 0 : buf + 1;
        sb_a = rm_a == 0.f ? 1.f : __fdiv_rn(rm_a, p.qm);
        sb_b = rm_b == 0.f ? 1.f : __fdiv_rn(rm_b, p.qm);
        inv_a = __frcp_rn(sb_a); inv_b = __frcp_rn(sb_b);
        if (sx == 0) {                                           // a4 reads the scale: its previous tile of this parity must be done
          ok = mbar_wait_warp(bar_tempty(tc & 1), ((tc >> 1) & 1) ^ 1, abort_flag, p.status, LQ_STAGE_QUANT);
          if (!ok) break;
          if (lc < 2) row_sb[(tc & 1) * 64 + sr] = lc ? sb_b : sb_a;
          if (vs) p.sXb[ms] = lc ? sb_b : sb_a;
        }
        ok = walk(No(), Yes(), true);
      } else {
        ok = walk(Yes(), std::integral_constant<bool, BR != BR_NONE>(), true);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (BR != BR_NONE && warp == 2) {
    tc_fence_after();
    tmem_dealloc(__shfl_sync(0xffffffffu, *tmem_slot, 0), (uint32_t)p.tmem_cols);
  }
}

// How a launch is cut.  Cost model in chunk times of a full complement of warps: a CTA's tiles times (its chunks, twice
// where a tile is walked twice, plus what starting and finishing a tile costs); among equals the higher tile, which reads
// the first factor less often.
bool plan_cut(int br, QuantParams& p, int sms) {
  const int walks = br == BR_INT ? 2 : 1, room = 227 * 1024 - 1024;
  double best = 1e30;
  QuantParams out = p;
  for (int groups = 8; groups >= 1; --groups) {
    if (g_lq_quant_warps > 0 && groups != std::min(8, g_lq_quant_warps)) continue;
    for (int stages = std::min(QWARPS / groups, p.nst); stages >= 1; --stages) {
      if (g_lq_quant_ctas > 0 && stages != g_lq_quant_ctas) continue;
      QuantParams c = p;
      c.groups = groups; c.stages = stages;
      c.ntiles = lq_ceil_div(p.M, 8 * groups);
      c.nchunks = lq_ceil_div(p.nst, stages);
      c.xslots = 0;
      // operand slots first, then as many chunks of X as fit; an integer branch would rather hold a whole tile of X
      const int want = br == BR_INT ? c.nchunks : 4;
      for (int slots = br == BR_NONE ? 1 : MAX_SLOTS; slots >= (br == BR_NONE ? 1 : 2) && c.xslots < want; --slots) {
        const QuantSmem s = quant_smem(br, 8 * groups, stages, p.rn, p.bplanes, slots, 0);
        const int fit = std::min(MAX_XSLOTS, (room - s.total) / s.xslot);
        if (fit > c.xslots && fit >= 2) { c.xslots = fit; c.slots = slots; }
      }
      if (c.xslots < 2) continue;
      c.xslots = std::min(c.xslots, 2 * c.nchunks);
      c.refetch = br == BR_INT && c.xslots < c.nchunks;
      c.smem = quant_smem(br, 8 * groups, stages, p.rn, p.bplanes, c.slots, c.xslots).total + 1024;
      const double chunk = 0.4 + 0.6 * groups * stages / QWARPS;
      const double cost = lq_ceil_div(c.ntiles, sms) * (c.nchunks * walks * chunk + 1.0) + 3.0;
      if (cost < best) { best = cost; out = c; }
    }
  }
  p = out;
  return best < 1e30;
}

template <int MAIN, int BR>
cudaError_t launch_quant(const void* X, const CUtensorMap& tm, QuantParams& p, int sms, cudaStream_t st) {
  static bool attr_set[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (!attr_set[dev & 63]) {
    const cudaError_t e = cudaFuncSetAttribute(lq_quant_kernel<MAIN, BR>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return e;
    attr_set[dev & 63] = true;
  }
  if (!plan_cut(BR, p, sms)) return cudaErrorInvalidConfiguration;
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
  p.M = M; p.K = L->K; p.Kpad = L->Kpad; p.Mpad = A->Mpad; p.G = L->G;
  p.nst = L->Kpad / LQ_KSTAGE;
  p.qx8 = A->d_qx8; p.sx = A->d_sx; p.sfa = A->d_sfa;
  p.qb = g_lq_store_qb ? A->d_qb : nullptr;
  p.sXb = A->d_sXb; p.sL1 = L->d_sL1; p.sfl1 = L->d_sfl1;
  p.sft = A->d_sft; p.tq = A->d_tq; p.sT = A->d_sT;
  p.r = L->r; p.rn = lq_l1_rows(L);
  p.bplanes = lq_l1_planes(L);
  p.tq_stride = A->tq_stride;
  // Floating-point branches: a tile's stages alternate over two to four accumulators, which are added in fp32 at the end;
  // tensor memory holds two such sets and the scale bytes' columns.
  p.nacc = L->integer_branch ? 1 : p.rn <= 48 ? 4 : p.rn <= 112 ? 2 : 1;
  if (L->f16_branch && p.rn > 48) p.nacc = 4;
  p.tmem_cols = 32;
  while (p.tmem_cols < 2 * p.nacc * p.rn + ((L->mxfp || L->a8) ? 16 : 0)) p.tmem_cols *= 2;
  p.act6 = (L->mxfp && L->cfg.act_fmt == LQ_ACT_MXFP6) ? 1 : 0;
  p.qm = abits > 0 ? (float)((1 << (abits - 1)) - 1) : 0.f;
  p.status = lq_device_status_ptr(A->device);
  if (!p.status) return LQ_ERR_CUDA;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, A->device) != cudaSuccess) return LQ_ERR_CUDA;
  cudaError_t e;
  if (L->mxfp) e = L->r > 0 ? launch_quant<MAIN_MXFP, BR_MXFP>(X, L->tmL1, p, sms, st) : launch_quant<MAIN_MXFP, BR_NONE>(X, L->tmL1, p, sms, st);
  else if (L->a8) e = L->r > 0 ? launch_quant<MAIN_MXINT8, BR_MXINT>(X, L->tmL1, p, sms, st) : launch_quant<MAIN_MXINT8, BR_NONE>(X, L->tmL1, p, sms, st);
  else if (L->mx)
    e = L->f16_branch ? launch_quant<MAIN_MXINT4, BR_F16>(X, L->tmL1, p, sms, st)
                      : L->integer_branch ? launch_quant<MAIN_MXINT4, BR_INT>(X, L->tmL1, p, sms, st) : launch_quant<MAIN_MXINT4, BR_NONE>(X, L->tmL1, p, sms, st);
  else
    e = L->f16_branch ? launch_quant<MAIN_SINT4, BR_F16>(X, L->tmL1, p, sms, st)
                      : L->integer_branch ? launch_quant<MAIN_SINT4, BR_INT>(X, L->tmL1, p, sms, st) : launch_quant<MAIN_SINT4, BR_NONE>(X, L->tmL1, p, sms, st);
  return lq_note_cuda(e) == cudaSuccess ? LQ_OK : LQ_ERR_CUDA;
}
