// Main W4A4 product of the layer on the 5th-generation tensor cores, with the per-group
// scales, the low-rank branch's up-projection and the bias applied in one epilogue:
//
//   Y[m,n] = sum_g sx[m,g] sw[g,n] (qx_g Wq_g)[m,n] + sT[m] sL2[n] (tq L2q)[m,n] + bias[n]
//
// (Figure 1: residual branch Q(X) Q1(P) plus low-rank branch; Appendix A.3: SINT4 carries one
// scale per block of 64 values on BOTH operands, so every 64-deep partial product needs its
// own rank-1 scale before it may be summed.)
//
// Shape of the kernel (persistent, one CTA per SM, warp-specialised, 12 warps):
//   warp 0      TMA producer: operand tiles (two groups = 128 bytes of K per stage row), the two groups' scale vectors and,
//               with a tile's first stage, the bias, all signalled on the stage's "full" barrier
//   warp 1      owns tensor memory; issues tcgen05.mma: each group of 64 codes is two K=32 MMAs into a FRESH 128 x 128
//               accumulator.  A stage's two groups fill one PAIR of accumulators as soon as the drain has read it out
//               and are handed over with one commit; two pairs alternate
//   warps 4-11  drain: each warp owns 32 rows x 64 columns of the tile.  Half a group's slice is two tcgen05.ld.16x256b.x4; it is
//               in flight into one register buffer while the half before is consumed from the other:
//               acc += (P * sx) * sw, packed f32x2, fp32 registers (the integer branch's stage: P * (sx * sw)).  A pair goes back as soon
//               as its last half sits in registers.  The next stage's scales are loaded, and the next tile's first half is requested,
//               before the last half is consumed
// What bounds it: the FP32 pipe's operand delivery and the drain's other instructions.  Per group and scheduler 64 packed products
// (2.0 to 2.6 clocks each, measured) and 64 packed FMAs (2.75 with an operand shared by neighbours, 3.9 with three of their own) are about 320
// clocks, the tensor pipe needs 128; the same loop over tensor memory without any hand-shake takes 400, 100 of them for the scales' way
// from shared memory, the kernel takes 430.  So everything that is not arithmetic is kept out of the drain's instruction stream: two
// wide warps per scheduler instead of four narrow ones, no wait or arrival for the scale vectors (they live in a ring deep
// enough that the accumulators' hand-shakes imply theirs), one wait per stage, 224 registers per drain thread, partly
// taken over from the other four warps (setmaxnreg).  M = 8192, K x N = 1152 x 3456 / 4608 x 1152: 85 / 96 us with sixteen
// narrow warps, 80 / 89 with one commit per group; then, timed in turn with other inputs each time, 81.1 / 88.3, 78.0 / 84.0 with P sx first,
// 72.4 / 81.6 with sectors stored whole, 70.1 / 78.1 with a stage's commits under one election, 64.5 / 70.9 with the issuer written out and the
// drain's last eight registers, 64.2 / 68.9 with halves of groups in flight and one hand-back a stage.  At K = 1152 a tile's end is a
// fifth of the launch: of 11.4 k clocks a tile 1.0 k are the branch's group, 0.8 k the stores, 0.5 k the way to the next tile's first
// stage.  Scalar FMAs lose their issue slots (94 - 104 us for 79); with whole groups in flight, scales of the next group loaded where
// this one's were used last made the kernel slower (73.6 for 68.8: registers); two column halves as pipelines of their own, each with an
// issuer, 67.9 for 66.5.
// Orders of rows and columns (lq_internal.h) are chosen for the drain's fragments: the columns of the tile are permuted in
// the weight operand so that a lane's 16 columns of a row are neighbours in Y - the epilogue converts and stores, no
// exchange - and the scale vectors are permuted so that a lane's come in one (rows) and four (columns) 16-byte loads
// without bank conflicts.
// Work is cut in 128 x 128 tiles; every CTA takes a contiguous, balanced run of them, row block major.
// The 4-bit codes ride in E4M3 operands (integers up to 7 are exact, fp32 accumulation of
// |sum| <= 3136 is exact); the branch's 8-bit codes use kind::i8 (exact int32), the fp16
// reference branch kind::f16.
// Every wait is bounded; on expiry the role records LQ_ERR_TIMEOUT in the device status word,
// raises a CTA-wide abort flag and all roles leave through the common teardown.
#include <cuda_fp16.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "lq_device.cuh"
#include "lq_gemm_cut.h"

#ifdef LQ_TIMELINE
// Timeline build only: copies the stamp lists of the last launch to the host ([TL_LISTS][TL_CAP] words) and clears them.
extern "C" int lq_debug_timeline(unsigned long long* host_out) {
  if (cudaDeviceSynchronize() != cudaSuccess) return 1;
  if (cudaMemcpyFromSymbol(host_out, g_lq_timeline, sizeof(unsigned long long) * lqdev::TL_LISTS * lqdev::TL_CAP) != cudaSuccess) return 1;
  static unsigned long long zeros[lqdev::TL_LISTS][lqdev::TL_CAP];
  return cudaMemcpyToSymbol(g_lq_timeline, zeros, sizeof(zeros)) == cudaSuccess ? 0 : 1;
}
#endif

namespace {

using namespace lqdev;

constexpr int UNIT = LQ_BN;                        // 128 output columns per tile
constexpr int NSTAGE = 4;                          // operand ring depth (a power of two: ring positions are masks)
constexpr int NPAIR = 2;                           // ring of accumulator pairs in tensor memory, a stage's two groups: 2 x 2 x 128 columns
constexpr int TCOLS = 128;                         // columns per accumulator
constexpr int STAGE_A_BYTES = LQ_BM * LQ_KSTAGE;   // 16 KB
constexpr int STAGE_B_BYTES = UNIT * LQ_KSTAGE;    // 16 KB
constexpr int STAGE_BYTES = STAGE_A_BYTES + STAGE_B_BYTES;
constexpr int SC_GROUP_FLOATS = LQ_BM + UNIT;      // sx[128] then sw[128]
constexpr int SC_STAGE_BYTES = (2 * SC_GROUP_FLOATS + UNIT) * 4;   // two groups, bias[128] (a tile's first stage)
constexpr int SC_RING = 8;                         // slots of the scale ring
constexpr int NUM_DRAIN_WARPS = 8;
constexpr int FIRST_DRAIN_WARP = 4;                // the first warpgroup: TMA, MMA, two idle warps
constexpr int GEMM_THREADS = (FIRST_DRAIN_WARP + NUM_DRAIN_WARPS) * 32;
constexpr int WCOLS = 64;                          // columns per drain warp
// 12 warps are launched with 168 registers a thread: 384 x 168 = 64512 = 128 x 56 + 256 x 224.  (216 for the drain: 64.6 / 73.1 us at the sizes
// above for 62.7 / 69.6; 232 and 40: 64.1 / 71.5, the producer spills)
constexpr int LAUNCH_REGS = 65536 / GEMM_THREADS & ~7, LEAN_REGS = 56, DRAIN_REGS = 224;
// setmaxnreg takes from what the CTA was launched with and would wait for ever for more: the only wait without a limit, so its sum is
// checked here and every instance's own count in lq_gemm_prepare
static_assert(FIRST_DRAIN_WARP * 32 * LEAN_REGS + NUM_DRAIN_WARPS * 32 * DRAIN_REGS <= GEMM_THREADS * LAUNCH_REGS, "registers of the split");
constexpr int SMEM_BAR_BYTES = 256;
constexpr int SMEM_BYTES = 1024 /*alignment slack*/ + NSTAGE * STAGE_BYTES + SC_RING * SC_STAGE_BYTES + SMEM_BAR_BYTES;
// TILE_SPLIT: and the cluster's partial sums of this CTA's part of the tile
constexpr int GATHER_ITEMS = 16;                   // of a drain thread's 4 rows x 16 columns, four neighbouring columns each
constexpr int GATHER_BYTES = GATHER_ITEMS * NUM_DRAIN_WARPS * 32 * 16;
static_assert(SMEM_BYTES + GATHER_BYTES <= 232448, "shared memory budget");
static_assert(STAGE_BYTES % 1024 == 0, "stages must keep the 1024-byte alignment of the swizzled tiles");
static_assert((NSTAGE & (NSTAGE - 1)) == 0 && (NPAIR & (NPAIR - 1)) == 0, "ring sizes must be powers of two");

struct GemmParams {
  int M, N, Mpad, Npad;
  int n_stages_main;      // Kpad / 128 (an odd last group's partner has zero codes and scales)
  int branch_mmas;        // MMAs of the branch stage (32 bytes of r each)
  int tiles_m, units_n;
  int split;              // CTAs (of a cluster) that share a tile's stages
  const float* sx;        // [Gpad][Mpad]
  const float* sw;        // [Gpad][Npad]
  const float* sT;        // [Mpad]
  const float* sL2;       // [Npad]
  const float* bias;      // [Npad]
  void* Y;
  int out_f32;
  int wide;               // TILE_SPLIT: Y and its rows begin on 32-byte boundaries
  int32_t* status;
};

// Half a group's slice of a drain warp, two accumulator slices of 16 rows x 32 columns in the layout of tcgen05.ld.16x256b
// (the accumulator-fragment layout of mma.sync m16n8: with g = lane / 4 and t = lane % 4, registers 4j .. 4j+3 of a
// slice hold row g, columns 8j + 2t and 8j + 2t + 1, then row g + 8, the same columns), times its scales, added to the accumulators.
// INT: the accumulator holds int32 (kind::i8); |P| < 2^22, so adding 1.5 * 2^23 in the integer domain and subtracting it
// in fp32 converts exactly without the conversion pipe.
typedef uint32_t Frag[16];                            // 16 rows x 32 columns
template <bool INT>
__device__ __forceinline__ float2 fragment_pair(uint32_t a, uint32_t b) {
  if constexpr (INT)
    return make_float2(__int_as_float((int)a + 0x4B400000) - 12582912.0f, __int_as_float((int)b + 0x4B400000) - 12582912.0f);
  else
    return make_float2(__uint_as_float(a), __uint_as_float(b));
}
struct Scales {                                       // a lane's four row scales and 16 column scales of a group
  float4 sx, sw[4];
};
__device__ __forceinline__ void load_scales(Scales& v, uint32_t sx_at, uint32_t sw_at) {
  v.sx = *reinterpret_cast<const float4*>(__cvta_shared_to_generic(sx_at));           // rows g, g + 8, g + 16, g + 24
#pragma unroll
  for (int k = 0; k < 4; ++k) v.sw[k] = *reinterpret_cast<const float4*>(__cvta_shared_to_generic(sw_at + 64 * k));
}
// Two orders of the same products.  The codes' sums have 12 bits and the fp16 scales 11, so P sx and sx sw are exact alike and every FMA
// rounds the same number; P sx leaves an FMA with an operand (sw) that four rows in a row share, which costs the register file
// less (us, M = 8192, K x N = 1152 x 3456 / 4608 x 1152: 81.1 / 88.3 -> 78.0 / 84.0).  The integer branch's scales have 24 bits, its sums up
// to 22: there sx sw is rounded first.
template <bool INT, int HALF>
__device__ __forceinline__ void drain_half(const Frag (&v)[2], float2 (&acc)[2][16], const Scales& sc) {
  const float4 sx = sc.sx;
  const float2 s0 = make_float2(sx.x, sx.x), s1 = make_float2(sx.y, sx.y), s2 = make_float2(sx.z, sx.z), s3 = make_float2(sx.w, sx.w);
#pragma unroll
  for (int k = 2 * HALF; k < 2 * HALF + 2; ++k) {
    const float4 w = sc.sw[k];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int j = 2 * k + e, q = 4 * (j & 3);
      const float2 sw = e ? make_float2(w.z, w.w) : make_float2(w.x, w.y);
      const float2 p0 = fragment_pair<INT>(v[0][q], v[0][q + 1]), p1 = fragment_pair<INT>(v[0][q + 2], v[0][q + 3]);
      const float2 p2 = fragment_pair<INT>(v[1][q], v[1][q + 1]), p3 = fragment_pair<INT>(v[1][q + 2], v[1][q + 3]);
      float2 &a0 = acc[0][2 * j], &a1 = acc[0][2 * j + 1], &a2 = acc[1][2 * j], &a3 = acc[1][2 * j + 1];
      if constexpr (INT) {
        a0 = __ffma2_rn(p0, __fmul2_rn(s0, sw), a0); a1 = __ffma2_rn(p1, __fmul2_rn(s1, sw), a1);
        a2 = __ffma2_rn(p2, __fmul2_rn(s2, sw), a2); a3 = __ffma2_rn(p3, __fmul2_rn(s3, sw), a3);
      } else {
        const float2 t0 = __fmul2_rn(p0, s0), t1 = __fmul2_rn(p1, s1), t2 = __fmul2_rn(p2, s2), t3 = __fmul2_rn(p3, s3);
        a0 = __ffma2_rn(t0, sw, a0); a1 = __ffma2_rn(t1, sw, a1); a2 = __ffma2_rn(t2, sw, a2); a3 = __ffma2_rn(t3, sw, a3);
      }
    }
  }
}
__device__ __forceinline__ void fetch_half(uint32_t taddr, Frag (&v)[2]) {
#pragma unroll
  for (int i = 0; i < 2; ++i) tmem_ld_16x256b_x4(taddr + ((uint32_t)(16 * i) << 16), v[i]);
}

// A group's two MMAs under one election (both groups of a stage under one were 1 to 2 % slower), predicated instead of branched around:
// the control flow of the issuing warp stays uniform.  (An `if` of one lane around them and around the commits, with a loop over the
// groups: a stage's way through the issuer, 1.2 k clocks, was as long as the drain's.  us, M = 8192, K x N = 1152 x 3456 / 4608 x 1152:
// 72.4 / 81.6 -> 64.5 / 70.9, with the drain's eight registers.)
#define LQ_GROUP_MMAS                                                   \
  "{\n\t.reg .pred P, T, F;\n\t"                                       \
  "elect.sync _|P, 0xffffffff;\n\t"                                    \
  "setp.eq.b32 T, 0, 0;\n\t"                                           \
  "setp.ne.b32 F, 0, 0;\n\t"                                           \
  "@P tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %3, %5, F;\n\t"  \
  "@P tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %2, %4, %5, T;\n\t"
__device__ __forceinline__ void issue_group(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc) {
  asm volatile(LQ_GROUP_MMAS "}" ::"r"(d), "l"(a), "l"(a + 2), "l"(b), "l"(b + 2), "r"(idesc) : "memory");
}
// a stage's last group: and the commits
__device__ __forceinline__ void issue_group(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t bar_group, uint32_t bar_stage) {
  asm volatile(LQ_GROUP_MMAS
               "@P tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%6];\n\t"
               "@P tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%7];\n\t}"
               ::"r"(d), "l"(a), "l"(a + 2), "l"(b), "l"(b + 2), "r"(idesc), "r"(bar_group), "r"(bar_stage)
               : "memory");
}

enum { BRANCH_NONE = 0, BRANCH_I8 = 1, BRANCH_F16 = 2 };
enum { TILE_WHOLE = 0, TILE_SECTORS = 1, TILE_SPLIT = 2 };

// TILE_SPLIT: the CTAs of a cluster share one tile, each with a part of the stages (K and the branch).  Every CTA adds up a part of the
// tile: the others copy their partial sums of it into its shared memory, and it waits for the bytes.  What bounds it is that one trip.
// (Rendezvous, loads of all parts from the others' shared memory and a second rendezvous before leaving: us, M x K x N by two, four,
// eight CTAs, 120 x 1152 x 4608 8.40 -> 7.57, 256 x 4608 x 1152 11.05 -> 10.27, 1 x 1152 x 1152 5.46 -> 4.80, 120 x 8192 x 1152 11.26 ->
// 9.83.  Stores of 16 bytes by every thread instead of copies from a staging place: 4.60 with one row, but 8.90 with 128; both, by the
// number of rows: 4.68 and 7.8.)  TILE_SECTORS: every row of Y begins on a 32-byte boundary.  (An instance of its own: with both kinds of
// stores in one epilogue the drain's registers were worse allocated: 63.6 / 69.4 us for 62.3 / 69.0, M = 8192, K x N = 1152 x 3456 / 4608 x 1152.)
template <int BRANCH, int TILE>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
lq_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmT, const __grid_constant__ CUtensorMap tmL2,
               const GemmParams p) {
  constexpr bool SPLIT = TILE == TILE_SPLIT, SECTORS = TILE == TILE_SECTORS;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t sm_stage = base;
  const uint32_t sm_sc = base + NSTAGE * STAGE_BYTES;
  const float* sc_ptr = reinterpret_cast<const float*>(smem + NSTAGE * STAGE_BYTES);
  const uint32_t sm_bar = sm_sc + SC_RING * SC_STAGE_BYTES;
  uint8_t* bar_ptr = smem + NSTAGE * STAGE_BYTES + SC_RING * SC_STAGE_BYTES;
  // barrier map (8 bytes each)
  auto bar_full = [&](int s) { return sm_bar + 8u * (uint32_t)s; };                        // operands + scales landed
  auto bar_empty = [&](int s) { return sm_bar + 8u * (uint32_t)(NSTAGE + s); };           // MMAs of the stage retired
  auto bar_tfull = [&](int b) { return sm_bar + 8u * (uint32_t)(2 * NSTAGE + b); };
  // (With a branch 16 bytes apart: 8 bytes apart, as they fit, the same code is 1.5 to 2.5 % slower, without one 2 to 4 % faster; what in it is
  // not known.  No branch, us 16 / 8 bytes apart: M = 8192, K x N = 1152 x 3456 / 4608 x 1152 59.0 / 56.8, 69.1 / 66.1, M = 23821, 712 x 6328 251 / 246.)
  constexpr int EMPTY_AT = BRANCH == BRANCH_NONE ? 0 : 1, EMPTY_STRIDE = BRANCH == BRANCH_NONE ? 1 : 2;
  auto bar_tempty = [&](int b) { return sm_bar + 8u * (uint32_t)(2 * NSTAGE + NPAIR + EMPTY_AT + EMPTY_STRIDE * b); };
  [[maybe_unused]] const uint32_t bar_gather = sm_bar + 8u * (uint32_t)(2 * NSTAGE + 3 * NPAIR);
  constexpr int NBAR = 2 * NSTAGE + 3 * NPAIR + 1;
  static_assert(NBAR * 8 + 16 <= SMEM_BAR_BYTES, "barrier area too small");
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_ptr + NBAR * 8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_ptr + NBAR * 8 + 8);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);   // provably warp-uniform
  const int lane = threadIdx.x & 31;
  const int stages_per_tile = p.n_stages_main + (BRANCH != BRANCH_NONE ? 1 : 0);
  // this CTA's contiguous run of 128 x 128 tiles, row block major (SPLIT: its cluster's only one)
  const long long units = (long long)p.tiles_m * p.units_n;
  const int u_begin = SPLIT ? (int)blockIdx.x / p.split : (int)((units * blockIdx.x) / gridDim.x);
  const int u_end = SPLIT ? u_begin + 1 : (int)((units * (blockIdx.x + 1)) / gridDim.x);
  // and of a tile's stages
  const int part = SPLIT ? (int)blockIdx.x % p.split : 0;
  const int s_begin = SPLIT ? stages_per_tile * part / p.split : 0;
  const int s_end = SPLIT ? stages_per_tile * (part + 1) / p.split : stages_per_tile;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NSTAGE; ++s) {
      mbar_init(bar_full(s), 1);
      mbar_init(bar_empty(s), 1);
    }
    for (int b = 0; b < NPAIR; ++b) { mbar_init(bar_tfull(b), 1); mbar_init(bar_tempty(b), NUM_DRAIN_WARPS); }
    *abort_flag = 0;
    if constexpr (SPLIT) mbar_init(bar_gather, 1);
    mbar_init_fence();
    if constexpr (SPLIT) {
      // what the cluster's other CTAs will copy here: of this part's items those of eight rows that exist, by two warps (column halves) each
      int items = 0;
      for (int j = part * GATHER_ITEMS / p.split; j < (part + 1) * GATHER_ITEMS / p.split; ++j)
        for (int q = 0; q < 4; ++q) items += (u_begin / p.units_n) * LQ_BM + 32 * q + 8 * (j >> 2) < p.M;
      mbar_expect_tx(bar_gather, (uint32_t)((p.split - 1) * 2 * items * 512));
    }
  }
  if (warp == 1) tmem_alloc(smem_u32(tmem_slot), 512);
  tc_fence_before();
  __syncthreads();
  if constexpr (SPLIT) cluster_arrive();
  grid_launch_dependents();
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  // SPLIT: the place of a drain warp's items (n_items of 32 lanes x 16 bytes, then the next warp's) that CTA `from` of the cluster has
  // summed for this one; and where this CTA's own sums wait, by the part that they are for (the operands' place: every MMA has retired)
  [[maybe_unused]] const int n_items = SPLIT ? GATHER_ITEMS / p.split : 0;
  auto items_at = [&](uint32_t area, int block, int dwarp) { return area + (uint32_t)((block * NUM_DRAIN_WARPS + dwarp) * n_items) * 512; };
  [[maybe_unused]] const uint32_t sm_gather = sm_bar + SMEM_BAR_BYTES;
  bool drained = false;

  LQ_TL_DECL((blockIdx.x == 0 && lane == 0)
                 ? (warp == 0 ? (int)TL_PRODUCER : warp == 1 ? (int)TL_MMA : warp == FIRST_DRAIN_WARP ? (int)TL_DRAIN_FIRST
                    : warp == FIRST_DRAIN_WARP + NUM_DRAIN_WARPS - 1 ? (int)TL_DRAIN_LAST : -1)
                 : -1);

  if (warp < FIRST_DRAIN_WARP) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(LEAN_REGS));
    if (warp == 0) {
      // ------------------------------------------------------------------ TMA producer
      uint32_t it = 0, armed = 0;
      bool ok = true;
      // The weights' half of a stage (with the announcement of all of it) and the activations' half.
      auto load_weights = [&](uint32_t i, int s, int n0) {
        const int st = i & (NSTAGE - 1);
        const uint32_t b_dst = sm_stage + st * STAGE_BYTES + STAGE_A_BYTES, sc_dst = sm_sc + (i & (SC_RING - 1)) * SC_STAGE_BYTES;
        const uint32_t full = bar_full(st);
        const bool is_main = s < p.n_stages_main;
        if (elect_one()) {
          mbar_expect_tx(full, STAGE_BYTES + (is_main ? 2 : 1) * SC_GROUP_FLOATS * 4 + (s == s_begin ? UNIT * 4 : 0));
          if (s == s_begin) bulk_load(sc_dst + 2 * SC_GROUP_FLOATS * 4, p.bias + n0, UNIT * 4, full);
          if (is_main) {
            tma_load_2d(b_dst, &tmB, s * LQ_KSTAGE, n0, full);
            for (int q = 0; q < 2; ++q)
              bulk_load(sc_dst + q * SC_GROUP_FLOATS * 4 + LQ_BM * 4, p.sw + (size_t)(2 * s + q) * p.Npad + n0, UNIT * 4, full);
          } else {
            tma_load_2d(b_dst, &tmL2, 0, n0, full);
            bulk_load(sc_dst + LQ_BM * 4, p.sL2 + n0, UNIT * 4, full);
          }
        }
        __syncwarp();
      };
      auto load_acts = [&](uint32_t i, int s, int m0) {
        const int st = i & (NSTAGE - 1);
        const uint32_t a_dst = sm_stage + st * STAGE_BYTES, sc_dst = sm_sc + (i & (SC_RING - 1)) * SC_STAGE_BYTES, full = bar_full(st);
        if (elect_one()) {
          if (s < p.n_stages_main) {
            tma_load_2d(a_dst, &tmA, s * LQ_KSTAGE, m0, full);
            for (int q = 0; q < 2; ++q)
              bulk_load(sc_dst + q * SC_GROUP_FLOATS * 4, p.sx + (size_t)(2 * s + q) * p.Mpad + m0, LQ_BM * 4, full);
          } else {
            tma_load_2d(a_dst, &tmT, 0, m0, full);
            bulk_load(sc_dst, p.sT + m0, LQ_BM * 4, full);
          }
        }
        __syncwarp();
      };
      // Weights do not depend on earlier kernels: the first ring's worth is requested before they are waited for.
      const uint32_t early = u_begin < u_end ? (uint32_t)min(NSTAGE, s_end - s_begin) : 0;
      for (uint32_t i = 0; i < early; ++i) load_weights(i, s_begin + (int)i, (u_begin % p.units_n) * UNIT);
      grid_dependency_wait();
      for (int u = u_begin; u < u_end && ok; ++u) {
        const int mb = u / p.units_n, nu = u - mb * p.units_n;
        for (int s = s_begin; s < s_end && ok; ++s, ++it) {
          if (it >= early) {
            ok = mbar_wait_warp(bar_empty(it & (NSTAGE - 1)), ((it / NSTAGE) & 1) ^ 1, abort_flag, p.status, LQ_STAGE_PRODUCER);
            if (!ok) break;
            // (Nothing says that the drain is done with the slot's old scale vectors, eight stages back, and nothing has to: the
            // MMAs that have just retired, four stages back, had to wait for the accumulators of six stages back to be in the
            // drain's registers, and by then it had used up the scales of the stages before.)
            LQ_TL(EV_P_SLOT_FREE, s);
            load_weights(it, s, nu * UNIT);
          }
          load_acts(it, s, mb * LQ_BM);
          ++armed;
          LQ_TL(EV_P_ISSUED, s);
        }
      }
      armed = armed > early ? armed : early;
      if (!ok && lane == 0) {
        // aborting: give the copies already issued a bounded time to land before the CTA's shared memory goes away
        const uint32_t n = armed < (uint32_t)NSTAGE ? armed : (uint32_t)NSTAGE;
        for (uint32_t i = 1; i <= n; ++i) {
          const uint32_t j = armed - i;
          mbar_settle(bar_full(j % NSTAGE), (j / NSTAGE) & 1);
        }
      }
    } else if (warp == 1) {
      // ------------------------------------------------------------------ MMA issuer
      uint32_t it = 0;
      bool ok = true;
      const uint32_t shape = idesc_shape(UNIT);
      for (int u = u_begin; u < u_end && ok; ++u) {
        for (int s = s_begin; s < s_end && ok; ++s, ++it) {
          const int st = it & (NSTAGE - 1);
          ok = mbar_wait_warp(bar_full(st), (it / NSTAGE) & 1, abort_flag, p.status, LQ_STAGE_MMA);
          if (!ok) break;
          tc_fence_after();
          LQ_TL(EV_M_STAGE_FULL, s);
          const uint32_t a_addr = sm_stage + st * STAGE_BYTES, b_addr = a_addr + STAGE_A_BYTES;
          const uint64_t adesc = make_smem_desc(a_addr), bdesc = make_smem_desc(b_addr);
          // The stage's groups to the accumulators of one pair, as soon as the drain has read them out; one commit
          const int pair = it & (NPAIR - 1);
          const uint32_t d = tmem_base + 2 * pair * TCOLS;
          ok = mbar_wait_warp(bar_tempty(pair), ((it / NPAIR) & 1) ^ 1, abort_flag, p.status, LQ_STAGE_MMA);
          if (!ok) break;
          tc_fence_after();
          LQ_TL(EV_M_ACC_FREE, s);
          if (s < p.n_stages_main) {
            issue_group(d, adesc, bdesc, IDESC_F8 | shape);
            issue_group(d + TCOLS, adesc + 4, bdesc + 4, IDESC_F8 | shape, bar_tfull(pair), bar_empty(st));
          } else {
            if (elect_one()) {
              for (int j = 0; j < p.branch_mmas; ++j) {
                if (BRANCH == BRANCH_F16) tc_mma<TC_F16>(d, adesc + 2 * j, bdesc + 2 * j, IDESC_F16 | shape, (uint32_t)j);
                else tc_mma<TC_I8>(d, adesc + 2 * j, bdesc + 2 * j, IDESC_I8 | shape, (uint32_t)j);
              }
              tc_commit(bar_tfull(pair));
              tc_commit(bar_empty(st));
            }
            __syncwarp();
          }
          LQ_TL(EV_M_ISSUED, s);
        }
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(DRAIN_REGS));
    // ------------------------------------------------------------------ drain + epilogue
    const int quad = warp & 3;                          // tensor-memory lanes 32*quad .. 32*quad+31
    const int coff = ((warp - FIRST_DRAIN_WARP) >> 2) * WCOLS;   // which half of the tile's columns
    const uint32_t tlane = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)coff;
    const int fg = lane >> 2, ft = lane & 3;            // fragment coordinates
    const int row_at = 32 * quad + 4 * fg, col_at = coff + 4 * ft;    // this lane's places in the scale vectors
    uint32_t it = 0;                                    // operand stages since the kernel began: ring positions it & (NPAIR-1),
                                                        // it & (SC_RING-1)
    bool ok = true;
    Frag va[2], vb[2];                                  // two halves of groups: one being consumed, one being fetched
    auto pair_at = [&](uint32_t i) { return tlane + (i & (NPAIR - 1)) * (2 * TCOLS); };
    // Requests stage i's first half once its pair is complete (its scale vectors landed before its MMAs were issued).  The
    // request is made whatever the wait says, and even where no stage is left (it reads some accumulator, nothing looks at it).
    auto open_stage = [&](uint32_t i, bool exists) {
      if (exists) ok = mbar_wait_inline(bar_tfull(i & (NPAIR - 1)), (i / NPAIR) & 1, abort_flag, p.status, LQ_STAGE_DRAIN) && ok;
      tc_fence_after();
      fetch_half(pair_at(i), va);
    };
    // The stage's pair is in registers: it goes back, before the next request (the fence waits for every load that is in flight: 71.1 us for 64.0).
    auto give_back = [&](uint32_t i) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_tempty(i & (NPAIR - 1)));
    };
    Scales sc, sd;                                      // of the two groups of a stage
    auto load_scales_of = [&](Scales& sc, uint32_t i, int q) {
      const uint32_t at = sm_sc + (i & (SC_RING - 1)) * SC_STAGE_BYTES + q * SC_GROUP_FLOATS * 4;
      load_scales(sc, at + row_at * 4, at + (LQ_BM + col_at) * 4);
    };
    if constexpr (SPLIT) cluster_wait();                // the other CTAs' barriers are set up
    grid_dependency_wait();                             // Y may be what an earlier kernel still reads
    open_stage(0, u_begin < u_end);
    load_scales_of(sc, 0, 0);
    for (int u = u_begin; u < u_end && ok; ++u) {
      const int mb = u / p.units_n, nu = u - mb * p.units_n;
      const int m0 = mb * LQ_BM, n0 = nu * UNIT;
      LQ_TL(EV_TILE, 0);
      // this thread's 4 rows x 16 columns: acc[h][2 j + i] = rows 16 h + fg + 8 i, columns 16 ft + 2 j, + 1; from the bias
      float2 acc[2][16];
      {
        const float* bias = sc_ptr + (it & (SC_RING - 1)) * (SC_STAGE_BYTES / 4) + 2 * SC_GROUP_FLOATS + col_at;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float4 v = *reinterpret_cast<const float4*>(bias + 16 * k);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            acc[0][4 * k + i] = acc[1][4 * k + i] = make_float2(v.x, v.y);
            acc[0][4 * k + 2 + i] = acc[1][4 * k + 2 + i] = make_float2(v.z, v.w);
          }
          if (SPLIT && part != 0) {
#pragma unroll
            for (int j = 4 * k; j < 4 * k + 4; ++j) acc[0][j] = acc[1][j] = make_float2(0.f, 0.f);
          }
        }
      }
      const bool last_tile = u + 1 == u_end;
      const int s_main = SPLIT ? min(s_end, p.n_stages_main) : p.n_stages_main;
      for (int s = s_begin; s < s_main && ok; ++s, ++it) {
        const bool more = s + 1 < s_end || !last_tile;
        LQ_TL(EV_D_OPEN, s);
        tmem_ld_wait();
        LQ_TL(EV_D_WAITED, s);
        fetch_half(pair_at(it) + WCOLS / 2, vb);
        drain_half<false, 0>(va, acc, sc);
        tmem_ld_wait();
        fetch_half(pair_at(it) + TCOLS, va);
        load_scales_of(sd, it, 1);
        drain_half<false, 1>(vb, acc, sc);
        LQ_TL(EV_D_HALF, s);
        tmem_ld_wait();
        fetch_half(pair_at(it) + TCOLS + WCOLS / 2, vb);
        drain_half<false, 0>(va, acc, sd);
        tmem_ld_wait();
        give_back(it);
        LQ_TL(EV_D_LOADED, s);
        open_stage(it + 1, more);
        LQ_TL(EV_D_ACC_FULL, s);
        load_scales_of(sc, it + 1, 0);
        drain_half<false, 1>(vb, acc, sd);
        LQ_TL(EV_D_DONE, s);
        ok = __all_sync(0xffffffffu, ok);
      }
      if (!ok) break;
      if (BRANCH != BRANCH_NONE && (!SPLIT || s_end > p.n_stages_main)) {
        tmem_ld_wait();
        fetch_half(pair_at(it) + WCOLS / 2, vb);
        drain_half<BRANCH == BRANCH_I8, 0>(va, acc, sc);
        tmem_ld_wait();
        give_back(it);
        sd = sc;
        ++it;
        open_stage(it, !last_tile);
        load_scales_of(sc, it, 0);
        drain_half<BRANCH == BRANCH_I8, 1>(vb, acc, sd);
        ok = __all_sync(0xffffffffu, ok);
      }
      if (!ok) break;
      LQ_TL(EV_D_EPI_BEGIN, 0);
      if constexpr (SPLIT) {
        // the partial sums to the CTAs that add them up
        const int dwarp = warp - FIRST_DRAIN_WARP, row0 = m0 + 32 * quad;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            if (row0 + 8 * (2 * h + i) >= p.M) break;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int item = 4 * (2 * h + i) + k, to = item * p.split / GATHER_ITEMS;
              sts_v4(items_at(sm_stage, to, dwarp) + (uint32_t)((item - to * n_items) * 512 + lane * 16),
                     make_uint4(__float_as_uint(acc[h][4 * k + i].x), __float_as_uint(acc[h][4 * k + i].y),
                                __float_as_uint(acc[h][4 * k + 2 + i].x), __float_as_uint(acc[h][4 * k + 2 + i].y)));
            }
          }
        fence_proxy_async();
        __syncwarp();
        if (lane < p.split && lane != part) {            // a lane for each other CTA: the items that have a row
          int n = 0;
          for (int j = lane * n_items; j < (lane + 1) * n_items; ++j) n += row0 + 8 * (j >> 2) < p.M;
          if (n > 0)
            peer_copy(peer_smem(items_at(sm_gather, part, dwarp), lane), items_at(sm_stage, lane, dwarp), (uint32_t)n * 512,
                      peer_smem(bar_gather, lane));
        }
      } else {
        // Epilogue straight from registers: 16 neighbouring columns of four rows per lane, 128 of a row per quad.  Two lanes' stores of 16
        // bytes never meet in a 32-byte sector here, so each would write half of one; where all of Y's rows are whole sectors a lane
        // stores 32 bytes at once (us, M = 8192, K x N = 1152 x 3456: 78.0 -> 72.4).
        const int c = n0 + coff + 16 * ft;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int r = m0 + 32 * quad + 16 * h + 8 * i + fg;
            if (r >= p.M) continue;
            if (p.out_f32) {
              float* Y = reinterpret_cast<float*>(p.Y) + (size_t)r * p.N + c;
#pragma unroll
              for (int k = 0; k < 2; ++k) {
                uint32_t w[8];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  w[2 * j] = __float_as_uint(acc[h][8 * k + 2 * j + i].x);
                  w[2 * j + 1] = __float_as_uint(acc[h][8 * k + 2 * j + i].y);
                }
                if (c + 8 * k < p.N) stg_32<SECTORS>(Y + 8 * k, w);
              }
            } else {
              __half* Y = reinterpret_cast<__half*>(p.Y) + (size_t)r * p.N + c;
              uint32_t w[8];
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const __half2 q = __floats2half2_rn(acc[h][2 * j + i].x, acc[h][2 * j + i].y);
                w[j] = *reinterpret_cast<const uint32_t*>(&q);
              }
              if constexpr (SECTORS) {                      // (N is then a multiple of 16)
                if (c < p.N) stg_v8(Y, w);
              } else {
                if (c < p.N) *reinterpret_cast<uint4*>(Y) = make_uint4(w[0], w[1], w[2], w[3]);
                if (c + 8 < p.N) *reinterpret_cast<uint4*>(Y + 8) = make_uint4(w[4], w[5], w[6], w[7]);
              }
            }
          }
      }
      LQ_TL(EV_D_EPI_END, 0);
    }
    tmem_ld_wait();                                     // the last request
    drained = ok;
  }
  if constexpr (SPLIT) {
    // Every CTA of the cluster adds up its items, in the order of the stages, and stores them.
    if (warp < FIRST_DRAIN_WARP) cluster_wait();
    const bool gathered = drained && mbar_wait_warp<PEER_DATA>(bar_gather, 0, abort_flag, p.status, LQ_STAGE_DRAIN);
    if (warp >= FIRST_DRAIN_WARP && !gathered) mbar_settle(bar_gather, 0);
    cluster_arrive<false>();                            // nothing is on its way to this CTA any more
    if (gathered) {
      const int dwarp = warp - FIRST_DRAIN_WARP, mb = u_begin / p.units_n, nu = u_begin - mb * p.units_n;
      const int row = mb * LQ_BM + 32 * (warp & 3) + (lane >> 2), col = nu * UNIT + ((warp - FIRST_DRAIN_WARP) >> 2) * WCOLS + 16 * (lane & 3);
#pragma unroll 2
      for (int i = 0; i < n_items; i += 2) {                     // two items: eight columns
        const int j = part * n_items + i, r = row + 8 * (j >> 2), c = col + 4 * (j & 3);
        if (r >= p.M || c >= p.N) continue;
        float y[8] = {};
#pragma unroll 4
        for (int k = 0; k < p.split; ++k) {
          const uint32_t from = (k == part ? items_at(sm_stage, part, dwarp) : items_at(sm_gather, k, dwarp)) + (uint32_t)(i * 512 + lane * 16);
          const uint4 a = lds_v4(from), b = lds_v4(from + 512);
          y[0] += __uint_as_float(a.x); y[1] += __uint_as_float(a.y); y[2] += __uint_as_float(a.z); y[3] += __uint_as_float(a.w);
          y[4] += __uint_as_float(b.x); y[5] += __uint_as_float(b.y); y[6] += __uint_as_float(b.z); y[7] += __uint_as_float(b.w);
        }
        if (p.out_f32) {
          uint32_t w[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) w[k] = __float_as_uint(y[k]);
          float* Y = reinterpret_cast<float*>(p.Y) + (size_t)r * p.N + c;
          if (p.wide) stg_32<true>(Y, w);
          else stg_32<false>(Y, w);
        } else {
          uint32_t w[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const __half2 q = __floats2half2_rn(y[2 * k], y[2 * k + 1]);
            w[k] = *reinterpret_cast<const uint32_t*>(&q);
          }
          *reinterpret_cast<uint4*>(reinterpret_cast<__half*>(p.Y) + (size_t)r * p.N + c) = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
    }
  }

  // ---------------------------------------------------------------------- teardown
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
  // SPLIT: this CTA's own copies are read from its shared memory, and only who receives them knows when they have landed.  So it stays
  // until every CTA of the cluster has what it was to be sent, also where a wait has run out.  The stores of Y lie between arriving and
  // waiting.  (us, leaving at once / staying / staying, with an arrival that releases what was written: M x K x N = 1 x 1152 x 1152
  // 4.62 / 4.67 / 4.83, 120 x 1152 x 4608 7.43 / 7.52 / 7.66, 120 x 8192 x 1152 9.56 / 9.64 / 9.82.)
  if constexpr (SPLIT) cluster_wait();
}

// Self-test of the bounded wait: one warp waits on a barrier that nothing ever arrives on.
__global__ void lq_wait_probe_kernel(int32_t* status, long long limit) {
  __shared__ uint64_t barrier_word;
  __shared__ int abort_word;
  const uint32_t bar = smem_u32(&barrier_word);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    abort_word = 0;
    mbar_init_fence();
  }
  __syncwarp();
  mbar_wait_slow(bar, 0, &abort_word, status, LQ_STAGE_TEARDOWN, limit);
}

int g_clusters[64][3];                                // how many clusters of 2, 4, 8 the device holds at once

}  // namespace

lq_status lq_launch_wait_probe(int device, cudaStream_t st) {
  if (cudaSetDevice(device) != cudaSuccess) return LQ_ERR_CUDA;
  int32_t* status = lq_device_status_ptr(device);
  if (!status) return LQ_ERR_CUDA;
  lq_wait_probe_kernel<<<1, 32, 0, st>>>(status, 200000000ll);   // ~0.1 s
  return lq_note_cuda(cudaGetLastError()) == cudaSuccess ? LQ_OK : LQ_ERR_CUDA;
}

lq_status lq_gemm_prepare(int device) {
  if (cudaSetDevice(device) != cudaSuccess) return LQ_ERR_CUDA;
  for (auto* kernel : {lq_gemm_kernel<BRANCH_NONE, TILE_WHOLE>, lq_gemm_kernel<BRANCH_I8, TILE_WHOLE>, lq_gemm_kernel<BRANCH_F16, TILE_WHOLE>,
                       lq_gemm_kernel<BRANCH_NONE, TILE_SECTORS>, lq_gemm_kernel<BRANCH_I8, TILE_SECTORS>, lq_gemm_kernel<BRANCH_F16, TILE_SECTORS>,
                       lq_gemm_kernel<BRANCH_NONE, TILE_SPLIT>, lq_gemm_kernel<BRANCH_I8, TILE_SPLIT>, lq_gemm_kernel<BRANCH_F16, TILE_SPLIT>}) {
    cudaFuncAttributes at;
    if (lq_note_cuda(cudaFuncGetAttributes(&at, kernel)) != cudaSuccess) return LQ_ERR_CUDA;
    if (at.numRegs < LAUNCH_REGS) return LQ_ERR_UNSUPPORTED;
    if (lq_note_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES + GATHER_BYTES)) != cudaSuccess) return LQ_ERR_CUDA;
  }
  // once per device: launches of other threads read g_clusters without the lock, each after its own layer's upload came through here
  static std::mutex mu;
  static bool done[64] = {false};
  std::lock_guard<std::mutex> lk(mu);
  if (done[device & 63]) return LQ_OK;
  for (int i = 0; i < 3; ++i) {
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2u << i; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    lc.gridDim = dim3(2u << i); lc.blockDim = dim3(GEMM_THREADS); lc.dynamicSmemBytes = SMEM_BYTES + GATHER_BYTES; lc.attrs = at; lc.numAttrs = 1;
    if (lq_note_cuda(cudaOccupancyMaxActiveClusters(&g_clusters[device & 63][i], lq_gemm_kernel<BRANCH_I8, TILE_SPLIT>, &lc)) != cudaSuccess)
      return LQ_ERR_CUDA;
  }
  done[device & 63] = true;
  return LQ_OK;
}

lq_status lq_launch_gemm(const lq_layer* L, const lq_act* A, void* Y, lq_out_dtype dt, cudaStream_t st) {
  if (cudaSetDevice(A->device) != cudaSuccess) return LQ_ERR_CUDA;
  if (L->main_kind != LQ_KIND_E4M3) return LQ_ERR_UNSUPPORTED;
  GemmParams p;
  p.M = A->M; p.N = L->N; p.Mpad = A->Mpad; p.Npad = L->Npad;
  p.n_stages_main = L->Kpad / LQ_KSTAGE;
  p.branch_mmas = L->r == 0 ? 0 : (L->f16_branch ? lq_ceil_div(L->r, 16) : lq_ceil_div(L->r, 32));
  p.tiles_m = lq_ceil_div(A->M, LQ_BM);
  p.units_n = L->Npad / UNIT;
  p.sx = A->d_sx; p.sw = L->d_sw; p.sT = A->d_sT; p.sL2 = L->d_sL2; p.bias = L->d_bias;
  p.Y = Y; p.out_f32 = dt == LQ_OUT_F32 ? 1 : 0; p.wide = lq_rows_of_sectors(Y, L->N, dt);
  p.status = lq_device_status_ptr(A->device);
  if (!p.status) return LQ_ERR_CUDA;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, A->device) != cudaSuccess) return LQ_ERR_CUDA;
  int ctas = g_lq_gemm_ctas > 0 ? g_lq_gemm_ctas : sms;
  const long long units = (long long)p.tiles_m * p.units_n;
  // (by the whole call's rows, so that a row's sums are the same in every chunk of it)
  p.split = pick_split(A->M_call, (long long)lq_ceil_div(A->M_call, LQ_BM) * p.units_n, p.n_stages_main + (L->r > 0), ctas,
                       g_clusters[A->device & 63], g_lq_gemm_split);
  ctas = (int)std::min<long long>(ctas, units * p.split);
  auto kernel = [&](auto tile) {
    constexpr int T = decltype(tile)::value;
    return L->r == 0 ? lq_gemm_kernel<BRANCH_NONE, T> : L->f16_branch ? lq_gemm_kernel<BRANCH_F16, T> : lq_gemm_kernel<BRANCH_I8, T>;
  };
  auto* k = p.split > 1 ? kernel(std::integral_constant<int, TILE_SPLIT>())
            : lq_rows_of_sectors(Y, L->N, dt) ? kernel(std::integral_constant<int, TILE_SECTORS>())
                                              : kernel(std::integral_constant<int, TILE_WHOLE>());
  const size_t smem = SMEM_BYTES + (p.split > 1 ? GATHER_BYTES : 0);
  const cudaError_t e = lq_launch_cluster(k, ctas, GEMM_THREADS, p.split, smem, st, A->tmA, L->tmB, A->tmT, L->tmL2, p);
  return lq_note_cuda(e != cudaSuccess ? e : cudaGetLastError()) == cudaSuccess ? LQ_OK : LQ_ERR_CUDA;
}
