// MXINT4 variant of the layer's main product (Appendix A.3: blocks of 32 values with a power-of-two E8M0 scale;
// Table 2 quantizes the residual branch with it):
//
//   Y[m,n] = sum_b 2^(ex[m,b] + ew[b,n]) (qx_b Wq_b)[m,n] + sT[m] sL2[n] (tq L2q)[m,n] + bias[n]
//
// Here the tensor core applies the scales itself: tcgen05.mma kind::mxf8f6f4.block_scale takes one E8M0 scale
// per operand row and 32-deep K block from tensor memory, so ALL blocks of a tile accumulate into ONE fp32
// accumulator and nothing has to be drained per block.  The activations' codes ride in E4M3 operands as in the SINT4
// kernel, the weights' in packed E2M3 ones (MXFP4: E2M1).  Products q q' 2^(e+e') are exact in fp32; their sum is rounded by the tensor
// core's fp32 accumulation.
//
// Shape of the kernel (persistent, one CTA per SM, warp-specialised, 18 warps): tiles of 128 rows x W columns, W chosen by
// the launcher (pick_width).
//   warp 0      TMA producer: per stage 128 bytes of K of A (128 rows) and B (W rows) plus the stage's scale bytes (512 B per
//               128 rows: four K blocks, already in the 32 x 16-byte layout tensor memory wants); per tile one or two more
//               stages with the branch operands (tq, L2q) and the vectors sT, sL2, bias for the drain.  Weights do not depend
//               on earlier kernels: the first ring's worth is requested before the grid dependency is waited for
//   warp 1      owns tensor memory; per stage: tcgen05.cp of the scale bytes into tensor-memory columns, then four
//               K = 32 block-scaled MMAs into the tile's accumulator; after the last stage the low-rank branch's
//               up-projection: MX and fp16 branches onto the same accumulator, integer branches (U = tq L2q, kind::i8, exact
//               int32; fp32 scales that the tensor core cannot apply) into an accumulator of their own
//   warps 2-17  drain, 32 rows x 32 columns at a time: y = main + sT sL2 U + bias, convert, store.  The columns of a block
//               of 32 are permuted in the weight operand (lq_col32_slot) so that a lane's eight are neighbours in Y: 16
//               bytes of a row, no exchange
// Two accumulators alternate (with an integer branch: two and the branch's), so a tile's output leaves under the next tile's
// main loop: 2 W (3 W) columns and 12 for the scale factors of a stage (one slot: the tensor pipe executes one thread's
// tcgen05 copies and MMAs in issue order).  A single 256-column accumulator spent a third of a short-K launch on the
// hand-over and the stores behind it (M = 8192, K x N = 1152 x 3456, MXFP rank 64: 36.4 us, 28 without the stores).
// What bounds it: power.  The tensor pipe needs 2 W clocks a stage and the L2 delivers 70-78 bytes per clock and SM with all SMs
// at it, which at W = 192 and pairs comes to about the same; a stage takes 440 clocks of 384, at the 1.45-1.5 GHz that the
// power cap leaves (1.82 GHz with narrow tiles that keep the pipe waiting).  So bytes not moved count twice: pairs stage half
// the weights each, and the weights stay packed up to shared memory, 4 bits as e2m1 (MXFP4) or 6 as e2m3 (integer codes),
// where TMA spreads them out.  M = 8192, MXFP: 1152 x 3456 30.6 -> 29.4 us, 2240 x 6720 95.3 -> 91.1, 5600 x 2240 79.4 ->
// 75.5; integer codes 33.8 -> 33.4 and 51.3 -> 50.5.
// So do the weights that a pair needs for its next tile, too: where K is short enough they stay in shared memory, and the pair goes down its columns
// (RESIDENT; weights_stay has the rule).  6 % less time on average where it applies, and about as much under the power cap.
// What was measured on the way here (PixArt block, four GEMMs): the branch on mma.sync in the drain warps took tensor
// time from the main loop; TMA stores of the output (32 boxes of 2 KB, or 8 of 8 KB, per tile) cost 15 % against
// plain stores - they share the TMA unit with the operand loads.
// Every wait is bounded as in lq_gemm.cu.
#include <cuda_fp16.h>

#include <algorithm>

#include "lq_device.cuh"
#include "lq_gemm_mx_cut.h"

#ifdef LQ_TIMELINE
// Timeline build only: copies this kernel's stamp lists of the last launch to the host and clears them.
extern "C" int lq_debug_timeline_mx(unsigned long long* host_out) {
  if (cudaDeviceSynchronize() != cudaSuccess) return 1;
  if (cudaMemcpyFromSymbol(host_out, g_lq_timeline, sizeof(unsigned long long) * lqdev::TL_LISTS * lqdev::TL_CAP) != cudaSuccess) return 1;
  static unsigned long long zeros[lqdev::TL_LISTS][lqdev::TL_CAP];
  return cudaMemcpyToSymbol(g_lq_timeline, zeros, sizeof(zeros)) == cudaSuccess ? 0 : 1;
}
#endif

namespace {

using namespace lqdev;
using namespace lqmx;

constexpr int NUM_DRAIN_WARPS = 16;
constexpr int FIRST_DRAIN_WARP = 2;
constexpr int GEMM_THREADS = (FIRST_DRAIN_WARP + NUM_DRAIN_WARPS) * 32;
// tensor-memory columns: accumulators at 0 and W, the branch's at 2 W; 4 columns of A scales and 8 of B scales
constexpr int TM_SFA = 496, TM_SFB = TM_SFA + 4;

struct MxParams {
  int M, N, Npad;
  int k_stages;           // stages of A per tile: Kpad / 128, times two when 8-bit activation codes come as two digit planes
  int branch_steps;       // 0: no branch; else MMAs of the branch stage (32 bytes of r each)
  int branch_f16;         // the branch operands are halves (W16A16 reference branch): no scales, summed by the tensor core
  int branch_mx;          // the branch is MX as well: its up-projection is one more block-scaled stage onto the main
                          // accumulator.  1: MXFP elements, K blocks in order.  2: 8-bit integer codes as digit planes on
                          // both sides - the stage's four K blocks are (hi, 0), (hi, 1), (lo, 0), (lo, 1) and every
                          // (plane of T, plane of L2) pair of the same rank block is one MMA.  3: the same codes with 4-bit
                          // factors (one plane) and rank up to 128: two stages like mode 1, one per plane of T
  int tiles_m, tiles_n;
  int width, stages;      // W, operand ring depth
  int b_row;              // bytes of a weight row that a stage copies
  uint32_t b_format;      // format field of the weights in the instruction descriptor
  int b_wrap;             // Kpad / 128: stage s reads B (and its scales) at stage s mod b_wrap - the planes share the weights
  int b_slots;            // RESIDENT: places of B in shared memory, the branch's last
  const LqMxMaps* maps;   // of the layer, for this width; its scale bytes are rows of 512: sfb [Kpad/128][tiles_n][sf_chunks], sfl2 (branch_mx)
                          // [tiles_n][sf_chunks].  The activations': tmSfa [Mpad/128][k_stages], tmSft (branch_mx) [Mpad/128][1 or 2]
  int sf_chunks;          // ceil(W / 128)
  int block0;             // first row block of the launch in tmSfa and tmSft
  const float* sT;        // [Mpad]
  const float* sL2;       // [Npad]
  const float* bias;      // [Npad]
  void* Y;
  int out_f32;
  int wide;               // Y and its rows begin on 32-byte boundaries
  int32_t* status;
};

// A stage's instructions under one election, predicated instead of branched around: the control flow of the issuing warps stays
// uniform.  (With an `if` of one lane around them, stamps gave 320-370 clocks for the MMA warp's stage and 270 for the producer's;
// the MMAs of a stage take 2 W.)
//   main stage of the MMA warp: scale bytes to tensor memory, four K = 32 MMAs, the stage's return
__device__ __forceinline__ void issue_main_stage_one(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint64_t sfa, uint64_t sfb, uint32_t two,
                                                 uint32_t accumulate, uint32_t empty) {
  asm volatile(
      "{\n\t.reg .pred P, Q, T, A;\n\t"
      "elect.sync _|P, 0xffffffff;\n\t"
      "setp.ne.and.b32 Q, %12, 0, P;\n\t"
      "setp.ne.b32 A, %13, 0;\n\t"
      "setp.eq.b32 T, 0, 0;\n\t"
      "@P tcgen05.cp.cta_group::1.32x128b.warpx4 [%14], %9;\n\t"
      "@P tcgen05.cp.cta_group::1.32x128b.warpx4 [%15], %10;\n\t"
      "@Q tcgen05.cp.cta_group::1.32x128b.warpx4 [%16], %11;\n\t"
      "@P tcgen05.mma.cta_group::1.kind::mxf8f6f4.block_scale [%0], %1, %5, %17, [%14], [%15], A;\n\t"
      "@P tcgen05.mma.cta_group::1.kind::mxf8f6f4.block_scale [%0], %2, %6, %18, [%14], [%15], T;\n\t"
      "@P tcgen05.mma.cta_group::1.kind::mxf8f6f4.block_scale [%0], %3, %7, %19, [%14], [%15], T;\n\t"
      "@P tcgen05.mma.cta_group::1.kind::mxf8f6f4.block_scale [%0], %4, %8, %20, [%14], [%15], T;\n\t"
      "@P tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%21];\n\t}"
      ::"r"(d), "l"(a), "l"(a + 2), "l"(a + 4), "l"(a + 6), "l"(b), "l"(b + 2), "l"(b + 4), "l"(b + 6), "l"(sfa), "l"(sfb),
      "l"(sfb + (SF_BYTES >> 4)), "r"(two), "r"(accumulate), "r"((uint32_t)TM_SFA), "r"((uint32_t)TM_SFB), "r"((uint32_t)(TM_SFB + 4)),
      "r"(idesc), "r"(idesc | idesc_mx_ids(1)), "r"(idesc | idesc_mx_ids(2)), "r"(idesc | idesc_mx_ids(3)), "r"(empty)
      : "memory");
}
__device__ __forceinline__ void issue_main_stage_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint64_t sfa, uint64_t sfb, uint32_t two,
                                                 uint32_t accumulate, uint32_t empty) {
  asm volatile(
      "{\n\t.reg .pred P, Q, T, A;\n\t"
      "elect.sync _|P, 0xffffffff;\n\t"
      "setp.ne.and.b32 Q, %12, 0, P;\n\t"
      "setp.ne.b32 A, %13, 0;\n\t"
      "setp.eq.b32 T, 0, 0;\n\t"
      "@P tcgen05.cp.cta_group::2.32x128b.warpx4 [%14], %9;\n\t"
      "@P tcgen05.cp.cta_group::2.32x128b.warpx4 [%15], %10;\n\t"
      "@Q tcgen05.cp.cta_group::2.32x128b.warpx4 [%16], %11;\n\t"
      "@P tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale [%0], %1, %5, %17, [%14], [%15], A;\n\t"
      "@P tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale [%0], %2, %6, %18, [%14], [%15], T;\n\t"
      "@P tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale [%0], %3, %7, %19, [%14], [%15], T;\n\t"
      "@P tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale [%0], %4, %8, %20, [%14], [%15], T;\n\t"
      "@P tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%21], %22;\n\t}"
      ::"r"(d), "l"(a), "l"(a + 2), "l"(a + 4), "l"(a + 6), "l"(b), "l"(b + 2), "l"(b + 4), "l"(b + 6), "l"(sfa), "l"(sfb),
      "l"(sfb + (SF_BYTES >> 4)), "r"(two), "r"(accumulate), "r"((uint32_t)TM_SFA), "r"((uint32_t)TM_SFB), "r"((uint32_t)(TM_SFB + 4)),
      "r"(idesc), "r"(idesc | idesc_mx_ids(1)), "r"(idesc | idesc_mx_ids(2)), "r"(idesc | idesc_mx_ids(3)), "r"(empty), "h"((uint16_t)3)
      : "memory");
}
//   main stage of the producer: the weights' half, which announces the whole stage (tx bytes; 0: the pair's other CTA does) on
//   `own`, and the activations' half.  Copies complete on `full`.
#define LQ_LOAD_WEIGHTS(TMA)                                     \
  "{\n\t.reg .pred P, Q;\n\t"                                    \
  "elect.sync _|P, 0xffffffff;\n\t"                             \
  "setp.ne.and.b32 Q, %1, 0, P;\n\t"                            \
  "@Q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t" \
  "@P " TMA " [%3], [%4, {%5, %6}], [%2];\n\t"                  \
  "@P " TMA " [%7], [%8, {%9, %10}], [%2];\n\t}"
template <bool PAIR>
__device__ __forceinline__ void load_weights_stage(uint32_t own, uint32_t tx, uint32_t full, uint32_t dst, const CUtensorMap* tm, int x, int y,
                                                   uint32_t sf_dst, const CUtensorMap* tm_sf, int sf_row) {
  const uint64_t t = reinterpret_cast<uint64_t>(tm), ts = reinterpret_cast<uint64_t>(tm_sf);
  if constexpr (PAIR)
    asm volatile(LQ_LOAD_WEIGHTS(LQ_TMA_2D_PAIR) ::"r"(own), "r"(tx), "r"(full), "r"(dst), "l"(t), "r"(x), "r"(y), "r"(sf_dst), "l"(ts), "r"(0),
                 "r"(sf_row)
                 : "memory");
  else
    asm volatile(LQ_LOAD_WEIGHTS(LQ_TMA_2D) ::"r"(own), "r"(tx), "r"(full), "r"(dst), "l"(t), "r"(x), "r"(y), "r"(sf_dst), "l"(ts), "r"(0),
                 "r"(sf_row)
                 : "memory");
}
#define LQ_LOAD_ACTS(TMA)                        \
  "{\n\t.reg .pred P;\n\t"                       \
  "elect.sync _|P, 0xffffffff;\n\t"             \
  "@P " TMA " [%1], [%2, {%3, %4}], [%0];\n\t"  \
  "@P " TMA " [%5], [%6, {%7, %8}], [%0];\n\t}"
template <bool PAIR>
__device__ __forceinline__ void load_acts_stage(uint32_t full, uint32_t dst, const CUtensorMap* tm, int x, int y, uint32_t sf_dst, const CUtensorMap* tm_sf,
                                                int sf_row) {
  const uint64_t t = reinterpret_cast<uint64_t>(tm), ts = reinterpret_cast<uint64_t>(tm_sf);
  if constexpr (PAIR)
    asm volatile(LQ_LOAD_ACTS(LQ_TMA_2D_PAIR) ::"r"(full), "r"(dst), "l"(t), "r"(x), "r"(y), "r"(sf_dst), "l"(ts), "r"(0), "r"(sf_row) : "memory");
  else
    asm volatile(LQ_LOAD_ACTS(LQ_TMA_2D) ::"r"(full), "r"(dst), "l"(t), "r"(x), "r"(y), "r"(sf_dst), "l"(ts), "r"(0), "r"(sf_row) : "memory");
}

// BRANCH_ACC: the layer has an integer branch with fp32 scales, whose product needs an accumulator of its own.  The
// other instance (no branch, fp16 branch, MX branches) carries none of that code or its registers.
// PAIR: two CTAs of a cluster work on 256 rows x W columns (cta_group::2): each stages its own 128 rows of A and half of the
// tile's columns of B, and each SM's tensor core reads B from both.  Both CTAs' copies complete on the first one's barrier, whose
// CTA issues the MMAs for both.
// RESIDENT (pairs): a tile's columns of B - all stages of K, and the branch's - stay in shared memory while the pair goes through its run of tiles
// column by column; only A comes anew with every tile.
template <bool BRANCH_ACC, bool PAIR, bool RESIDENT>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
lq_gemm_mx_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmT,
                  const __grid_constant__ CUtensorMap tmSfa, const __grid_constant__ CUtensorMap tmSft,
                  const __grid_constant__ MxParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - smem_u32(smem_raw));
  const int W = p.width, NST = p.stages;
  constexpr int CTAS = PAIR ? 2 : 1;
  const int BW = W / CTAS;                                // columns of B in this CTA's shared memory
  const uint32_t rank = PAIR ? blockIdx.x & 1 : 0;
  const uint32_t b_bytes = (uint32_t)BW * LQ_KSTAGE, stage_bytes = STAGE_A_BYTES + (RESIDENT ? 0 : b_bytes);
  constexpr uint32_t SF_STAGE = RESIDENT ? SF_BYTES : STAGE_SF_BYTES, SFB_SLOT = STAGE_SF_BYTES - SF_BYTES;
  const uint32_t off_b = (uint32_t)NST * stage_bytes, off_sf = off_b + (RESIDENT ? p.b_slots * b_bytes : 0u), off_sfb = off_sf + NST * SF_STAGE;
  const uint32_t off_sc = off_sfb + (RESIDENT ? p.b_slots * SFB_SLOT : 0u), off_bar = off_sc + 2 * SC_FLOATS * 4;
  const uint32_t sm_stage = base, sm_sf = base + off_sf, sm_sc = base + off_sc, sm_bar = base + off_bar;
  // a stage's B and its scale bytes: in the ring's slot, or RESIDENT in their own
  auto b_at = [&](int st, int slot) { return RESIDENT ? base + off_b + (uint32_t)slot * b_bytes : sm_stage + (uint32_t)st * stage_bytes + STAGE_A_BYTES; };
  auto sfb_at = [&](int st, int slot) { return RESIDENT ? base + off_sfb + (uint32_t)slot * SFB_SLOT : sm_sf + (uint32_t)st * SF_STAGE + SF_BYTES; };
  const float* sc_ptr = reinterpret_cast<const float*>(smem + off_sc);
  uint8_t* bar_ptr = smem + off_bar;
  // barrier map (8 bytes each)
  constexpr int B_FULL = 0, B_EMPTY = MAX_STAGES, B_TFULL = 2 * MAX_STAGES, B_TEMPTY = B_TFULL + 2, B_RFULL = B_TEMPTY + 2,
                B_REMPTY = B_RFULL + 2, B_BEMPTY = B_REMPTY + 2, NBAR = B_BEMPTY + 1;
  auto bar = [&](int idx) { return sm_bar + 8u * (uint32_t)idx; };
  static_assert(NBAR * 8 + 16 <= SMEM_BAR_BYTES, "barrier area too small");
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_ptr + NBAR * 8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_ptr + NBAR * 8 + 8);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);   // provably warp-uniform
  const int lane = threadIdx.x & 31;
  const bool has_branch = p.branch_steps > 0;
  const int nbst = !has_branch ? 0 : p.branch_mx == 3 ? 2 : 1;             // stages of the branch per tile
  // this CTA's (pair's) contiguous run of tiles, row block major, RESIDENT column major
  const int unit = (int)blockIdx.x / CTAS, units = (int)gridDim.x / CTAS, blocks_m = (p.tiles_m + CTAS - 1) / CTAS;
  auto tile_at = [&](int w, int& mp, int& nu) {
    if (RESIDENT) { nu = w / blocks_m; mp = w - nu * blocks_m; }
    else { mp = w / p.tiles_n; nu = w - mp * p.tiles_n; }
  };
  const long long work = (long long)blocks_m * p.tiles_n;
  const int w_begin = (int)((work * unit) / units);
  const int w_end = (int)((work * (unit + 1)) / units);

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) { mbar_init(bar(B_FULL + s), 1); mbar_init(bar(B_EMPTY + s), 1); }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar(B_TFULL + b), 1); mbar_init(bar(B_TEMPTY + b), CTAS * NUM_DRAIN_WARPS);
      mbar_init(bar(B_RFULL + b), 1); mbar_init(bar(B_REMPTY + b), NUM_DRAIN_WARPS);
    }
    mbar_init(bar(B_BEMPTY), CTAS * NUM_DRAIN_WARPS);
    *abort_flag = 0;
    mbar_init_fence();
  }
  if (warp == 1) {
    if (PAIR) tmem_alloc_pair(smem_u32(tmem_slot), 512);
    else tmem_alloc(smem_u32(tmem_slot), 512);
  }
  tc_fence_before();
  if (PAIR) cluster_sync();
  else __syncthreads();
  tc_fence_after();
  grid_launch_dependents();
  // All 512 columns are this CTA's, so they start at 0.
  constexpr uint32_t tmem_base = 0;

  LQ_TL_DECL((blockIdx.x == 0 && lane == 0)
                 ? (warp == 0 ? (int)TL_PRODUCER : warp == 1 ? (int)TL_MMA : warp == FIRST_DRAIN_WARP ? (int)TL_DRAIN_FIRST
                    : warp == FIRST_DRAIN_WARP + NUM_DRAIN_WARPS - 1 ? (int)TL_DRAIN_LAST : -1)
                 : -1);

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    uint32_t tc = 0, rarmed = 0, par = 1;              // parity of the ring slot's "empty" barrier
    int st = 0, armed = 0;                             // ring slot; stages announced (up to the ring's depth)
    bool ok = true;
    const uint32_t sfb_bytes = (uint32_t)p.sf_chunks * SF_BYTES;
    const uint32_t first_bar = PAIR ? peer_smem(sm_bar, 0) : sm_bar;   // where the pair's copies complete
    auto full_bar = [&](int st) { return first_bar + 8u * (uint32_t)(B_FULL + st); };
    const uint32_t arm = rank == 0 ? CTAS : 0;         // CTAs whose bytes this one announces
    const int block_last = p.tiles_m - 1;
    // The weights' half of main stage s; announces the whole stage.  RESIDENT: only where they are not there yet.  (Their place is free:
    // the MMAs that read it last are at least as many stages back as the ring has slots, and the slot's own wait was for those.)
    auto load_b = [&](int st, int s, int nu, bool there) {
      const int sb = s >= p.b_wrap ? s - p.b_wrap : s; // the lo digits' plane runs over the same weights
      const uint32_t acts = STAGE_A_BYTES + SF_BYTES;
      if (RESIDENT && (there || s >= p.b_wrap)) {
        if (arm != 0 && elect_one()) mbar_expect_tx(bar(B_FULL + st), arm * acts);
        __syncwarp();
      } else {
        load_weights_stage<PAIR>(bar(B_FULL + st), arm * (acts + (uint32_t)BW * p.b_row + sfb_bytes), full_bar(st), b_at(st, sb), &p.maps->b, sb * LQ_KSTAGE,
                                 nu * W + (int)rank * BW, sfb_at(st, sb), &p.maps->sfb, (sb * p.tiles_n + nu) * p.sf_chunks);
      }
    };
    auto load_a = [&](int st, int s, int mb) {
      load_acts_stage<PAIR>(full_bar(st), sm_stage + st * stage_bytes, &tmA, s * LQ_KSTAGE, mb * LQ_BM, sm_sf + st * SF_STAGE, &tmSfa,
                            (p.block0 + min(mb, block_last)) * p.k_stages + s);
    };
    auto advance = [&]() {
      ++armed;
      if (++st == NST) { st = 0; par ^= 1; }
    };
    int early = 0;                                     // stages of the first tile whose weights were requested ahead
    int mp, nu, nu_there = -1;                         // nu_there: whose weights are resident
    if (w_begin < w_end) {
      tile_at(w_begin, mp, nu);
      early = min(NST, p.k_stages);
      for (int s = 0; s < early; ++s) load_b(s, s, nu, false);
    }
    grid_dependency_wait();
    for (int w = w_begin; w < w_end && ok; ++w, ++tc) {
      tile_at(w, mp, nu);
      const int mb = mp * CTAS + (int)rank;            // (a pair's second block may not exist)
      const bool there = RESIDENT && nu == nu_there;
      nu_there = nu;
      const int m0 = mb * LQ_BM, n0 = nu * W, mc = min(mb, block_last);
      for (int s = 0; s < p.k_stages; ++s) {
        const bool ahead = tc == 0 && s < early;
        if (!ahead) {
          ok = mbar_wait_warp(bar(B_EMPTY + st), par, abort_flag, p.status, LQ_STAGE_PRODUCER);
          if (!ok) break;
        }
        LQ_TL(EV_P_SLOT_FREE, s);
        if (!ahead) load_b(st, s, nu, there);
        load_a(st, s, mb);
        advance();
        LQ_TL(EV_P_ISSUED, s);
      }
      // the branch operands: the containers of tq (128 rows) and L2q (W rows), r contiguous; mode 3 brings the two
      // digit planes of tq as two stages against the same L2q
      for (int bs = 0; bs < nbst && ok; ++bs) {
        ok = mbar_wait_warp(bar(B_EMPTY + st), par, abort_flag, p.status, LQ_STAGE_PRODUCER);
        if (!ok) break;
        const uint32_t a_dst = sm_stage + st * stage_bytes, full = full_bar(st);
        const bool fetch = !RESIDENT || (!there && bs == 0);
        if (elect_one()) {
          const uint32_t acts = STAGE_A_BYTES + (p.branch_mx ? SF_BYTES : 0), weights = b_bytes + (p.branch_mx ? sfb_bytes : 0);
          if (arm != 0) mbar_expect_tx(bar(B_FULL + st), arm * (acts + (fetch ? weights : 0u)));
          tma_load_2d<PAIR>(a_dst, &tmT, bs * LQ_KSTAGE, m0, full);
          if (fetch) tma_load_2d<PAIR>(b_at(st, p.b_wrap), &p.maps->l2, 0, n0 + (int)rank * BW, full);
          if (p.branch_mx) {   // the block scales of T (rows) and of L2 (columns) along the rank
            tma_load_2d<PAIR>(sm_sf + st * SF_STAGE, &tmSft, 0, (p.block0 + mc) * nbst + bs, full);
            if (fetch) tma_load_2d<PAIR>(sfb_at(st, p.b_wrap), &p.maps->sfl2, 0, nu * p.sf_chunks, full);
          }
        }
        __syncwarp();
        advance();
      }
      if (!ok) break;
      {   // the tile's scale vectors and bias, for the drain
        const int rb = tc & 1;
        ok = mbar_wait_warp(bar(B_REMPTY + rb), ((tc >> 1) & 1) ^ 1, abort_flag, p.status, LQ_STAGE_PRODUCER);
        if (!ok) break;
        if (elect_one()) {
          const uint32_t rfull = bar(B_RFULL + rb), dst = sm_sc + rb * SC_FLOATS * 4, cb = (uint32_t)min(W, p.Npad - n0) * 4;
          mbar_expect_tx(rfull, LQ_BM * 4 + 2 * cb);
          bulk_load(dst, p.sT + mc * LQ_BM, LQ_BM * 4, rfull);
          bulk_load(dst + LQ_BM * 4, p.sL2 + n0, cb, rfull);
          bulk_load(dst + (LQ_BM + MAX_W) * 4, p.bias + n0, cb, rfull);
        }
        __syncwarp();
        ++rarmed;
      }
    }
    if (!ok && lane == 0) {
      // aborting: give the copies already issued a bounded time to land before the CTA's shared memory goes away
      // (the pair's second CTA cannot see its own: a barrier of its that nothing completes gives them that time)
      if (rank != 0) mbar_settle(bar(B_FULL), 0);
      for (int i = rank != 0 ? 0 : max(min(armed, NST), early); i > 0; --i) {
        if (--st < 0) { st = NST - 1; par ^= 1; }
        mbar_settle(bar(B_FULL + st), par ^ 1);
      }
      for (uint32_t i = 1; i <= min(rarmed, 2u); ++i) {                 // and the tiles' scale vectors
        const uint32_t j = rarmed - i;
        mbar_settle(bar(B_RFULL + (int)(j & 1)), (j >> 1) & 1);
      }
    }
  } else if (warp == 1 && rank != 0) {
    // the pair's first CTA issues for both
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    uint32_t tc = 0, par = 0;
    int st = 0;                                        // ring slot and its parity
    bool ok = true;
    const uint32_t tsfa = tmem_base + TM_SFA, tsfb = tmem_base + TM_SFB;
    auto copy_scales = [&](int st, int slot) {
      const uint32_t sfb = sfb_at(st, slot);
      auto cp = [&](uint32_t to, uint32_t from) {
        if (PAIR) tc_cp_sf_pair(to, make_smem_desc_plain(from, 16, 128));
        else tc_cp_sf(to, make_smem_desc_plain(from, 16, 128));
      };
      cp(tsfa, sm_sf + st * SF_STAGE);
      cp(tsfb, sfb);
      if (p.sf_chunks == 2) cp(tsfb + 4, sfb + SF_BYTES);
    };
    auto mma_mx = [&](uint32_t d, uint64_t a, uint64_t b, uint32_t idesc) {
      if (PAIR) tc_mma_mx_pair(d, a, b, idesc, tsfa, tsfb, 1u);
      else tc_mma_mx(d, a, b, idesc, tsfa, tsfb, 1u);
    };
    auto commit = [&](uint32_t b) {
      if (PAIR) tc_commit_pair(b);
      else tc_commit(b);
    };
    constexpr uint32_t ROWS256 = PAIR ? (uint32_t)(LQ_BM >> 4) << 24 : 0;    // added to a 128-row descriptor's M field: 256
    auto stage_full = [&]() { return mbar_wait_warp(bar(B_FULL + st), par, abort_flag, p.status, LQ_STAGE_MMA); };
    for (int w = w_begin; w < w_end && ok; ++w, ++tc) {
      const int buf = tc & 1;
      const uint32_t d = tmem_base + (uint32_t)(buf * W);
      // the accumulator is free once the drain has read the tile before last out of it
      ok = mbar_wait_warp<PAIR>(bar(B_TEMPTY + buf), ((tc >> 1) & 1) ^ 1, abort_flag, p.status, LQ_STAGE_MMA);
      if (!ok) break;
      tc_fence_after();
      LQ_TL(EV_M_ACC_FREE, 0);
      for (int s = 0; s < p.k_stages; ++s) {
        ok = stage_full();
        if (!ok) break;
        tc_fence_after();
        LQ_TL(EV_M_STAGE_FULL, s);
        const int sb = s >= p.b_wrap ? s - p.b_wrap : s;
        const uint64_t adesc = make_smem_desc(sm_stage + st * stage_bytes), bdesc = make_smem_desc(b_at(st, sb));
        auto issue = PAIR ? issue_main_stage_pair : issue_main_stage_one;
        issue(d, adesc, bdesc, (idesc_mx(W, 0) | p.b_format) + ROWS256, make_smem_desc_plain(sm_sf + st * SF_STAGE, 16, 128),
              make_smem_desc_plain(sfb_at(st, sb), 16, 128),
              (uint32_t)(p.sf_chunks == 2), (uint32_t)s, bar(B_EMPTY + st));
        if (++st == NST) { st = 0; par ^= 1; }
        LQ_TL(EV_M_ISSUED, s);
      }
      for (int bs = 0; bs < nbst && ok; ++bs) {
        ok = stage_full();
        if (!ok) break;
        if (BRANCH_ACC) {
          // the drain has read the previous tile's branch accumulator (long ago: it does that under this tile's main loop)
          ok = mbar_wait_warp<PAIR>(bar(B_BEMPTY), (tc & 1) ^ 1, abort_flag, p.status, LQ_STAGE_MMA);
          if (!ok) break;
        }
        tc_fence_after();
        const uint64_t adesc = make_smem_desc(sm_stage + st * stage_bytes), bdesc = make_smem_desc(b_at(st, p.b_wrap));
        if (elect_one()) {
          if (p.branch_mx) {
            copy_scales(st, p.b_wrap);
            if (p.branch_mx == 2) {
              for (int c = 0; c < p.branch_steps; ++c)
                for (int q = 0; q < 4; ++q) {
                  const int ja = c + 2 * (q >> 1), jb = c + 2 * (q & 1);   // K block of T's plane, of L2's plane
                  mma_mx(d, adesc + 2 * ja, bdesc + 2 * jb, idesc_mx2(W, ja, jb) + ROWS256);
                }
            } else {
              for (int j = 0; j < p.branch_steps; ++j)
                mma_mx(d, adesc + 2 * j, bdesc + 2 * j, idesc_mx(W, j) + ROWS256);
            }
          } else {
            for (int j = 0; j < p.branch_steps; ++j) {
              constexpr int KIND = BRANCH_ACC ? TC_I8 : TC_F16;                // (16 halves each)
              const uint32_t to = BRANCH_ACC ? tmem_base + 2 * W : d, idesc = (BRANCH_ACC ? IDESC_I8 : IDESC_F16) + idesc_shape(W) + ROWS256;
              if (PAIR) tc_mma_pair<KIND>(to, adesc + 2 * j, bdesc + 2 * j, idesc, BRANCH_ACC ? (uint32_t)j : 1u);
              else tc_mma<KIND>(to, adesc + 2 * j, bdesc + 2 * j, idesc, BRANCH_ACC ? (uint32_t)j : 1u);
            }
          }
          commit(bar(B_EMPTY + st));
        }
        __syncwarp();
        if (++st == NST) { st = 0; par ^= 1; }
      }
      if (!ok) break;
      if (elect_one()) commit(bar(B_TFULL + buf));
      __syncwarp();
      LQ_TL(EV_TILE, 0);
    }
  } else {
    // ------------------------------------------------------------------ drain + epilogue
    const int quad = warp & 3;                          // tensor-memory lanes 32*quad .. 32*quad+31
    const int cgi = (warp - FIRST_DRAIN_WARP) >> 2;     // blocks of 32 columns cgi, cgi + 4
    const int g = lane >> 2, t = lane & 3;              // fragment coordinates: rows g + 8 i, eight columns from 8 t
    const uint32_t tlane = tmem_base + ((uint32_t)(quad * 32) << 16);
    const int blocks = W >> 5;
    auto give_back = [&](uint32_t b) {                  // to the issuer, which sits in the pair's first CTA
      if (PAIR) peer_arrive(peer_smem(b, 0));
      else mbar_arrive(b);
    };
    uint32_t tc = 0;
    bool ok = true;
    grid_dependency_wait();                             // Y may be what an earlier kernel still reads
    for (int w = w_begin; w < w_end && ok; ++w, ++tc) {
      int mp, nu;
      tile_at(w, mp, nu);
      const int mb = mp * CTAS + (int)rank, buf = tc & 1;
      LQ_TL(EV_D_OPEN, 0);
      ok = mbar_wait_warp(bar(B_TFULL + buf), (tc >> 1) & 1, abort_flag, p.status, LQ_STAGE_DRAIN) &&
           mbar_wait_warp(bar(B_RFULL + buf), (tc >> 1) & 1, abort_flag, p.status, LQ_STAGE_DRAIN);
      if (!ok) break;
      tc_fence_after();
      LQ_TL(EV_D_ACC_FULL, 0);
      const float* sc = sc_ptr + buf * SC_FLOATS;
      const int row0 = quad * 32 + g;                   // this thread's rows inside the tile: row0 + 8 i
#pragma unroll 1
      for (int b = cgi; b < blocks; b += 4) {
        uint32_t v[2][16], u[BRANCH_ACC ? 2 : 1][16];
#pragma unroll
        for (int h = 0; h < 2; ++h) tmem_ld_16x256b_x4(tlane + ((uint32_t)(16 * h) << 16) + buf * W + 32 * b, v[h]);
        if constexpr (BRANCH_ACC) {
#pragma unroll
          for (int h = 0; h < 2; ++h) tmem_ld_16x256b_x4(tlane + ((uint32_t)(16 * h) << 16) + 2 * W + 32 * b, u[h]);
        }
        const float* cb = sc + LQ_BM + MAX_W + 32 * b + 8 * t;
        const float4 b0 = *reinterpret_cast<const float4*>(cb), b1 = *reinterpret_cast<const float4*>(cb + 4);
        const float bias[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
        float sl[8];
        if constexpr (BRANCH_ACC) {
          const float4 l0 = *reinterpret_cast<const float4*>(cb - MAX_W), l1 = *reinterpret_cast<const float4*>(cb - MAX_W + 4);
          sl[0] = l0.x; sl[1] = l0.y; sl[2] = l0.z; sl[3] = l0.w; sl[4] = l1.x; sl[5] = l1.y; sl[6] = l1.z; sl[7] = l1.w;
        }
        tmem_ld_wait();
        if (b + 4 >= blocks) {                          // this warp's last block: the accumulators go back
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            give_back(bar(B_TEMPTY + buf));
            if (BRANCH_ACC) give_back(bar(B_BEMPTY));
          }
          LQ_TL(EV_D_LOADED, 0);
        }
        const int c = nu * W + 32 * b + 8 * t;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          // fragment registers 4 j .. 4 j + 3: row g, columns 2 j, 2 j + 1 of this lane's eight, then row g + 8 the same columns.
          // U is an exact int32 with |U| < 2^22: converted exactly with the 1.5 * 2^23 trick
          const int h = i >> 1, q = 2 * (i & 1), r = mb * LQ_BM + row0 + 8 * i;
          float y[8];
          const float st = BRANCH_ACC ? sc[row0 + 8 * i] : 0.f;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            y[j] = __uint_as_float(v[h][4 * (j >> 1) + q + (j & 1)]) + bias[j];
            if constexpr (BRANCH_ACC)
              y[j] = fmaf(__int_as_float((int)u[h][4 * (j >> 1) + q + (j & 1)] + 0x4B400000) - 12582912.0f, st * sl[j], y[j]);
          }
          if (r < p.M && c < p.N) {
            if (p.out_f32) {                                // (whole sectors; us, M = 1365, 1160 x 2312: 12.0 by 16 bytes, 9.9 so)
              uint32_t o[8];
#pragma unroll
              for (int j = 0; j < 8; ++j) o[j] = __float_as_uint(y[j]);
              float* Y = reinterpret_cast<float*>(p.Y) + (size_t)r * p.N + c;
              if (p.wide) stg_32<true>(Y, o);
              else stg_32<false>(Y, o);
            } else {
              uint32_t o[4];
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const __half2 x = __floats2half2_rn(y[2 * j], y[2 * j + 1]);
                o[j] = *reinterpret_cast<const uint32_t*>(&x);
              }
              *reinterpret_cast<uint4*>(reinterpret_cast<__half*>(p.Y) + (size_t)r * p.N + c) = make_uint4(o[0], o[1], o[2], o[3]);
            }
          }
        }
      }
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(bar(B_REMPTY + buf));
        if (cgi >= blocks) {                            // a tile narrower than 128 columns has nothing for this warp
          give_back(bar(B_TEMPTY + buf));
          if (BRANCH_ACC) give_back(bar(B_BEMPTY));
        }
      }
      LQ_TL(EV_D_EPI_END, 0);
    }
  }

  // ---------------------------------------------------------------------- teardown
  tc_fence_before();
  if (PAIR) cluster_sync();      // the peer's MMAs and arrivals reach into this CTA's shared memory until here
  else __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    if (PAIR) tmem_dealloc_pair(tmem_base, 512);
    else tmem_dealloc(tmem_base, 512);
  }
}

}  // namespace

lq_status lq_gemm_mx_prepare(int device) {
  if (cudaSetDevice(device) != cudaSuccess) return LQ_ERR_CUDA;
  for (auto* kernel : {lq_gemm_mx_kernel<false, false, false>, lq_gemm_mx_kernel<true, false, false>, lq_gemm_mx_kernel<false, true, false>,
                       lq_gemm_mx_kernel<true, true, false>, lq_gemm_mx_kernel<false, true, true>, lq_gemm_mx_kernel<true, true, true>})
    if (lq_note_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM)) != cudaSuccess) return LQ_ERR_CUDA;
  return LQ_OK;
}

lq_status lq_launch_gemm_mx(const lq_layer* L, const lq_act* A, void* Y, lq_out_dtype dt, cudaStream_t st) {
  if (cudaSetDevice(A->device) != cudaSuccess) return LQ_ERR_CUDA;
  if (!L->mx || !A->mx) return LQ_ERR_UNSUPPORTED;
  MxParams p;
  p.M = A->M; p.N = L->N; p.Npad = L->Npad;
  p.b_wrap = L->Kpad / LQ_KSTAGE;
  p.k_stages = p.b_wrap * A->planes;
  p.branch_f16 = L->f16_branch ? 1 : 0;
  p.branch_mx = L->r == 0 ? 0 : L->mxfp ? 1 : !L->a8 ? 0 : L->cfg.branch == LQ_BRANCH_MXINT4 ? 3 : 2;
  p.branch_steps = L->r == 0 ? 0 : lq_ceil_div(L->r, L->f16_branch ? 16 : 32);   // a8: rank blocks of 32 (at most two)
  p.tiles_m = lq_ceil_div(A->M, LQ_BM);
  p.status = lq_device_status_ptr(A->device);
  if (!p.status) return LQ_ERR_CUDA;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, A->device) != cudaSuccess) return LQ_ERR_CUDA;
  const bool acc = p.branch_steps > 0 && !p.branch_f16 && !p.branch_mx;
  const MxShape shape = {A->M, L->N, p.b_wrap, A->planes, L->r > 0, acc, lq_mx_weight_bits(L), dt == LQ_OUT_F32 ? 4 : 2};
  MxCut cut;
  if (!plan_mx(shape, g_lq_gemm_ctas > 0 ? g_lq_gemm_ctas : sms, g_lq_gemm_width, g_lq_gemm_pair != 0, cut) || !L->d_sfbw[cut.width_index])
    return LQ_ERR_INVALID_ARG;
  p.width = cut.width; p.stages = cut.stages; p.b_slots = cut.b_slots; p.tiles_n = cut.tiles_n; p.sf_chunks = lq_ceil_div(p.width, 128);
  p.b_row = LQ_KSTAGE / 8 * lq_mx_weight_bits(L); p.b_format = L->mxfp ? IDESC_MX_B_E2M1 : IDESC_MX_B_E2M3;
  p.block0 = A->block0;
  p.sT = A->d_sT; p.sL2 = L->d_sL2; p.bias = L->d_bias;
  p.Y = Y; p.out_f32 = dt == LQ_OUT_F32 ? 1 : 0; p.wide = lq_rows_of_sectors(Y, L->N, dt);
  auto* kernel = cut.resident ? (acc ? lq_gemm_mx_kernel<true, true, true> : lq_gemm_mx_kernel<false, true, true>)
                 : acc        ? (cut.pair ? lq_gemm_mx_kernel<true, true, false> : lq_gemm_mx_kernel<true, false, false>)
                              : (cut.pair ? lq_gemm_mx_kernel<false, true, false> : lq_gemm_mx_kernel<false, false, false>);
  p.maps = L->d_maps + 2 * cut.width_index + cut.pair;
  const cudaError_t e = lq_launch_cluster(kernel, cut.ctas, GEMM_THREADS, 1 + cut.pair, (size_t)cut.smem, st, A->tmA, A->tmT, A->tmSfa, A->tmSft, p);
  return lq_note_cuda(e != cudaSuccess ? e : cudaGetLastError()) == cudaSuccess ? LQ_OK : LQ_ERR_CUDA;
}
