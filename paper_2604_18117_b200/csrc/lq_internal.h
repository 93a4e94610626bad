// Internal declarations shared by the library's translation units (not part of the C ABI).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "lq.h"

#define LQ_GROUP 64
#define LQ_MX_BLOCK 32          // MXINT4: blocks of 32 with a power-of-two (E8M0) scale
#define LQ_BM 128            // rows per output tile (one tcgen05 MMA, M = 128)
#define LQ_BN 128            // columns per output tile
#define LQ_KSTAGE 128        // bytes of K per shared-memory stage row (two groups of 64 codes)
#define LQ_RCONT 128         // bytes per row of the branch containers (tq, L2q): rank <= 128
#define LQ_MAX_K 8192
#define LQ_MAX_RANK 128
#define LQ_HOST_CHUNKS 8       // row chunks (at most) lq_linear_forward_host overlaps (copy in / compute / copy out)

// role identifiers reported through the device status word
enum { LQ_STAGE_NONE = 0, LQ_STAGE_PRODUCER = 1, LQ_STAGE_MMA = 2, LQ_STAGE_DRAIN = 3, LQ_STAGE_TEARDOWN = 4, LQ_STAGE_QUANT = 5 };

enum { LQ_KIND_I8 = 0, LQ_KIND_E4M3 = 1 };

static inline int lq_ceil_div(int a, int b) { return (a + b - 1) / b; }
static inline int lq_round_up(int a, int b) { return lq_ceil_div(a, b) * b; }

// offset of the scale byte of row (or column) i and 32-block kb inside its [tile][kb/4] chunk of 512 bytes
static inline size_t lq_sf_offset(int i, int kb, int Kpad) {
  return ((size_t)(i / 128) * (Kpad / 128) + kb / 4) * 512 + 16 * (i % 32) + 4 * ((i % 128) / 32) + kb % 4;
}

// Tile widths the MX GEMM is launched with.  Layers with an integer branch, whose product needs a third accumulator in tensor
// memory, go up to 160 columns, the others up to 224.
constexpr int LQ_MX_WIDTHS[] = {64, 128, 160, 192, 224};
constexpr int LQ_MX_NWIDTHS = 5;
static inline bool lq_mx_width_used(int width, bool branch_acc) { return branch_acc ? width <= 160 : width != 160; }
// the same for the weight scales of operand row n when the columns are cut in `tiles` tiles of `width`: chunks [kb/4][tile][half]
static inline size_t lq_sfb_offset(int n, int kb, int width, int tiles) {
  const int i = n % width, chunks = lq_ceil_div(width, 128);
  return (((size_t)(kb / 4) * tiles + n / width) * chunks + i / 128) * 512 + 16 * (i % 32) + 4 * ((i % 128) / 32) + kb % 4;
}

// Orders the GEMMs' operands are laid out in, for the accumulator fragments its drain lanes hold (rows g, g + 8, g + 16,
// g + 24 of 32; columns 8 j + 2 t + {0, 1} of 64):
//   place of row m in the row-scale vectors: a lane's four are neighbours
__host__ __device__ static inline int lq_row_slot(int m) { return (m & ~31) | ((m & 7) << 2) | ((m >> 3) & 3); }
//   row of the weight operand that carries output column n: a lane's 16 columns are neighbours in the output
static inline int lq_col_slot(int n) { return (n & ~63) | (((n >> 1) & 7) << 3) | (((n >> 4) & 3) << 1) | (n & 1); }
//   the same for the MX GEMM, whose lanes hold eight columns of 32
static inline int lq_col32_slot(int n) { return (n & ~31) | (((n >> 1) & 3) << 3) | (((n >> 3) & 3) << 1) | (n & 1); }
//   place of column n in the column-scale vectors and the bias: a lane's come in four 16-byte loads, neighbours across lanes
static inline int lq_colscale_slot(int n) { return (n & ~63) | (((n >> 2) & 3) << 4) | (((n >> 4) & 3) << 2) | (n & 3); }

static inline bool lq_branch_is_mxfp(int branch) {
  return branch == LQ_BRANCH_MXFP8 || branch == LQ_BRANCH_MXFP6 || branch == LQ_BRANCH_MXFP4;
}
// An 8-bit code c in [-127, 127] as two digits, c = 16 hi + lo with lo in [-8, 7] and hi in [-8, 8]: both are exact
// E4M3 values, so a block-scaled MMA can carry an 8-bit integer operand as two planes with scales 2^(e+4) and 2^e.
static inline void lq_split_digits(int c, int* hi, int* lo) {
  const int l = ((c + 8) & 15) - 8;
  *lo = l; *hi = (c - l) / 16;
}
// E4M3 byte of an integer in [-8, 8] (bias 7, three mantissa bits; 8 = 1.0 * 2^3)
static inline uint8_t lq_digit_e4m3(int d) {
  static const uint8_t mag[9] = {0x00, 0x38, 0x40, 0x44, 0x48, 0x4A, 0x4C, 0x4E, 0x50};
  return (uint8_t)((d < 0 ? 0x80 : 0x00) | mag[d < 0 ? -d : d]);
}
static inline bool lq_branch_is_mxint(int branch) { return branch == LQ_BRANCH_MXINT8 || branch == LQ_BRANCH_MXINT4; }
static inline int lq_branch_wbits(int branch) {
  return branch == LQ_BRANCH_W8A8 ? 8 : branch == LQ_BRANCH_W6A6 ? 6 : branch == LQ_BRANCH_W4A8 ? 4 : 0;
}
static inline int lq_branch_abits(int branch) {
  return branch == LQ_BRANCH_W8A8 ? 8 : branch == LQ_BRANCH_W6A6 ? 6 : branch == LQ_BRANCH_W4A8 ? 8 : 0;
}

// Tensor maps of an MX layer for one tile width, in device memory: as launch parameters four maps more cost the calling thread 0.4 us
struct LqMxMaps {
  CUtensorMap b, l2;           // over d_Wq8 and d_L2c, box [width][128B] (pairs: half the width), 128B swizzle
  CUtensorMap sfb, sfl2;       // over d_sfbw and d_sfl2w, rows of 512 bytes, box [ceil(width/128)] rows
};

struct lq_layer {
  lq_config cfg;
  int K, N, r, G;          // logical sizes
  int Kpad, Npad, Gpad;    // Kpad: multiple of 128; Npad: multiple of LQ_BN; Gpad = Kpad / 64
  bool integer_branch, f16_branch, has_bias;
  bool mx;                     // MX main branch (cfg.group == 32): G counts blocks of 32, sw holds powers of two
  bool mxfp;                   // MXFP4 weights x MXFP8e4 activations (implies mx); the branch, if any, is MXFP too
  bool a8;                     // MXINT4 weights x MXINT8 activations (implies mx): 8-bit codes travel as two E4M3 digit
                               // planes (hi, lo); factors: int8 codes in L1q / L2q with block scales in s1b / s2b
  std::vector<uint8_t> Wq8h;   // mxfp: [K][N] e4m3 bytes of the e2m1 weight elements
  std::vector<uint8_t> L1e, L2e;   // mxfp: e4m3 bytes of the factor elements, [K][r] and [r][N]
  std::vector<float> s1b, s2b; // mxfp: block scales 2^e of L1 [ceil(K/32)][r] and of L2 [ceil(r/32)][N]
  // host copy, canonical layouts
  std::vector<int8_t> Wq;      // [K][N]
  std::vector<uint16_t> sw;    // [G][N] half bits
  std::vector<int8_t> L1q;     // [K][r]
  std::vector<int8_t> L2q;     // [r][N]
  std::vector<float> sL1, sL2; // [r], [N]
  std::vector<uint16_t> L1h;   // [K][r] half bits (W16A16)
  std::vector<uint16_t> L2h;   // [r][N]
  std::vector<uint16_t> bias;  // [N]
  // device copy, operand layouts
  int device;
  int main_kind;               // LQ_KIND_*: byte encoding of the 4-bit codes in the MMA operands
  uint8_t* d_Wq8;              // MX: packed, [Npad][Kpad] e2m1 (mxfp) or e2m3 elements; SINT4: [Npad][Kpad] e4m3 bytes, K contiguous
                               // (B operand, K-major; rows in lq_col_slot order, MX: lq_col32_slot)
  float* d_sw;                 // [Gpad][Npad] fp32 (exact images of the fp16 scales), in lq_colscale_slot order
  uint8_t* d_L1c;              // [planes * rn][Kpad] bytes (W16A16: [rn][Kpad] halves), K contiguous: first factor as the B operand of
                               // the down-projection; rn = lq_l1_rows; MXINT8 factors: the hi digits' rows, then the lo digits'
  uint8_t* d_sfl1;             // MX branches: E8M0 bytes of L1's block scales, [Kpad/128][512] in the tensor-memory layout (row = row of d_L1c)
  int l1_shift;                // the scales in d_sfl1 are 2^l1_shift times the factor's; the quantizer takes that off the intermediate again
  float* d_sL1;                // [LQ_MAX_RANK]
  uint8_t* d_L2c;              // [Npad][LQ_RCONT] bytes: int8 codes (or up to 64 halves) of column n, r contiguous
  float* d_sL2;                // [Npad]  (ones for W16A16); d_L2c in d_Wq8's row order; SINT4: d_sL2 and d_bias in
                               // lq_colscale_slot order
  float* d_bias;               // [Npad]  (zeros without bias)
  // MX, one per tile width in use (LQ_MX_WIDTHS):
  uint8_t* d_sfbw[LQ_MX_NWIDTHS];   // E8M0 bytes of the weight scales, [Kpad/128][tiles][ceil(width/128)][512] in the 32 x 16-byte
                                    // layout tensor memory wants (byte 16*(i%32) + 4*((i%128)/32) + block%4)
  uint8_t* d_sfl2w[LQ_MX_NWIDTHS];  // MX branches: the same for L2's block scales along the rank, [tiles][ceil(width/128)][512]
  LqMxMaps* d_maps;            // [LQ_MX_NWIDTHS][2]: of single CTAs, of pairs
  CUtensorMap tmB;             // over d_Wq8, box [LQ_BN][128B], 128B swizzle
  CUtensorMap tmL1;            // over d_L1c, box [all rows][128B], 128B swizzle
  CUtensorMap tmL2;            // over d_L2c, box [LQ_BN][128B], 128B swizzle
};

struct lq_act {
  int K, N, r, G, Kpad, Gpad, branch;
  bool mx, mxfp, a8;
  int planes;                  // 1, or 2 (a8): digit planes of the main codes; qx8 rows are planes * Kpad bytes
  int tq_stride;               // bytes per row of d_tq: LQ_RCONT, or 2 LQ_RCONT when the intermediate's two digit planes get a
                               // container each (a8 with MXINT4 factors: rank up to 128), d_sft then holds two chunks per row block
  uint8_t* d_sft;              // mxfp: E8M0 bytes of the rank-r intermediate's block scales, [Mpad/128][1][512]
  uint8_t* d_sfa;              // MX: E8M0 bytes of the activation scales, [Mpad/128][Kpad/128][512], same layout
  int M_max, Mpad, device, main_kind;
  int M;                       // rows of the last lq_quantize_act
  int M_call;                  // rows of the caller's call (more than M in a chunk of one): what the order of a sum may depend on
  uint8_t* d_qx8;              // [Mpad][Kpad] operand bytes of the 4-bit codes (A operand, K-major)
  float* d_sx;                 // [Gpad][Mpad] fp32 images of the fp16 scales, in lq_row_slot order
  int8_t* d_qb;                // [Mpad][Kpad] branch activation codes; MXFP: the quantizer's near elements
  float* d_sXb;                // [Mpad]
  uint8_t* d_tq;               // [Mpad][LQ_RCONT] bytes: int8 codes (or halves) of T, r contiguous
  float* d_sT;                 // [Mpad] (ones for W16A16); SINT4: in lq_row_slot order; MXFP: the quantizer's bits of near blocks
  void* d_Xstage;              // lazily allocated staging for lq_linear_forward_host
  void* d_Ystage;
  size_t ystage_bytes;
  cudaStream_t s_h2d, s_d2h;   // copy streams of lq_linear_forward_host's row-chunk pipeline (created on first use)
  cudaEvent_t ev_x[LQ_HOST_CHUNKS], ev_y[LQ_HOST_CHUNKS], ev_begin, ev_end;
  bool pipe_ready;
  CUtensorMap tmA;             // over d_qx8, box [LQ_BM][128B], 128B swizzle
  CUtensorMap tmT;             // over d_tq,  box [LQ_BM][128B], 128B swizzle
  CUtensorMap tmSfa, tmSft;    // MX: over all of d_sfa and d_sft, one row of 512 bytes
  int block0;                  // a view's first row / 128 (tmA and tmT begin there, tmSfa and tmSft at the record's first row)
};

// remembers the last failing CUDA runtime code (per host thread) for lq_last_cuda_error(); returns its argument
cudaError_t lq_note_cuda(cudaError_t e);

// device status word (one per device, allocated on first use): {code, stage}
int32_t* lq_device_status_ptr(int device);

// kernels' host launchers (defined in lq_quant.cu / lq_gemm.cu)
lq_status lq_launch_quantize(const lq_layer* L, const void* X, int M, lq_act* A, cudaStream_t st);
lq_status lq_launch_gemm(const lq_layer* L, const lq_act* A, void* Y, lq_out_dtype dt, cudaStream_t st);
lq_status lq_gemm_prepare(int device);
lq_status lq_launch_gemm_mx(const lq_layer* L, const lq_act* A, void* Y, lq_out_dtype dt, cudaStream_t st);
lq_status lq_gemm_mx_prepare(int device);
lq_status lq_launch_wait_probe(int device, cudaStream_t st);   // bounded-wait self-test kernel

// columns of the down-projection's MMA (the rank rounded up to 16) and digit planes of its first factor
static inline int lq_l1_rows(const lq_layer* L) { return lq_round_up(L->r > 0 ? L->r : 16, 16); }
static inline int lq_l1_planes(const lq_layer* L) { return L->a8 && L->cfg.branch == LQ_BRANCH_MXINT8 ? 2 : 1; }

// TMA descriptor (lq_api.cu): 2-D byte tensor [rows][row_bytes], box [box_rows][128 bytes], 128-byte swizzle.
lq_status lq_make_tmap_bytes(CUtensorMap* tm, void* base, uint64_t rows, uint64_t row_bytes, uint32_t box_rows);

// whether every row of Y begins on a 32-byte boundary (callers promise 16 bytes, and N a multiple of 8)
static inline int lq_rows_of_sectors(const void* Y, int N, lq_out_dtype dt) {
  return (((uintptr_t)Y | (uintptr_t)N * (dt == LQ_OUT_F32 ? 4 : 2)) & 31) == 0;
}

// byte an MMA operand carries for a 4-bit code q in [-7, 7]
static inline uint8_t lq_encode_code_host(int q, int kind) {
  if (kind == LQ_KIND_I8) return (uint8_t)(int8_t)q;
  static const uint8_t mag[8] = {0x00, 0x38, 0x40, 0x44, 0x48, 0x4A, 0x4C, 0x4E};  // E4M3 of 0..7
  int a = q < 0 ? -q : q;
  return (uint8_t)(mag[a] | (q < 0 ? 0x80 : 0));
}

// bits of a packed weight element of the MX GEMM: MXFP4 as e2m1, the 4-bit integer codes as e2m3 (the narrowest type that has them)
static inline int lq_mx_weight_bits(const lq_layer* L) { return L->mxfp ? 4 : 6; }
// E2M3 of an integer in [-7, 7] (bias 1, three mantissa bits)
static inline uint8_t lq_code_e2m3(int q) {
  static const uint8_t mag[8] = {0, 8, 16, 20, 24, 26, 28, 30};
  return (uint8_t)((q < 0 ? 0x20 : 0) | mag[q < 0 ? -q : q]);
}

extern int g_lq_main_kind;   // option "main_kind"
extern int g_lq_gemm_ctas;   // option "gemm_ctas" (0 = one per SM)
extern int g_lq_gemm_pair;   // option "gemm_pair": 1 = pairs of CTAs share an MX GEMM's tile where there are enough rows
extern int g_lq_gemm_split;  // option "gemm_split": CTAs that share a tile of the SINT4 GEMM where there is room for them, 0 = chosen by the launcher
extern int g_lq_gemm_width;  // option "gemm_width": tile width of the MX GEMM, 0 = chosen by the launcher
// options "quant_warps", "quant_ctas": the quantizer's row groups per tile and stages per chunk, 0 = chosen by the launcher
extern int g_lq_quant_warps, g_lq_quant_ctas;
extern int g_lq_overlap;     // option "overlap": launch kernels with programmatic stream serialization
extern int g_lq_store_qb;    // option "store_qb": also write the branch activation codes to HBM (parity export)

#ifdef __CUDACC__
// Launches `kernel` on `st`.  With the "overlap" option the launch carries programmatic stream serialization: the
// kernel's CTAs may become resident and run their set-up (barriers, tensor memory) while the previous kernel on the
// stream is still draining its last tiles; every kernel of this library executes griddepcontrol.wait after that set-up,
// before it reads what an earlier kernel may write or writes global memory (weights, which no kernel writes, and the quantizer's
// prefetch of X to the L2 come before it), and griddepcontrol.launch_dependents after the set-up, so that the chain
// quantizer -> GEMM -> next quantizer overlaps its launch gaps and tails.  All kernels here are persistent (the whole
// grid is resident at once), so a waiting successor never holds an SM that a predecessor CTA still needs.
template <typename... KArgs, typename... Args>
static inline cudaError_t lq_launch_cluster(void (*kernel)(KArgs...), int grid, int block, int cluster, size_t smem, cudaStream_t st,
                                            Args&&... args) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)grid); lc.blockDim = dim3((unsigned)block); lc.dynamicSmemBytes = smem; lc.stream = st;
  cudaLaunchAttribute at[2];
  int n = 0;
  if (g_lq_overlap) {
    at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    at[n].id = cudaLaunchAttributeClusterDimension;
    at[n].val.clusterDim.x = (unsigned)cluster; at[n].val.clusterDim.y = 1; at[n].val.clusterDim.z = 1;
    ++n;
  }
  lc.attrs = at; lc.numAttrs = (unsigned)n;
  return cudaLaunchKernelEx(&lc, kernel, std::forward<Args>(args)...);
}
template <typename... KArgs, typename... Args>
static inline cudaError_t lq_launch(void (*kernel)(KArgs...), int grid, int block, size_t smem, cudaStream_t st, Args&&... args) {
  return lq_launch_cluster(kernel, grid, block, 1, smem, st, std::forward<Args>(args)...);
}
#endif
