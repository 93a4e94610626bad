// Device-side building blocks shared by the library's kernels: mbarrier and bulk-copy (TMA) wrappers, bounded
// waits, tcgen05 (tensor memory / 5th-generation MMA) wrappers and the descriptor builders.  Internal: not part
// of the C ABI.  Everything is inline PTX written from the PTX ISA description of sm_100a.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "lq_internal.h"

namespace lqdev {

constexpr long long WAIT_LIMIT_CYCLES = 4000000000ll;   // ~2 s at 2 GHz: no device wait is unbounded

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// ---- mbarrier -----------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// SCOPE: whose arrivals the wait is for.  PEER_TMEM: another CTA's of the cluster, too, which hand over tensor memory (peer_arrive).
// PEER_DATA: copies of other CTAs into this one's shared memory (peer_copy), which the wait makes visible.
enum { OWN_CTA = 0, PEER_TMEM = 1, PEER_DATA = 2 };
template <int SCOPE = OWN_CTA>
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  if constexpr (SCOPE == PEER_DATA)
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
  else if constexpr (SCOPE == PEER_TMEM)
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.relaxed.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
  return ok != 0;
}

// Bounded wait.  Returns false when the CTA is aborting or the deadline passed (then it raises the abort flag
// and records who gave up in the device status word {code, stage}).
template <int SCOPE = OWN_CTA>
static __device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* status,
                                            int role, long long limit = WAIT_LIMIT_CYCLES) {
  const long long t0 = clock64();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait<SCOPE>(bar, parity)) return true;
    if ((it & 0xFF) == 0) {
      if (*abort_flag) return false;
      if (clock64() - t0 > limit) {
        *abort_flag = 1;
        if (atomicCAS(status, 0, (int)LQ_ERR_TIMEOUT) == 0) status[1] = role;
        return false;
      }
    }
  }
}
template <int SCOPE = OWN_CTA>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* status,
                                          int role) {
  if (mbar_try_wait<SCOPE>(bar, parity)) return true;
  return mbar_wait_slow<SCOPE>(bar, parity, abort_flag, status, role);
}
// The same wait without a call on its slow path: for a warp whose registers are full of data.
__device__ __forceinline__ bool mbar_wait_inline(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* status, int role) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 0xFF) == 0) {
      if (*abort_flag) return false;
      if (clock64() - t0 > WAIT_LIMIT_CYCLES) {
        *abort_flag = 1;
        if (atomicCAS(status, 0, (int)LQ_ERR_TIMEOUT) == 0) status[1] = role;
        return false;
      }
    }
  }
}
// The same wait for a whole warp: all lanes go on, or none.
template <int SCOPE = OWN_CTA>
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* status,
                                               int role) {
  const bool ok = mbar_wait<SCOPE>(bar, parity, abort_flag, status, role);
  return __all_sync(0xffffffffu, ok);
}
// Abort path only: gives a transaction that is still in flight on `bar` a bounded time to land, so that no
// copy writes into shared memory after the CTA has left.  Never raises a new error.
__device__ __forceinline__ void mbar_settle(uint32_t bar, uint32_t parity, long long limit = 4000000ll) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity) && clock64() - t0 < limit) { }
}

// Programmatic dependent launch: let the next kernel on the stream start its set-up, then wait until the previous
// kernel on the stream has completed and its writes are visible (both are no-ops for a plain launch).
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---- thread-block clusters: rendezvous, and barriers of a peer CTA ---------------------------
// HANDS_OVER: what this thread has written before is for the others to read once they have waited.
template <bool HANDS_OVER = true>
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();      // the barrier's aligned form wants the warp's lanes together, whatever branches lie behind them
  if constexpr (HANDS_OVER) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  else asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync() {
  cluster_arrive();
  cluster_wait();
}
__device__ __forceinline__ uint32_t peer_smem(uint32_t addr, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
  return a;
}
// Arrival on a barrier of another CTA that hands over tensor memory and nothing else: tcgen05.wait::ld has emptied it, and the tcgen05
// fences on both sides order the accesses to it, so arrival and wait may be relaxed.  (As a release the arrival waits for the
// thread's earlier stores - a drain warp's stores of Y - to be performed, over a thousand clocks.)
__device__ __forceinline__ void peer_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Copies shared memory (16-byte multiples) to another CTA's, counted on a barrier of that CTA when it is there.
__device__ __forceinline__ void peer_copy(uint32_t peer_dst, uint32_t src, uint32_t bytes, uint32_t peer_bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(peer_dst), "r"(src), "r"(bytes),
               "r"(peer_bar) : "memory");
}
// ---- shared memory by 32-bit address ---------------------------------------------------------
__device__ __forceinline__ uint4 lds_v4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts_v4(uint32_t a, const uint4& v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void sts_u32(uint32_t a, uint32_t v) { asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
// 32 bytes (of an address that is a multiple of 32) to global memory: a whole sector in one request
__device__ __forceinline__ void stg_v8(void* p, const uint32_t (&w)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]),
               "r"(w[6]), "r"(w[7]) : "memory");
}
// the same of an address that is a multiple of 32 (SECTORS) or only of 16
template <bool SECTORS>
__device__ __forceinline__ void stg_32(void* p, const uint32_t (&w)[8]) {
  if constexpr (SECTORS) {
    stg_v8(p, w);
  } else {
    reinterpret_cast<uint4*>(p)[0] = make_uint4(w[0], w[1], w[2], w[3]);
    reinterpret_cast<uint4*>(p)[1] = make_uint4(w[4], w[5], w[6], w[7]);
  }
}
// generic-proxy writes to shared memory become visible to the asynchronous proxy (MMA operands, tensor-memory copies)
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.b32 %0, 1, 0, P;\n\t}" : "=r"(pred));
  return pred != 0;
}

// ---- bulk copies (TMA): every copy goes to the issuing CTA only -----------------------------
#define LQ_TMA_2D "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
// of a pair of CTAs: the barrier may be the other CTA's
#define LQ_TMA_2D_PAIR "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
template <bool PAIR = false>
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tm, int x, int y, uint32_t bar) {
  if constexpr (PAIR)
    asm volatile(LQ_TMA_2D_PAIR " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(bar) : "memory");
  else
    asm volatile(LQ_TMA_2D " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(bar) : "memory");
}
// with a word on how long the L2 should keep what is read
__device__ __forceinline__ uint64_t l2_evict_first() {
  uint64_t v;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(v));
  return v;
}
__device__ __forceinline__ uint64_t l2_evict_normal() {
  uint64_t v;
  asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(v));
  return v;
}
__device__ __forceinline__ void tma_load_2d_hint(uint32_t dst, const CUtensorMap* tm, int x, int y, uint32_t bar, uint64_t policy) {
  asm volatile(LQ_TMA_2D ".L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(bar),
               "l"(policy)
               : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar)
               : "memory");
}
// Brings global memory (16-byte multiples) into the L2.  A hint: what it finds there may still be written, by a kernel before, say.
__device__ __forceinline__ void bulk_prefetch(const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(reinterpret_cast<uint64_t>(src)), "r"(bytes) : "memory");
}

// ---- tcgen05 ------------------------------------------------------------------------------
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t slot_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot_smem), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}

// the same for a pair of CTAs (cta_group::2): both CTAs allocate and free, the first one issues copies, MMAs and commits for both
__device__ __forceinline__ void tmem_alloc_pair(uint32_t slot_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot_smem), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
// arrives on the barrier at this address in both CTAs once the MMAs issued so far have retired
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"((uint16_t)3)
               : "memory");
}

enum { TC_I8 = 0, TC_F16 = 1 };
template <int KIND>
__device__ __forceinline__ void tc_mma_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  if constexpr (KIND == TC_I8) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  }
}
__device__ __forceinline__ void tc_mma_mx_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t tsfa,
                                               uint32_t tsfb, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale [%0], %1, %2, %3, [%5], [%6], p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(tsfa), "r"(tsfb)
      : "memory");
}
__device__ __forceinline__ void tc_cp_sf_pair(uint32_t taddr, uint64_t sdesc) {
  asm volatile("tcgen05.cp.cta_group::2.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(sdesc) : "memory");
}

template <int KIND>
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  if constexpr (KIND == TC_I8) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  }
}
// block-scaled MMA: 8-bit-class operands, E8M0 scales (one per row and 32-deep K block) read from tensor memory
__device__ __forceinline__ void tc_mma_mx(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t tsfa,
                                          uint32_t tsfb, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::mxf8f6f4.block_scale [%0], %1, %2, %3, [%5], [%6], p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(tsfa), "r"(tsfb)
      : "memory");
}
// 32 rows x 16 bytes of shared memory -> 4 tensor-memory columns, replicated into the four 32-lane quarters
__device__ __forceinline__ void tc_cp_sf(uint32_t taddr, uint64_t sdesc) {
  asm volatile("tcgen05.cp.cta_group::1.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(sdesc) : "memory");
}

// 32 lanes x 16 consecutive 32-bit columns: thread t of the warp receives row (lane base + t).
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}
// 16 lanes x 32 consecutive 32-bit columns in the accumulator-fragment layout of mma.sync m16n8: with g = lane / 4 and
// t = lane % 4, registers 4j .. 4j+3 hold (row g, columns 8j + 2t, 8j + 2t + 1) and (row g + 8, the same columns).
__device__ __forceinline__ void tmem_ld_16x256b_x4(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows of 128 bytes, 8-row atoms 1024 bytes
// apart.  Adding (bytes >> 4) steps along K inside the swizzled row.
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t smem_addr) {
  const uint32_t lo = ((smem_addr & 0x3FFFFu) >> 4) | (1u << 16);          // start address, LBO = 1 (unused)
  const uint32_t hi = (1024u >> 4) | (1u << 14) | (2u << 29);              // SBO = 1024 B, version 1, SWIZZLE_128B
  return ((uint64_t)hi << 32) | lo;
}
// Shared-memory matrix descriptor without swizzle (K-major, 8-row x 16-byte core matrices stored contiguously).
__device__ __forceinline__ uint64_t make_smem_desc_plain(uint32_t smem_addr, uint32_t lbo, uint32_t sbo) {
  const uint32_t lo = ((smem_addr & 0x3FFFFu) >> 4) | ((lbo >> 4) << 16);
  const uint32_t hi = (sbo >> 4) | (1u << 14);                             // version 1, no swizzle
  return ((uint64_t)hi << 32) | lo;
}

// instruction descriptor: accumulator format, operand formats, N >> 3 at bit 17, M >> 4 at bit 24
__device__ __forceinline__ constexpr uint32_t idesc_shape(int n) { return ((uint32_t)(n >> 3) << 17) | ((uint32_t)(LQ_BM >> 4) << 24); }
constexpr uint32_t IDESC_I8 = (2u << 4) | (1u << 7) | (1u << 10);    // S8 x S8 -> S32
constexpr uint32_t IDESC_F8 = (1u << 4) | (0u << 7) | (0u << 10);    // E4M3 x E4M3 -> F32
constexpr uint32_t IDESC_F16 = (1u << 4) | (0u << 7) | (0u << 10);   // F16 x F16 -> F32
// instruction descriptor of the block-scaled kind: E4M3 x E4M3, E8M0 scales, K-major operands, scale-byte ids
__device__ __forceinline__ constexpr uint32_t idesc_mx2(int n, int a_sf_id, int b_sf_id) {
  return ((uint32_t)b_sf_id << 4) | ((uint32_t)(n >> 3) << 17) | (1u << 23) | ((uint32_t)(LQ_BM >> 4) << 24) | ((uint32_t)a_sf_id << 29);
}
constexpr uint32_t IDESC_MX_B_E2M1 = 5u << 10, IDESC_MX_B_E2M3 = 3u << 10;   // added: the B operand is E2M1, E2M3
__device__ __forceinline__ constexpr uint32_t idesc_mx_ids(int sf_id) { return ((uint32_t)sf_id << 4) | ((uint32_t)sf_id << 29); }   // the scale-byte ids alone
__device__ __forceinline__ constexpr uint32_t idesc_mx(int n, int sf_id) { return idesc_mx2(n, sf_id, sf_id); }

// ---- timeline build (-DLQ_TIMELINE): per-role clock stamps of CTA 0 ----------------------
// A stamp is one 8-byte store by lane 0 of the stamping warp: (event id << 48) | (tag << 40) | (clock64 & 2^40-1),
// appended to that warp's list g_lq_timeline[list][...] (a zero word ends a list).  The regular build compiles
// every LQ_TL_* macro to nothing.
#ifdef LQ_TIMELINE
constexpr int TL_LISTS = 4, TL_CAP = 8192;
enum { TL_PRODUCER = 0, TL_MMA = 1, TL_DRAIN_FIRST = 2, TL_DRAIN_LAST = 3 };
enum {
  EV_P_SLOT_FREE = 1, EV_P_ISSUED = 2,                          // producer: stage free / copies issued
  EV_M_STAGE_FULL = 3, EV_M_ACC_FREE = 4, EV_M_ISSUED = 5,      // MMA warp: operands landed / accumulator free / MMAs + commit issued
  EV_D_OPEN = 6, EV_D_ACC_FULL = 7, EV_D_LOADED = 8, EV_D_DONE = 9,   // drain: starts waiting / accumulator ready / slice in registers / arithmetic done
  EV_D_EPI_BEGIN = 10, EV_D_EPI_END = 11, EV_TILE = 12, EV_D_HALF = 13, EV_D_LD_ISSUED = 14, EV_D_WAITED = 15
};
}  // namespace lqdev
static __device__ unsigned long long g_lq_timeline[lqdev::TL_LISTS][lqdev::TL_CAP];   // one per translation unit
namespace lqdev {
struct TlCursor { int list; unsigned n; };
__device__ __forceinline__ void tl_stamp(TlCursor& c, int ev, int tag) {
  if (c.list >= 0 && c.n + 1 < (unsigned)TL_CAP)
    g_lq_timeline[c.list][c.n++] = ((unsigned long long)ev << 48) | ((unsigned long long)(tag & 0xFF) << 40) |
                                   ((unsigned long long)clock64() & 0xFFFFFFFFFFull);
}
#define LQ_TL_DECL(LIST_EXPR) lqdev::TlCursor tl_cur{(LIST_EXPR), 0u}
#define LQ_TL(EV, TAG) lqdev::tl_stamp(tl_cur, (EV), (TAG))
#else
#define LQ_TL_DECL(LIST_EXPR)
#define LQ_TL(EV, TAG)
#endif

}  // namespace lqdev
