// Device-side building blocks shared by the sm_100a kernels: mbarrier / TMA / ldmatrix / mma
// wrappers (inline PTX), bounded waits, small numeric helpers.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/specvlm.h"

namespace specvlm {

constexpr int kTileTokens = 64;        // tokens per K/V tile (= one cache page)
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Programmatic dependent launch.  Every kernel of the path is launched so that it may start while the
// kernel before it in the stream still runs (launch_after) and waits for the predecessor's completion, in every CTA,
// before its first access to global memory: what precedes the wait (barriers, tensor memory, descriptors, the launch
// itself) costs no time on the stream.  It lets its own successor start once all its CTAs run, and have their tensor
// memory where they use it (tmem_alloc_launch_next), so that a successor's CTA that waits holds nothing that the kernel
// it waits for still needs.  The finishing kernels of acceptance do not release early (accept.cu).  Data that an earlier kernel may have written is therefore never read through the non-coherent path
// (__ldg, const __restrict__): a line cached before the wait would not be dropped by it.
__device__ __forceinline__ void pdl_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// All threads of the cluster (of the CTA, where the launch has no clusters): what came before it in any of them is
// visible after it in all of them, shared memory of the other CTAs included.
__device__ __forceinline__ void cluster_barrier() {
  __syncwarp();                            // .aligned: the warp arrives as one
  asm volatile(
      "barrier.cluster.arrive.release.aligned;\n\t"
      "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address of this CTA's shared-memory word `addr` in the cluster's CTA `rank`
__device__ __forceinline__ uint32_t cluster_map(uint32_t addr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

// ------------------------------------------------------------------------------ mbarrier
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// A waiting thread may stay suspended for up to this long before try_wait reports "not yet" (it
// resumes at once when the phase completes): fewer polling instructions from the roles that wait
// most.  No effect on a single call; 1.7 % on the verification kernel under sustained load, where
// the chip runs at its power cap (364 -> 357 us per call at 1.45 GHz).
#ifndef SPECVLM_SUSPEND_HINT_NS
#define SPECVLM_SUSPEND_HINT_NS 20000
#endif
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
#if SPECVLM_SUSPEND_HINT_NS > 0
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"((uint32_t)SPECVLM_SUSPEND_HINT_NS)
      : "memory");
#else
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
#endif
  return ok != 0;
}
// Non-blocking: has the phase with the given parity completed?
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// Wait for the phase with the given parity to complete.  Every wait is bounded: after a burst
// of fast polls the wall clock is consulted, and after kWaitLimitNs the wait gives up.  A CTA
// shares one abort flag in shared memory so that one expired wait ends all the others at once.
constexpr uint64_t kWaitLimitNs = 2000000000ull;   // 2 s
__device__ __forceinline__ bool mbar_wait_limit(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                                const uint64_t limit_ns) {
#pragma unroll 1
  for (int i = 0; i < 2048; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
#pragma unroll 1
  while (true) {
#pragma unroll 1
    for (int i = 0; i < 256; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (global_timer_ns() - t0 > limit_ns) {
      *abort_flag = 1;
      return false;
    }
  }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return mbar_wait_limit(bar, parity, abort_flag, kWaitLimitNs);
}
// The same for phases that are mostly over already: a plain test sees them in half the time (49 against
// 106 cycles with the vote around it).  Verification of 80 layers of 6400 tokens 322 -> 316.5 us; the
// rating passes and the decode kernel, whose waits really wait, lose 0.5 to 1 % by it.
__device__ __forceinline__ bool mbar_wait_soon(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return mbar_test_wait(bar, parity) || mbar_wait(bar, parity, abort_flag);
}

// Waits of a whole warp: the vote makes the outcome the same in every lane, whichever lanes saw the abort flag.
__device__ __forceinline__ bool warp_all(bool ok) { return __all_sync(0xffffffffu, ok) != 0; }
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return warp_all(mbar_wait(bar, parity, abort_flag));
}
__device__ __forceinline__ bool warp_wait_soon(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return warp_all(mbar_wait_soon(bar, parity, abort_flag));
}

__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// True in one lane of the (whole, converged) warp, the same one every time.  What a warp issues for itself -- tensor
// instructions, their commits, TMA copies -- goes behind this in code that all of its lanes run, and not into a branch of
// `lane == 0`: eight tcgen05.mma of fixed operands take 402 cycles to issue there and 133 behind this; with operands that
// change from tile to tile 760 in the first form.  (Why was not looked into: the operands are in uniform registers, and
// presumably the compiler can keep them there only where no lane stands out.)  Verification, sustained, at 80 layers of 6400
// tokens: a tree of 208 rows 669 -> 648 us (4310 -> 3700 cycles a tile), 48 rows 360 -> 353.5.  Not in the rating passes,
// whose issuer is never late: 32 polling lanes there cost 0.6 to 1 % at the power cap; nor for the copies of the decode kernel
// with a CTA per item (even), but on slices (9 layers of 16 sequences, d = 64, 56.0 -> 54.9 us; 13 layers of 43 856 tokens,
// 16 rows, 598 -> 594).
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(e));
  return e != 0;
}

// ------------------------------------------------------------------------------ TMA
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* m) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
// 5-D tiled load global -> shared, completion on an mbarrier (bytes), with an L2 cache policy
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* m, uint32_t bar, int c0,
                                            int c1, int c2, int c3, int c4, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%0], [%1, {%3, %4, %5, %6, %7}], [%2], %8;"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
      "r"(c4), "l"(policy)
      : "memory");
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// ------------------------------------------------------------------------------ tensor cores
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2,
                                            uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1,
                                                  uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
// D(16x8, fp32) += A(16x16, bf16, row) * B(16x8, bf16, col)
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                               uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Packed pairs of fp32 (sm_100 issues an f32x2 operation on two values in one slot).
__device__ __forceinline__ uint64_t f2_pack(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t f2_sub(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// 2^t for a pair of arguments t <= 0 on the FMA and integer pipes, leaving the special-function
// unit to other elements: t = n + f with n = round(t) and |f| <= 1/2 (adding 1.5 * 2^23 leaves n in
// the low mantissa bits), 2^f by a degree-4 polynomial (least-maximum relative error 2.7e-6 on
// [-1/2, 1/2], fitted for this file), and n added to the exponent field.  Arguments below -125 give
// 2^-125 instead of 0.
__device__ __forceinline__ uint64_t f2_exp2_poly(uint64_t t2) {
  float a, b;
  f2_unpack(t2, a, b);
  t2 = f2_pack(fmaxf(a, -125.f), fmaxf(b, -125.f));
  const uint64_t magic = f2_pack(12582912.f, 12582912.f);
  const uint64_t r2 = f2_add(t2, magic);
  const uint64_t f2 = f2_sub(t2, f2_sub(r2, magic));
  uint64_t p = f2_fma(f2_pack(0.009569965302944183f, 0.009569965302944183f), f2,
                      f2_pack(0.05591750890016556f, 0.05591750890016556f));
  p = f2_fma(p, f2, f2_pack(0.240247443318367f, 0.240247443318367f));
  p = f2_fma(p, f2, f2_pack(0.6931218504905701f, 0.6931218504905701f));
  p = f2_fma(p, f2, f2_pack(0.9999992847442627f, 0.9999992847442627f));
  float p0, p1, r0, r1;
  f2_unpack(p, p0, p1);
  f2_unpack(r2, r0, r1);
  p0 = __int_as_float(__float_as_int(p0) + (__float_as_int(r0) << 23));
  p1 = __int_as_float(__float_as_int(p1) + (__float_as_int(r1) << 23));
  return f2_pack(p0, p1);
}
__device__ __forceinline__ uint64_t f2_exp2_sfu(uint64_t t2) {
  float a, b;
  f2_unpack(t2, a, b);
  return f2_pack(fast_exp2(a), fast_exp2(b));
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&t);
}

// Byte offset of (token row t, 16-byte chunk c16) inside a K or V tile of kTileTokens rows as
// written by a 128-byte-swizzled tensor-map load: the tile is split in halves of 64 channels
// (128 B per row); inside a half the 16-byte chunk index is XORed with (row & 7).
template <int D>
__device__ __forceinline__ uint32_t tile_offset(int t, int c16) {
  if constexpr (D == 128) {
    return static_cast<uint32_t>((c16 >> 3) * (kTileTokens * 128) + t * 128 +
                                 (((c16 & 7) ^ (t & 7)) << 4));
  } else {
    return static_cast<uint32_t>(t * 128 + ((c16 ^ (t & 7)) << 4));
  }
}

}  // namespace specvlm

// ------------------------------------------------------------------------------ tcgen05 / TMEM
// (5th-generation tensor cores: operands in shared memory described by 64-bit matrix
// descriptors, accumulators in tensor memory, completion signalled on mbarriers)
namespace specvlm {

// Allocates `ncols` (power of two >= 32) TMEM columns; the base address is written to shared
// memory at `smem_dst`.  Warp-collective.
__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
// The allocation of a kernel that takes part in programmatic dependent launch, by the one warp that releases the
// successor, once the CTA has its columns.  A release by another warp could come while this one still waits for columns:
// a successor's CTA that took them and then waited for this kernel would leave both waiting for ever.
__device__ __forceinline__ void tmem_alloc_launch_next(uint32_t smem_dst, uint32_t ncols) {
  tmem_alloc(smem_dst, ncols);
  pdl_launch_next();
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before_sync() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after_sync() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// Shared-memory matrix descriptor for a bf16 operand tile stored as rows of 128 bytes with the
// 128-byte swizzle (what a tensor-map load with CU_TENSOR_MAP_SWIZZLE_128B writes).
//   K-major  (the contraction dimension runs along the 128-byte row): lbo = 1, sbo = 1024 B
//   MN-major (the M/N dimension runs along the row): lbo = distance between 64-element column
//            blocks, sbo = 1024 B (8 rows)
// Field positions: start address [0,14) (>>4), leading byte offset [16,30) (>>4), stride byte
// offset [32,46) (>>4), descriptor version 1 at [46,48), swizzle mode 2 (128 B) at [61,64).
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t smem_addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  return (uint64_t)((smem_addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32) | (1ull << 46) | (2ull << 61);
}
// The same descriptor with its start address moved by `bytes` (a multiple of 16).
__device__ __forceinline__ uint64_t umma_desc_advance(uint64_t desc, uint32_t bytes) { return desc + (bytes >> 4); }
// Instruction descriptor of kind::f16 with bf16 A and B, fp32 accumulator.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int m, int n, bool a_mn_major, bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn_major ? 1u : 0u) << 15) | ((b_mn_major ? 1u : 0u) << 16) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
// D[tmem] (+)= A[smem] * B[smem]; issued by one thread.
__device__ __forceinline__ void umma_bf16_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                             uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives once on the mbarrier when every tcgen05.mma issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}
// Warp-collective load of 32 consecutive fp32 columns of this warp's 32 TMEM lanes: thread i gets
// lane (base lane + i), columns [col, col + 32).
__device__ __forceinline__ void tmem_ld_x32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
// The same for 16 columns.
__device__ __forceinline__ void tmem_ld_x16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

}  // namespace specvlm
