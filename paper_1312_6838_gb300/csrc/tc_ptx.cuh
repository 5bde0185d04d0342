// PTX of the tensor-core kernels (tc_gemm.cu, slice_gemm.cu): mbarriers with
// bounded waits, TMA copies, tcgen05 MMAs and TMEM loads.
#pragma once

#include <cuda.h>

#include "css_common.cuh"

namespace css {
namespace tc {

// ------------------------------------------------------------- PTX glue -----
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait for the phase with the given parity.  false: timed out (the
// error flag is set) or another role already failed.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* err,
                                          unsigned long long budget) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = gtimer();
  while (true) {
#pragma unroll 1
    for (int i = 0; i < 32; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (*(volatile int*)err != 0) return false;
    if (gtimer() - t0 > budget) {
      atomicCAS(err, 0, (int)CSS_ERR_TIMEOUT);
      return false;
    }
  }
}
// Wait used on the way out of a failed CTA: the copies and MMAs this CTA
// issued always complete, so it waits for them whatever the error flag says
// (a fixed bound of 1 s; it returns in microseconds in practice), so that no
// copy lands in, and no MMA reads, the shared memory or TMEM of an exited CTA.
__device__ __forceinline__ void mbar_drain(uint32_t bar, uint32_t parity) {
  const uint64_t t0 = gtimer();
  while (!mbar_try_wait(bar, parity))
    if (gtimer() - t0 > 1000000000ull) return;
}
// Shared-memory matrix descriptor, 128-byte swizzle (sm_100 format), as halves.
__device__ __forceinline__ uint32_t sw128_desc_lo(uint32_t saddr, uint32_t lbo) {
  return ((saddr >> 4) & 0x3FFFu) | ((lbo >> 4) & 0x3FFFu) << 16;
}
__host__ __device__ constexpr uint32_t sw128_desc_hi(uint32_t sbo) { return (sbo >> 4) | 1u << 14 | 2u << 29; }
// Instruction descriptor: kind::f16, BF16 x BF16 -> FP32.
__device__ __forceinline__ uint32_t make_idesc(int N, int M, bool a_mn, bool b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t e;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(e));
  return e;
}
// mbar_wait by the whole warp, with one answer
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, int* err, unsigned long long budget) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, err, budget));
}
// Issue by one elected lane of a warp that walks its loops as a whole, with
// warp-uniform values, so that addresses and descriptors live in uniform
// registers.  From a divergent thread each MMA cost about 150 clocks of moves
// into them, more than a 128 x 128 x 16 (64 clocks) or 128 x 256 x 16 (128)
// MMA takes.  Descriptors come as 32-bit halves; only the address field of the
// low one changes from one MMA to the next.
__device__ __forceinline__ void umma_elected(uint32_t elected, uint32_t tmem_d, uint32_t a_lo, uint32_t b_lo,
                                             uint32_t desc_hi, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p, q;\n .reg .b64 da, db;\n setp.ne.b32 p, %5, 0;\n setp.ne.b32 q, %6, 0;\n"
      " mov.b64 da, {%1, %4};\n mov.b64 db, {%2, %4};\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n}" ::"r"(tmem_d),
      "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(desc_hi), "r"(accumulate), "r"(elected)
      : "memory");
}
__device__ __forceinline__ void tma_load_2d_elected(uint32_t elected, uint32_t dst, const CUtensorMap* map,
                                                    uint32_t bar, int c0, int c1) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %5, 0;\n"
      " @q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
      "[%2];\n}" ::"r"(dst),
      "l"((uint64_t)map), "r"(bar), "r"(c0), "r"(c1), "r"(elected)
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}
__device__ __forceinline__ void fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
      "[%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

}  // namespace tc
}  // namespace css
