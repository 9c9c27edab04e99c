// Blackwell tensor-core plumbing (tcgen05 + TMEM + mbarrier), inline PTX for sm_103a.
//
// Operands live in shared memory in the no-swizzle K-major layout: 8-row x 16-byte core
// matrices, rows 16 bytes apart inside a core matrix, 8-row groups SBO bytes apart, and the
// second 8-element K chunk LBO bytes after the first. The accumulator D (M = 128 lanes x
// N fp32 columns) lives in tensor memory; lane i holds row i, and warp w of the CTA reads
// lanes 32 (w % 4) .. 32 (w % 4) + 31.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace dh {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// shared-memory matrix descriptor (tcgen05 format, version 1, no swizzle)
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// instruction descriptor of kind::f16: D f32, A and B bf16, both K-major, M x N
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

// the same with A and B MN-major (the reduction index strided): 8 contiguous rows x 8 K per
// core matrix, K rows 16 bytes apart, LBO between groups of 8 K, SBO between groups of 8 rows
__host__ __device__ constexpr uint32_t umma_idesc_bf16_mn(int M, int N) {
  return umma_idesc_bf16(M, N) | (1u << 15) | (1u << 16);
}

// One lane of the calling warp (all lanes call it; the same lane every time): 1 there, 0 on
// the others. A warp issues its MMAs as a whole, predicated on this: the loop, the waits and
// the descriptors then stay warp-uniform, which keeps them in the uniform registers that
// tcgen05.mma takes (from inside a one-lane branch every operand is moved there first).
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(e));
  return e;
}

// D += A B issued by the elected lane; descriptors as their low words and common high words
// (a start address moves within the low word)
__device__ __forceinline__ void umma_bf16_acc(uint32_t leader, uint32_t d_tmem, uint32_t a_lo,
                                              uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                              uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred e, p;\n\t.reg .b64 a, b;\n\tsetp.ne.b32 e, %0, 0;\n\t"
      "setp.eq.u32 p, %1, %1;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%1], a, b, %6, p;\n\t}\n" ::"r"(leader),
      "r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc));
}

// the same with D = A B where acc is 0 (an accumulator's first MMA)
__device__ __forceinline__ void umma_bf16(uint32_t leader, uint32_t d_tmem, uint32_t a_lo,
                                          uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                          uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred e, p;\n\t.reg .b64 a, b;\n\tsetp.ne.b32 e, %0, 0;\n\t"
      "setp.ne.b32 p, %7, 0;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%1], a, b, %6, p;\n\t}\n" ::"r"(leader),
      "r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(acc));
}

// arrive once on the mbarrier when every tcgen05.mma issued so far by the elected lane is done
__device__ __forceinline__ void umma_commit(uint32_t leader, uint64_t* mbar) {
  asm volatile(
      "{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %0, 0;\n\t"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%1];\n\t}\n" ::"r"(leader),
      "r"(smem_u32(mbar))
      : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* mbar) {
  uint64_t state;
  asm volatile("mbarrier.arrive.shared::cta.b64 %0, [%1];" : "=l"(state) : "r"(smem_u32(mbar)) : "memory");
  (void)state;
}

__device__ __forceinline__ void mbar_init(uint64_t* mbar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(count));
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Non-blocking check of phase `parity` of the mbarrier; 1 when it has completed.
__device__ __forceinline__ uint32_t mbar_test(uint64_t* mbar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(done)
      : "r"(smem_u32(mbar)), "r"(parity)
      : "memory");
  return done;
}

// Wait for phase `parity` of the mbarrier for at most limit_ns nanoseconds of the global
// timer (and at most 2^26 polls); returns 1 when the phase completed, 0 when the wait gave
// up. limit_ns = 0: one non-blocking check only. Short waits spin on the non-blocking check
// (waking a suspended thread takes about a microsecond, which the stages of a pipeline would
// pay one after another); after kSpinPolls of them each poll may suspend the thread for up to
// kSuspendNs until the phase completes, so a long wait does not spin on the issue slots the
// working warps of its scheduler need. The timer is read only after a first such poll has run
// out, so a wait gives up at most two polls after its limit.
constexpr int kSpinPolls = 64;
constexpr uint32_t kSuspendNs = 10000;
__device__ __forceinline__ uint32_t mbar_poll(uint64_t* mbar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(done)
      : "r"(smem_u32(mbar)), "r"(parity), "r"(kSuspendNs)
      : "memory");
  return done;
}
__device__ __forceinline__ uint32_t mbar_wait_ns(uint64_t* mbar, uint32_t parity, uint64_t limit_ns) {
  if (mbar_test(mbar, parity)) return 1;
  if (limit_ns == 0) return 0;
  for (int it = 0; it < kSpinPolls; ++it)
    if (mbar_test(mbar, parity)) return 1;
  if (mbar_poll(mbar, parity)) return 1;
  const uint64_t t0 = global_ns();
  for (int it = 0; it < (1 << 26); ++it) {
    if (mbar_poll(mbar, parity)) return 1;
    if (global_ns() - t0 >= limit_ns) return 0;
  }
  return 0;
}

// TMEM allocation of `ncols` columns (power of two, 32..512) by one whole warp; the base
// address is written to *slot (shared memory).
__device__ __forceinline__ void tmem_alloc_warp(uint32_t* slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(slot)),
               "r"(ncols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}

__device__ __forceinline__ void tmem_dealloc_warp(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// generic-proxy shared-memory writes -> visible to the tensor core (async proxy)
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// 16 consecutive fp32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

}  // namespace dh
