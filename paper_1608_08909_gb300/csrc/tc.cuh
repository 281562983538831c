// tcgen05 / mbarrier / bulk-copy primitives shared by the tensor-core kernels
// (inline PTX).  Every wait is bounded.
#pragma once
#include "common.cuh"

namespace ssm {

constexpr unsigned long long kTcWaitNs = 200000000ull;  // 200 ms

__device__ __forceinline__ uint32_t tc_smem(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool tc_try(uint32_t mbar, unsigned phase) {
  unsigned done = 0;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(mbar), "r"(phase)
      : "memory");
  return done != 0;
}

__device__ __forceinline__ bool tc_wait(uint32_t mbar, unsigned phase) {
  if (tc_try(mbar, phase)) return true;
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
    if (tc_try(mbar, phase)) return true;
    // the clock also runs while another process has the GPU: one more look
    if (globaltimer_ns() - t0 > kTcWaitNs) return tc_try(mbar, phase);
  }
}

// the same for a whole warp: one verdict for all lanes
__device__ __forceinline__ bool tc_wait_warp(uint32_t mbar, unsigned phase) {
  return __all_sync(0xffffffffu, tc_wait(mbar, phase)) != 0;
}

__device__ __forceinline__ void tc_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

// The forms below are executed by a whole warp (elect.sync picks the lane that
// issues, the same one every time): with warp-uniform control flow around them
// the descriptors live in uniform registers.

// arrives on mbar when every MMA this warp has issued is done
__device__ __forceinline__ void tc_commit_warp(uint32_t mbar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(mbar)
      : "memory");
}

__device__ __forceinline__ void tc_mma_f16_warp(uint32_t acc, uint64_t da, uint64_t db, uint32_t idesc, uint32_t add) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %4, 0;\n\telect.sync _|q, 0xffffffff;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(acc),
      "l"(da), "l"(db), "r"(idesc), "r"(add)
      : "memory");
}

__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}

// waits for this warp's tcgen05.ld; the values pass through so that no use of
// them moves ahead of the wait
__device__ __forceinline__ void tc_ld_wait(uint32_t (&v)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                 "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
               :
               : "memory");
}

// one thread: `bytes` (a multiple of 16, both addresses 16-byte aligned) from
// global to shared memory, completing on mbar together with this arrival
__device__ __forceinline__ void tc_bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t mbar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(mbar)
               : "memory");
}

__device__ __forceinline__ void tc_bulk_prefetch(const void *src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(src)), "r"(bytes) : "memory");
}

// one thread: adds `bytes` (a multiple of 16, both addresses 16-byte aligned) of
// 32-bit words in shared memory to global memory, atomically word by word
__device__ __forceinline__ void tc_bulk_add_u32(void *dst, uint32_t src, uint32_t bytes) {
  asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.u32 [%0], [%1], %2;" ::"l"(
                   __cvta_generic_to_global(dst)),
               "r"(src), "r"(bytes)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// ... and waits until they are done (the copy unit's own transfers: always ends)
__device__ __forceinline__ void tc_bulk_store_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

}  // namespace ssm
