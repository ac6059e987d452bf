// sv_tcgen05.cuh -- small wrappers over the PTX that the tensor-core sweeps share.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace sv {
namespace tc {

__device__ __forceinline__ uint32_t su32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// bounded wait for the phase of an mbarrier; false if the limit ran out
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t phase, int limit) {
  for (int it = 0; it < limit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(phase)
        : "memory");
    if (done) return true;
  }
  return false;
}

// the same for several warp roles that share a fail flag: a wait that runs out sets it,
// and every other wait then returns at once
__device__ __forceinline__ bool mbar_wait_or_fail(uint32_t bar, uint32_t phase, int limit, volatile int* fail) {
  for (int it = 0; it < limit; ++it) {
    if (mbar_wait(bar, phase, 1)) return true;
    if (*fail) return false;
  }
  *fail = 1;
  return false;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// UMMA shared-memory descriptor: K-major, no swizzle (layout type 0), version 1.  Low
// word: start address and lbo (bytes to the next core matrix along K), both / 16; a
// start further by `bytes` is the word + bytes / 16.  High word: sbo (bytes to the next
// 8-row group along M or N) / 16.
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr, uint32_t lbo) { return (saddr >> 4) | ((lbo >> 4) << 16); }
constexpr uint32_t desc_hi(uint32_t sbo) { return (sbo >> 4) | (1u << 14); }

// One MMA / commit by the lane with `on` set, executed by a whole warp with uniform
// operands: inside a branch of one lane the compiler moves every descriptor from vector
// to uniform registers, which took 75 clocks per MMA.
// The operands' 8-row groups follow each other (sbo = 128).
__device__ __forceinline__ void mma_f16(uint32_t on, uint32_t d, uint32_t a, uint32_t b, uint32_t idesc,
                                        uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p, q;\n .reg .b64 a, b;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
      " mov.b64 a, {%1, %6};\n mov.b64 b, {%2, %6};\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n}\n" ::"r"(d),
      "r"(a), "r"(b), "r"(idesc), "r"(accum), "r"(on), "n"(desc_hi(128)));
}
__device__ __forceinline__ void mma_commit(uint32_t on, uint32_t bar) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
      " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(bar),
      "r"(on)
      : "memory");
}
// 1 in one lane of a converged warp
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t on;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(on));
  return on;
}

// nine, ten consecutive accumulator columns of this lane
__device__ __forceinline__ void tmem_ld9(uint32_t taddr, uint32_t (&r)[9]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r[8]) : "r"(taddr + 8));
}

__device__ __forceinline__ void tmem_ld10(uint32_t taddr, uint32_t (&r)[10]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];" : "=r"(r[8]), "=r"(r[9]) : "r"(taddr + 8));
}

}  // namespace tc
}  // namespace sv
