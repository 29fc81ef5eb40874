// Bounded waits on words that other CTAs of a cooperative launch write.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lfx {

constexpr uint32_t kWaitPolls = 1u << 22;   // seconds of polls; a wait that runs out gives up
constexpr uint32_t kTestPolls = 1u << 12;   // milliseconds: the limit of waits that a test makes run out

__device__ __forceinline__ unsigned ld_relaxed(const unsigned *p) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
// thread 0: until *p reaches target (counts grow; wrap-safe); false after polls tries
__device__ __forceinline__ bool wait_for(const unsigned *p, unsigned target, uint32_t polls) {
  for (uint32_t i = 0; i < polls; ++i)
    if ((int)(ld_relaxed(p) - target) >= 0) {
      fence_gpu();
      return true;
    }
  return false;
}
// thread 0 of a CTA whose other threads have reached a barrier: count the CTA in (its writes before the count)
__device__ __forceinline__ void arrive(unsigned *p) {
  fence_gpu();
  asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}

}  // namespace lfx
