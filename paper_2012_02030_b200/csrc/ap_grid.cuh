// A bounded barrier for CTAs of one cooperative launch (all of them are resident).
#pragma once

#include "ap_common.cuh"

namespace ap {

__device__ __forceinline__ uint32_t ld_acquire_gpu(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// By one thread: waits (bounded) until `arrivals` has been counted up to `target`.
__device__ __forceinline__ bool reached(const uint32_t *arrivals, uint32_t target) {
  constexpr uint32_t kMaxPolls = 1u << 22;
  uint32_t polls = 0;
  while (ld_acquire_gpu(arrivals) < target)
    if (++polls >= kMaxPolls) return false;
  return true;
}

// By all threads of a CTA: returns once `arrivals` has been counted up to `target` (every participant adds one), with
// everything the others wrote before it visible.  false, and the device status word raised, if that takes too long.
__device__ __forceinline__ bool cta_barrier(uint32_t *arrivals, uint32_t target, unsigned *err) {
  __shared__ int ok_s;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(arrivals, 1u);
    ok_s = reached(arrivals, target);
    if (!ok_s) atomicOr(err, kDevErrTimeout);
    __threadfence();
  }
  __syncthreads();
  return ok_s != 0;
}

}  // namespace ap
