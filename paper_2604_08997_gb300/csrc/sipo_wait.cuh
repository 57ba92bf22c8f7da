// sipo_wait.cuh -- bounded waits on shared-memory barriers (mbarrier) and their
// self-test: a wait that outlives its budget of clock cycles gives up and says
// so, instead of holding the device.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace sipo {

constexpr long long kWaitCycles = 4000000000LL;  // ~2 s at 2 GHz: a wait that long has failed

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait for the phase with the given parity; false once `budget` SM
// clock cycles have passed without it.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long budget = kWaitCycles) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > budget) return false;
  return true;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Self-test of the bounded wait: one mbarrier expecting one arrival, which
// thread 0 makes only when `arrive` is set; every thread waits on the first
// phase with a budget of `budget` cycles.  out[0] = number of threads whose wait
// gave up (blockDim.x when nothing arrives, 0 otherwise).
__global__ void k_wait_selftest(long long budget, int arrive, unsigned int* out) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0 && arrive) mbar_arrive(&bar);
  if (!mbar_wait(&bar, 0u, budget)) atomicAdd(out, 1u);
}

}  // namespace sipo
