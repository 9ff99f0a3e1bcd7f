// PTX helpers shared by the tcgen05 kernels: bounded mbarrier waits, arrivals
// and MMA commits.
#pragma once

#include <cstdint>

namespace rtcc3 {

// Waits on other warps' progress spin for at most a budget of clock cycles
// (a kernel argument, kWaitBudget by default, about 2 s).  Waits for this
// CTA's own asynchronous work to land (its TMA / bulk copies, its MMAs) at
// exit use kDrainBudget: that work completes by itself, so these waits end
// whatever the progress budget was; they are what makes giving up safe
// (no copy or MMA may still target the CTA's shared or tensor memory when it
// frees them).
constexpr long long kWaitBudget = 4000000000LL;
constexpr long long kDrainBudget = 4000000000LL;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok = 0;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, long long budget) {
  if (mbar_try(bar, parity)) return true;  // most waits: the clock is not read
  const long long t0 = clock64();
  while (!mbar_try(bar, parity))
    if (clock64() - t0 > budget) return false;
  return true;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}

}  // namespace rtcc3
