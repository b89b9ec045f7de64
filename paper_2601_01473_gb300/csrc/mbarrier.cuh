// mbarrier.cuh -- shared-memory mbarriers with a wait that is bounded in time.
#pragma once

#include <stdint.h>

namespace agnes {

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Whether the phase with the given parity has completed.  try_wait may suspend
// the thread before it answers no, so waiting warps leave the shared-memory pipe
// to the others; for how long is up to the hardware, so polls do not bound a
// wait's time.
__device__ __forceinline__ bool mbar_poll(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// A wait gives up kMbarWaitNs after its first kMbarFastPolls polls, by the
// device's clock (or, should that stand still, after kMbarSlowPolls more).
constexpr int kMbarFastPolls = 64;
constexpr int kMbarSlowPolls = 1 << 24;
constexpr uint64_t kMbarWaitNs = 1000000000;

__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity) {
  const uint64_t start = global_ns();
  for (int it = 0; it < kMbarSlowPolls; ++it) {
    if (mbar_poll(bar, parity)) return true;
    if (global_ns() - start > kMbarWaitNs) break;
    __nanosleep(64);
  }
  return false;
}

// Waits for the phase with the given parity to complete; false when the time
// is up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  for (int it = 0; it < kMbarFastPolls; ++it)
    if (mbar_poll(bar, parity)) return true;
  return mbar_wait_slow(bar, parity);
}

}  // namespace agnes
