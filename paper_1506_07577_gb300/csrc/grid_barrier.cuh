// Grid-wide barrier of a cooperative launch (device code): one counter that
// only grows, arrivals with release, waits with acquire order.
#pragma once

namespace ebb {

constexpr long long kGridWaitCycles = 2000000000LL;  // about 1 s at 2 GHz

__device__ __forceinline__ void arrive_release(unsigned* bar) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
}
// Wait until the counter has reached `target` (which may have wrapped);
// false after about a second.
__device__ __forceinline__ bool wait_acquire(const unsigned* bar, unsigned target) {
  const long long t0 = clock64();
  while (true) {
    unsigned n;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(n) : "l"(bar) : "memory");
    if ((int)(n - target) >= 0) return true;
    if (clock64() - t0 > kGridWaitCycles) return false;
  }
}

// The barrier in two halves, so that work no other block waits for can run in
// between.  Round r is complete at r * gridDim.x arrivals.
__device__ __forceinline__ void grid_arrive(unsigned* bar, unsigned& round) {
  ++round;
  __syncthreads();
  if (threadIdx.x == 0) arrive_release(bar);
}

}  // namespace ebb
