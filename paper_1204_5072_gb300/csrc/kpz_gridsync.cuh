// kpz_gridsync.cuh -- building blocks of bounded waits between blocks, release
// to acquire: grid-wide barriers in cooperative launches (a counter that every
// block raises once a step) and the row counters of chained sweeps; a wait
// gives up after kWaitNs.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace kpz {

// Device words of a context's persistent kernels (in its 256-byte block of
// small values, on a 128-byte line of its own; zero between launches).
struct GridSync {
  uint32_t arrived;    // blocks that have finished a step
  uint32_t finished;   // blocks that have finished the launch
  uint32_t err;        // 1: a wait ran out of time; stays set
  uint32_t fired[4];   // kpz_rsu.cu: attempts made in a round
};

namespace gridsync {

constexpr uint64_t kWaitNs = 10000000000ull;   // bound of every grid wait

__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t add_acq_rel(uint32_t* p, uint32_t v) {
  uint32_t old;
  asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}
__device__ __forceinline__ void red_release(uint32_t* p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}
// One thread: waits until *s.arrived >= want; false (and s.err set) when the
// wait ran out of time or another block's did.
__device__ __forceinline__ bool wait_for(GridSync* s, uint32_t want) {
  if (ld_acquire(&s->arrived) >= want) return true;
  const uint64_t t0 = now_ns();
  for (uint32_t it = 1; ld_acquire(&s->arrived) < want; ++it) {
    if ((it & 63u) == 0u && (now_ns() - t0 > kWaitNs || *(volatile uint32_t*)&s->err)) {
      atomicExch(&s->err, 1u);
      return false;
    }
  }
  return true;
}

}  // namespace gridsync
}  // namespace kpz
