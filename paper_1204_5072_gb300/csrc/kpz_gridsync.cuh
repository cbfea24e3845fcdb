// kpz_gridsync.cuh -- building blocks of bounded waits between blocks, release
// to acquire: grid-wide barriers in cooperative launches (a counter that every
// block raises once a step) and the row counters of chained sweeps; a wait
// gives up after kWaitNs (or GridSync.wait_ms).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace kpz {

// Device words of a context's persistent kernels (in its 256-byte block of
// small values, on a 128-byte line of its own; zero between launches).
struct alignas(8) GridSync {
  uint32_t arrived;    // blocks that have finished a step
  uint32_t finished;   // blocks that have finished the launch
  uint32_t err;        // 1: a wait ran out of time; stays set
  uint32_t wait_ms;    // bound of every wait, 0: kWaitNs; nothing here sets it, a test does in its buffer
  uint32_t fired[4];   // kpz_rsu.cu: attempts made in a round
};

namespace gridsync {

constexpr uint64_t kWaitNs = 10000000000ull;

__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Whether a wait that began at t0 is over: another one gave up, or its time is.
// Out of line: eight random-sequential sweeps at L = 1024 take 1365 us, 1412 with
// it inlined; the other waits do not notice.
static __device__ __noinline__ bool gave_up(const GridSync* s, uint64_t t0) {
  uint32_t err, ms;
  asm volatile("ld.volatile.global.v2.u32 {%0, %1}, [%2];" : "=r"(err), "=r"(ms) : "l"(&s->err) : "memory");
  return err != 0u || now_ns() - t0 > (ms ? ms * 1000000ull : kWaitNs);
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
    if ((it & 63u) == 0u && gave_up(s, t0)) {
      atomicExch(&s->err, 1u);
      return false;
    }
  }
  return true;
}

}  // namespace gridsync
}  // namespace kpz
