// kpz_observe.h -- launch interface of the exact W^2 reduction (kpz_observe.cu).
#pragma once
#include "kpz_internal.h"

namespace kpz {

// Where the reduction puts its results; device-accessible memory, which may be
// mapped host memory (readable once the stream is synchronised).
struct RoughOut {
  uint32_t* ticket;                 // device word, zero between launches
  long long* sums;                  // [0] S1, [1] S2 lo, [2] S2 hi, [3] *h00, [4] *err
  const unsigned long long* h00;    // may be null
  const uint32_t* err;              // may be null
};

// Exact height sums, eq. (Wdef), in the gauge h(0,0) = 0; scratch: 24 L / 32
// bytes of device memory, 8-byte aligned.
cudaError_t launch_roughness(const uint32_t* lat, Geometry g, void* scratch, const RoughOut& out, cudaStream_t st);

}  // namespace kpz
