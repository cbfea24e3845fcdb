// kpz_resident.h -- many sweeps of one small or medium lattice per launch.
#pragma once
#include "kpz_internal.h"

namespace kpz {

// Device words the resident kernels keep between launches (in the context's
// 256-byte block of small values, on a 128-byte line of its own; all zero
// between launches).
struct ResidentSync {
  uint32_t arrived;   // grid barrier: blocks that have finished a step
  uint32_t finished;  // blocks that have finished the launch
  uint32_t err;       // 1: a wait ran out of time; stays set
};

// How launch_resident would serve this lattice on the current device: 0 not at
// all, 1 grid, 2 cluster. Served: 128 x 128 tiles of 4 x 4 cells, dead-border
// tiles or tile sets, at most 1024 tiles swept at a time. Sets the kernels'
// attributes on the device, so it precedes the first launch there.
uint32_t resident_kind(const SweepParams& P, bool tilesets);

// n sweeps from *P.t_dev on (n >= 1), which the launch advances by n. scratch:
// 2 L^2 / 8 bytes.
cudaError_t launch_resident(const SweepParams& P, bool tilesets, uint32_t kind, uint32_t n, uint32_t* scratch,
                            ResidentSync* sync, cudaStream_t st);

}  // namespace kpz
