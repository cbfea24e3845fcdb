// kpz_resident.h -- many sweeps of one small or medium lattice per launch.
#pragma once
#include "kpz_gridsync.cuh"
#include "kpz_internal.h"

namespace kpz {

// How launch_resident would serve this lattice on the current device: 0 not at
// all, 1 grid, 2 cluster. Served: 128 x 128 tiles of 4 x 4 cells, dead-border
// tiles or tile sets, at most 1024 tiles swept at a time. Sets the kernels'
// attributes on the device, so it precedes the first launch there.
uint32_t resident_kind(const SweepParams& P, bool tilesets);

// n sweeps from *P.t_dev on (n >= 1), which the launch advances by n. scratch:
// 2 L^2 / 8 bytes.
cudaError_t launch_resident(const SweepParams& P, bool tilesets, uint32_t kind, uint32_t n, uint32_t* scratch,
                            GridSync* sync, cudaStream_t st);

}  // namespace kpz
