// kpz_rsu.h -- launch interface of the exact random-sequential sweeps (kpz_rsu.cu).
#pragma once
#include "kpz_gridsync.cuh"
#include "kpz_internal.h"

namespace kpz {

// Device bytes of scratch the sweeps of an L x L lattice need (per-site lists
// of attempts and their progress, 20 L^2 bytes).
size_t rsu_scratch_bytes(uint32_t L);
// n sweeps from *P.t_dev on (n >= 1), which the launch advances by n, of
// random-sequential updates equal bit for bit to making the L^2 attempts of a
// sweep one at a time; `scratch` holds rsu_scratch_bytes(L) device bytes.
cudaError_t launch_rsu(const SweepParams& P, uint32_t n, void* scratch, GridSync* sync, cudaStream_t st);

}  // namespace kpz
