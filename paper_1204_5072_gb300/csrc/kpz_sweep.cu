// kpz_sweep.cu -- Monte Carlo sweeps of the octahedron KPZ model on GB300.
//
// One launch makes one sweep, or several chained ones. The resident warps take
// runs of P.run tiles of one tile row from a work queue (run::sweep_run, kpz_run.cuh); the Sec. 3
// decomposition and the Sec. 2.1 update rule are documented there, in
// kpz_rounds.cuh and in kpz_tilemem.cuh. On the p = 1, q = 0 path the Philox
// round keys are read from shared memory instead of being advanced per draw
// (at general rates that took 1.41 ms a sweep at L = 2^16 against 1.27).
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "kpz_gridsync.cuh"
#include "kpz_run.cuh"

namespace kpz {
namespace {

using run::WarpStage;
using run::kFull;
using run::kMaxWarpsPerCta;

// Persistent sweep: the resident warps take chunks of P.run tiles of one tile
// row from a work queue (row by row, one atomic per chunk, fetched a chunk
// ahead), so faster SMs take more chunks and the tail is one chunk. Every warp
// makes exactly one fetch past the last chunk; the warp whose fetch is the last
// of all returns the counter to zero for the next launch.
//
// kChain: n sweeps in a launch, without a barrier between them. A chunk waits
// for those rows of the sweep before that touch its sites, by done[], the
// chunks of an ordered row finished in this launch. Rows are ordered by where
// they start: the first row of a sweep is the first to start beyond the start y
// of the first one before it, y' = y + D, 1 <= D <= H (H the tile height). Row i
// covers, with its halo, y' + iH .. y' + iH + H; rows m of the sweep before
// cover y + mH .. y + mH + H, so m = i, i + 1 and, for D = H, i + 2 touch it (and
// the sweeps before that are done where those rows are). They were taken from
// the queue most of a sweep earlier, so the wait is over before it begins; the
// half-empty last wave and the launch that each sweep used to end with are left
// to the last one. A chunk waits only for chunks taken before it, so no wait is
// circular, whatever is resident; waits are bounded in time like all grid waits.
//
// Two orders of the same steps. With many chunks a warp (tight = false) the
// next chunk is taken from the queue while one is swept and a chunk is reported
// while the next one's rows are looked up: neither latency is seen, but every
// warp holds two chunks. With few (below three a warp and sweep) that leaves
// too little of a sweep between a row and the rows that wait for it, so a chunk
// is reported at once and the next one taken when it can begin: us per sweep,
// tight / not, p = 1: L = 8192 14.3 / 33, L = 32768 120 / 126 (2.7 chunks a
// warp), L = 65536 490 / 460. For the same reason warps beyond 0.6 of a sweep's
// chunks stay out (L = 8192 p = 1: 14.3, with all that fit 23).
//
// us per sweep at p = 1 / 0.95, a launch per sweep and chained: L = 8192 25 /
// 36.7 and 14.3 / 24.7, L = 16384 47 / 100 and 37 / 81, L = 32768 138 / 340 and
// 120 / 310, L = 65536 463 / 1275 and 467 / 1230.

// One warp: waits until the rows that ordered row i depends on have `want` chunks
// done, and reports a chunk of row `prev` (~0: none) meanwhile; false when the
// wait ran out of time. Lanes 0..2 acquire the counters; a vote orders no memory,
// so the warp is synchronised before the others read what the counters stand
// for. That order is also what keeps the cp.async copies through L1 (kpz_run.cuh)
// fresh now that sweeps share a launch.
__device__ __forceinline__ bool rows_done(uint32_t* done, uint32_t i, uint32_t nty, uint32_t want, uint32_t prev,
                                          uint32_t lane, GridSync* sync) {
  const uint32_t* d = done + ((i + lane) & (nty - 1u));
  auto ready = [&] { return __all_sync(kFull, lane > 2u || gridsync::ld_acquire(d) >= want); };
  const bool ok = ready();
  if (lane == 0u && prev != ~0u) gridsync::red_release(done + prev);
  if (ok) {
    __syncwarp();
    return true;
  }
  const uint64_t t0 = gridsync::now_ns();
  for (uint32_t it = 1; !ready(); ++it) {
    if ((it & 63u) == 0u && __any_sync(kFull, gridsync::gave_up(sync, t0))) {
      if (lane == 0u) atomicExch(&sync->err, 1u);
      return false;
    }
  }
  __syncwarp();
  return true;
}

template <int kMode, int CR, bool kC2>
struct StageOf {
  using type = WarpStage<CR>;
};
template <int kMode>
struct StageOf<kMode, 1, false> {
  using type = std::conditional_t<kMode == run::kGrowth, WarpStage<1>, run::WarpStageMem<1>>;
};
template <int kMode, int CR, bool kC2, bool kChain>
__device__ __forceinline__ void sweep(const SweepParams& P, uint32_t n, uint32_t* done, GridSync* sync, bool tight) {
  constexpr bool kGeneral = kMode != run::kGrowth;
  using Stage = typename StageOf<kMode, CR, kC2>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Stage& ws = reinterpret_cast<Stage*>(smem_raw)[threadIdx.x >> 5];
  __shared__ uint4 rk[kPhiloxRounds / 2];   // Philox round keys of (k0, k1)
  if (!kGeneral && threadIdx.x < kPhiloxRounds / 2) {
    const uint32_t r = 2u * threadIdx.x;
    rk[threadIdx.x] = make_uint4(P.k0 + r * kPhiloxWeylA, P.k1 + r * kPhiloxWeylB,
                                 P.k0 + (r + 1u) * kPhiloxWeylA, P.k1 + (r + 1u) * kPhiloxWeylB);
  }
  __shared__ tilemem::QuadTab tab;
  if (kGeneral && threadIdx.x < 4u) tilemem::fill_quad_tab(tab, threadIdx.x);
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t W = gridDim.x * (blockDim.x >> 5);
  const uint32_t cpr = P.ntx / P.run;              // chunks per tile row
  const uint32_t nchunks = cpr * P.nty;            // chunks per sweep
  const uint32_t L = P.g.L;
  uint32_t s = (uint32_t)(*P.t_dev) + P.s_add;
  uint32_t c = 0;
  // Device layer: a random origin of the tile grid for every sweep.
  if constexpr (!kChain) {
    const uint4 o = philox(kTagOrigin << 28, 0u, s, P.sample, P.k0, P.k1);
    const uint32_t ox = o.x & (L - 1u), oy = o.y & (L - 1u);
    if (lane == 0) c = atomicAdd(P.queue, 1u);
    c = __shfl_sync(kFull, c, 0);
    while (c < nchunks) {
      uint32_t next = 0;
      if (lane == 0) next = atomicAdd(P.queue, 1u);
      const uint32_t ty = c / cpr;
      run::sweep_run<kMode, CR, !kGeneral, false, kC2>(P, ws, rk, tab, lane, s, ox, oy, ty, (c - ty * cpr) * P.run,
                                                         P.run);
      c = __shfl_sync(kFull, next, 0);
    }
    if (lane == 0 && c == nchunks + W - 1u) atomicExch(P.queue, 0u);
  } else {
    const uint32_t H = L / P.nty;
    uint32_t y = 0u, prev = ~0u;
    if (lane == 0) c = atomicAdd(P.queue, 1u);
    c = __shfl_sync(kFull, c, 0);
    for (uint32_t k = 0; k < n; ++k, ++s, c -= nchunks) {   // c counts from the sweep's first chunk
      const uint4 o = philox(kTagOrigin << 28, 0u, s, P.sample, P.k0, P.k1);
      const uint32_t ox = o.x & (L - 1u), oy = o.y & (L - 1u);
      y = k == 0u ? oy : y + ((oy - y - 1u) & (H - 1u)) + 1u;   // where the first ordered row starts
      const uint32_t first = (y - oy) / H;
      while (c < nchunks) {
        uint32_t next = 0;
        if (lane == 0 && !tight) next = atomicAdd(P.queue, 1u);
        const uint32_t i = c / cpr;
        if (!rows_done(done, i, P.nty, k * cpr, prev, lane, sync)) return;
        prev = tight ? ~0u : i;
        run::sweep_run<kMode, CR, !kGeneral, false, kC2>(P, ws, rk, tab, lane, s, ox, oy, (first + i) & (P.nty - 1u),
                                                           (c - i * cpr) * P.run, P.run);
        __syncwarp();
        if (lane == 0 && tight) {
          gridsync::red_release(done + i);
          next = atomicAdd(P.queue, 1u);
        }
        c = __shfl_sync(kFull, next, 0) - k * nchunks;
      }
    }
    if (lane == 0 && prev != ~0u) gridsync::red_release(done + prev);
    if (lane == 0 && c == W - 1u) atomicExch(P.queue, 0u);
  }
}

constexpr int min_ctas(int mode, int cr) { return cr == 1 ? (mode != run::kGrowth ? 2 : 3) : (mode != run::kGrowth ? 1 : 2); }
template <int kMode, int CR, bool kC2>
__global__ void __launch_bounds__(256, min_ctas(kMode, CR)) sweep_kernel(const SweepParams P) {
  sweep<kMode, CR, kC2, false>(P, 1u, nullptr, nullptr, false);
}
template <int kMode, int CR, bool kC2>
__global__ void __launch_bounds__(256, min_ctas(kMode, CR)) sweep_chain_kernel(const SweepParams P, uint32_t n, uint32_t* done,
                                                                               GridSync* sync, bool tight) {
  sweep<kMode, CR, kC2, true>(P, n, done, sync, tight);
}
template <int kMode, int CR, bool kC2, bool kChain>
constexpr auto kernel_of() {
  if constexpr (kChain) return &sweep_chain_kernel<kMode, CR, kC2>;
  else return &sweep_kernel<kMode, CR, kC2>;
}

// SMs, and resident CTAs per SM of one sweep kernel at wpc warps per CTA (cached
// per device).
struct Room {
  uint32_t sms, per_sm;
};
template <int kMode, int CR, bool kC2, bool kChain>
cudaError_t resident_ctas(uint32_t wpc, Room& room) {
  constexpr int kMaxDev = 64;
  static std::mutex mu;
  static Room cache[kMaxDev][kMaxWarpsPerCta + 1] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  if (dev < kMaxDev && cache[dev][wpc].sms) { room = cache[dev][wpc]; return cudaSuccess; }
  const int bytes = (int)(kMaxWarpsPerCta * sizeof(typename StageOf<kMode, CR, kC2>::type));
  e = cudaFuncSetAttribute(kernel_of<kMode, CR, kC2, kChain>(), cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  int per_sm = 0, sms = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel_of<kMode, CR, kC2, kChain>(), (int)(wpc * 32u),
                                                    wpc * sizeof(typename StageOf<kMode, CR, kC2>::type));
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  room = Room{(uint32_t)(sms > 0 ? sms : 1), (uint32_t)(per_sm > 0 ? per_sm : 1)};
  if (dev < kMaxDev) cache[dev][wpc] = room;
  return cudaSuccess;
}

template <int kMode, int CR, bool kC2, bool kChain>
cudaError_t launch_as(const SweepParams& P, uint32_t wpc, uint32_t n, uint32_t* done, GridSync* sync, cudaStream_t st) {
  Room room;
  cudaError_t e = resident_ctas<kMode, CR, kC2, kChain>(wpc, room);
  if (e != cudaSuccess) return e;
  // One wave of resident warps, fewer if there are fewer tiles than warps; of
  // chained sweeps at most 0.6 of the chunks, in whole CTAs per SM.
  const uint64_t tiles = (uint64_t)P.ntx * P.nty, chunks = (uint64_t)P.runs_x * P.nty;
  uint64_t blocks = std::min<uint64_t>((uint64_t)room.per_sm * room.sms, (tiles + wpc - 1) / wpc);
  const size_t smem = wpc * sizeof(typename StageOf<kMode, CR, kC2>::type);
  if constexpr (kChain) {
    uint64_t most = std::max<uint64_t>(1u, chunks * 6u / 10u / wpc);
    if (most > room.sms) most -= most % room.sms;
    blocks = std::min(blocks, most);
    e = cudaMemsetAsync(done, 0, P.nty * sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
    sweep_chain_kernel<kMode, CR, kC2>
        <<<(unsigned)blocks, wpc * 32u, smem, st>>>(P, n, done, sync, chunks < 3u * blocks * wpc);
  } else {
    sweep_kernel<kMode, CR, kC2><<<(unsigned)blocks, wpc * 32u, smem, st>>>(P);
  }
  return cudaSuccess;
}

template <int kMode, int CR, bool kC2 = false>
cudaError_t launch_cr(const SweepParams& P, uint32_t wpc, uint32_t n, uint32_t* done, GridSync* sync, cudaStream_t st) {
  if constexpr (!(kC2 && kMode != run::kGrowth)) {
    if (n != 1u) return launch_as<kMode, CR, kC2, true>(P, wpc, n, done, sync, st);
  }
  return n == 1u ? launch_as<kMode, CR, kC2, false>(P, wpc, n, done, sync, st) : cudaErrorInvalidValue;
}

__global__ void advance_kernel(uint64_t* t_dev, uint32_t n) { *t_dev += n; }

}  // namespace

// Sweeps are chained where the end of a sweep is a good part of it and a sweep
// has chunks enough to hide the waits: from 1024 chunks (L = 4096, runs of one
// tile, p = 1: 14.7 -> 11.6 us; L = 1024, 16 chunks: 14 -> 20, so not there),
// and below 2^17 tiles (L = 65536: p = 1 463 -> 467, rates with a 0 or 1 1264 ->
// 1276), but at general rates at any size (L = 65536: 1275 -> 1230). 2 x 2 cells
// at general rates lose (L = 16384: 235 -> 293), 256-row tiles at p = 1 from L =
// 32768 (142 -> 150; L = 16384: 54.5 -> 43.6). About 2^40 attempts a launch.
uint32_t sweeps_per_launch(const SweepParams& P) {
  const uint64_t chunks = (uint64_t)P.runs_x * P.nty, sites = (uint64_t)P.g.L * P.g.L;
  const run::Mode mode = run::mode_of(P);
  if (chunks < 1024u || (P.cell == 2u && mode != run::kGrowth)) return 1u;
  if (mode == run::kGrowth && P.nty != P.ntx && P.ntx * P.nty >= 1u << 15) return 1u;
  if ((uint64_t)P.ntx * P.nty >= 1u << 17 && mode != run::kInner) return 1u;
  return (uint32_t)std::max<uint64_t>(1u, std::min<uint64_t>({(1ull << 40) / sites, (1ull << 31) / chunks, 1ull << 16}));
}

cudaError_t launch_sweep(const SweepParams& P, uint32_t warps_per_cta, uint32_t n, uint32_t* done, GridSync* sync,
                         cudaStream_t st) {
  // The tile height 128 CR follows from the number of tile rows.
  const uint32_t wpc = warps_per_cta ? warps_per_cta : 8u;
  if (wpc > kMaxWarpsPerCta) return cudaErrorInvalidValue;
  const uint32_t tile_y = P.g.L / P.nty;
  cudaError_t e;
  const run::Mode mode = run::mode_of(P);
  const bool general = mode != run::kGrowth;   // the variants without TileMem have one general form
  if (P.cell == 2u && tile_y == kTile)
    e = general ? launch_cr<run::kEdgeRate, 1, true>(P, wpc, n, done, sync, st) : launch_cr<run::kGrowth, 1, true>(P, wpc, n, done, sync, st);
  else if (P.cell == 2u)
    return cudaErrorInvalidValue;
  else if (tile_y == kTile)
    e = mode == run::kInner ? launch_cr<run::kInner, 1>(P, wpc, n, done, sync, st)
        : general           ? launch_cr<run::kEdgeRate, 1>(P, wpc, n, done, sync, st)
                            : launch_cr<run::kGrowth, 1>(P, wpc, n, done, sync, st);
  else if (tile_y == 2u * kTile)
    e = general ? launch_cr<run::kEdgeRate, 2>(P, wpc, n, done, sync, st) : launch_cr<run::kGrowth, 2>(P, wpc, n, done, sync, st);
  else
    return cudaErrorInvalidValue;
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_advance(uint64_t* t_dev, uint32_t n, cudaStream_t st) {
  advance_kernel<<<1, 1, 0, st>>>(t_dev, n);
  count_launch();
  return cudaGetLastError();
}

}  // namespace kpz
