// kpz_rsu.cu -- random-sequential updates on the GPU, equal bit for bit to
// making the attempts one at a time: the undecomposed dynamics that the
// decompositions of Sec. 3 (arXiv:1204.5072) approximate.
//
// Sweep s is the L^2 attempts a = 0 .. L^2 - 1 in order; attempt a draws
//   w = philox(4<<28, a, s, sample): site (w0 & (L-1), w1 & (L-1)), U = w2 >> 16
// and applies eq. (rule) there, a minimum rising when U < Tp and a maximum
// falling when U < Tq (the stream of the oracle's orc_rsu_run). An update at
// a site reads that site and its four neighbours and changes only the site,
// so attempt a depends on an earlier attempt b only when their sites are the
// same or neighbours. The sweep therefore runs in rounds: in each round every
// site whose next attempt comes before the next attempt of each of its four
// neighbours makes it. Two such sites are never neighbours, and every attempt
// waits for all earlier attempts that touch it, so the lattice after the sweep
// is the one the sequential order gives (a conservative parallel
// discrete-event schedule). A round reads the sites' next attempts of the
// previous round (two buffers), so no site sees a neighbour's move of the same
// round. There is always progress (the earliest pending attempt of the sweep
// is always ready).
//
// One cooperative launch makes all sweeps of a call; a grid barrier ends each
// phase and round, and the blocks count the attempts made themselves. What
// bounds a sweep is some thirty rounds of a pass over the L^2 next attempts
// and a barrier each. A site keeps its attempts as an unsorted list (one
// exchange per attempt; one attempt per site on average) and its next one in
// an array, so a round reads that array alone, 16 bytes a thread and four
// neighbours' worth beside them; the ready sites go through a list, so that
// every thread has one to work off (a thread doing its own four in turn waits
// for memory four times). Counting, prefix sums, scattering and sorting
// into buckets, rounds that looked up five buckets a site, and the host
// polling every eight rounds took 466 us a sweep at L = 1024 and 6.3 ms at
// L = 4096; this takes 154 us (320 with each thread doing its own four) and 2.4 ms.
#include <algorithm>

#include "kpz_rsu.h"

namespace kpz {
namespace {

constexpr uint32_t kTagRsu = 4u, kNone = 0xffffffffu, kThreads = 1024, kBatch = 2;

__device__ __forceinline__ size_t site_word(const Geometry& g, uint32_t x, uint32_t y) {
  return g.word(x >> 7, plane(y & 3u, x & 3u), y >> 2);
}
__device__ __forceinline__ uint32_t bit_of(const uint32_t* lat, const Geometry& g, uint32_t x, uint32_t y) {
  return (__ldcg(lat + site_word(g, x, y)) >> ((x >> 2) & 31u)) & 1u;
}

// First attempt after `last` (kNone: of all) in the list that starts at e;
// list entries are attempt + 1, 0 ends it.
__device__ __forceinline__ uint32_t next_attempt(const uint32_t* next, uint32_t e, uint32_t last) {
  uint32_t best = kNone;
  while (e) {
    const uint32_t a = e - 1u;
    if (a < best && (last == kNone || a > last)) best = a;
    e = __ldcg(next + a);
  }
  return best;
}

struct Scratch {
  uint32_t *head[2], *next, *cur[2];   // L^2 words each; head[0] of an even sweep is zero at its start
};

__global__ void __launch_bounds__(kThreads, 1) rsu_kernel(const SweepParams P, uint32_t nsweeps, Scratch S, GridSync* sync) {
  __shared__ uint32_t ok_s, fired_s, list[kThreads * kBatch * 2u];   // of four sites of a row at most two are ready
  const uint32_t L = P.g.L, m = L - 1u, n = L * L;
  const uint32_t gt = blockIdx.x * kThreads + threadIdx.x, T = gridDim.x * kThreads;
  const uint32_t t0 = (uint32_t)(*(const volatile uint64_t*)P.t_dev) + P.s_add;
  uint32_t step = 0;
  auto barrier = [&]() -> bool {
    __syncthreads();
    ++step;
    if (threadIdx.x == 0) {
      gridsync::red_release(&sync->arrived);
      ok_s = gridsync::wait_for(sync, step * gridDim.x) ? 1u : 0u;
    }
    __syncthreads();
    return ok_s != 0u;
  };
  if (threadIdx.x == 0) fired_s = 0u;
  uint32_t round = 0;   // over all sweeps: its counter is sync->fired[round & 3]
  for (uint32_t i = gt; i < n; i += T) __stcg(S.head[0] + i, 0u);
  if (!barrier()) return;
  for (uint32_t k = 0; k < nsweeps; ++k) {
    const uint32_t s = t0 + k;
    uint32_t* head = S.head[k & 1u];
    uint32_t* other = S.head[(k & 1u) ^ 1u];
    for (uint32_t a = gt; a < n; a += T) {
      const uint4 w = philox(kTagRsu << 28, a, s, P.sample, P.k0, P.k1);
      __stcg(S.next + a, atomicExch(head + (size_t)(w.y & m) * L + (w.x & m), a + 1u));
    }
    if (!barrier()) return;
    for (uint32_t i = gt; i < n; i += T) {
      __stcg(S.cur[0] + i, next_attempt(S.next, __ldcg(head + i), kNone));
      __stcg(other + i, 0u);
    }
    if (!barrier()) return;
    uint32_t made = 0;
    for (uint32_t r = 0; made < n; ++r, ++round) {
      const uint32_t* in = S.cur[r & 1u];
      uint32_t* out = S.cur[(r & 1u) ^ 1u];
      uint32_t total = 0;   // attempts this block makes in the round (thread 0)
      for (uint32_t c0 = blockIdx.x * kThreads; c0 < n / 4u; c0 += kBatch * T) {
        // The sites that are ready, of kBatch chunks of four a thread, into a list ...
#pragma unroll
        for (uint32_t b = 0; b < kBatch; ++b) {
          const uint32_t c = c0 + b * T + threadIdx.x, i = 4u * c;
          uint32_t ready = 0;
          if (c < n / 4u) {
            const uint32_t x = i & m, y = i / L;
            const uint4 own = __ldcg(reinterpret_cast<const uint4*>(in + i));
            if ((own.x & own.y & own.z & own.w) != kNone) {
              const uint4 up = __ldcg(reinterpret_cast<const uint4*>(in + (size_t)((y + m) & m) * L + x));
              const uint4 dn = __ldcg(reinterpret_cast<const uint4*>(in + (size_t)((y + 1u) & m) * L + x));
              const uint32_t lf = __ldcg(in + (size_t)y * L + ((x + m) & m)), rt = __ldcg(in + (size_t)y * L + ((x + 4u) & m));
              // kNone is below nothing.
              ready = (own.x < min(min(lf, own.y), min(up.x, dn.x)) ? 1u : 0u) |
                      (own.y < min(min(own.x, own.z), min(up.y, dn.y)) ? 2u : 0u) |
                      (own.z < min(min(own.y, own.w), min(up.z, dn.z)) ? 4u : 0u) |
                      (own.w < min(min(own.z, rt), min(up.w, dn.w)) ? 8u : 0u);
            }
            __stcg(reinterpret_cast<uint4*>(out + i), own);
          }
          uint32_t cnt = __popc(ready), pre = cnt;   // places in the list: warp prefix, one atomic a warp
#pragma unroll
          for (int d = 1; d < 32; d <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, pre, d);
            if ((threadIdx.x & 31u) >= (uint32_t)d) pre += v;
          }
          uint32_t at = 0;
          if ((threadIdx.x & 31u) == 31u && pre) at = atomicAdd(&fired_s, pre);
          at = __shfl_sync(0xffffffffu, at, 31) + pre - cnt;
#pragma unroll
          for (uint32_t j = 0; j < 4u; ++j)
            if (ready >> j & 1u) list[at++] = i + j;
        }
        __syncthreads();
        // ... which the block's threads work off, one site each.
        const uint32_t count = fired_s;
        for (uint32_t f = threadIdx.x; f < count; f += kThreads) {
          const uint32_t i = list[f], x = i & m, y = i / L, a = __ldcg(in + i), e = __ldcg(head + i);
          // Eq. (rule) on the height bits: neighbour q is higher iff b(q) ^ b(site) == parity(site).
          const uint32_t bs = bit_of(P.lat, P.g, x, y), hp = (x + y + P.g.par) & 1u;
          const uint32_t bl = bit_of(P.lat, P.g, (x + m) & m, y), br = bit_of(P.lat, P.g, (x + 1u) & m, y);
          const uint32_t bd = bit_of(P.lat, P.g, x, (y + m) & m), bu = bit_of(P.lat, P.g, x, (y + 1u) & m);
          const uint32_t U = philox(kTagRsu << 28, a, s, P.sample, P.k0, P.k1).z >> 16;
          const uint32_t nh = ((bl ^ bs) == hp) + ((br ^ bs) == hp) + ((bd ^ bs) == hp) + ((bu ^ bs) == hp);
          if ((nh == 4u && U < P.Tp) || (nh == 0u && U < P.Tq)) {
            atomicXor(P.lat + site_word(P.g, x, y), 1u << ((x >> 2) & 31u));
            if (i == 0u) atomicAdd(P.h00, (unsigned long long)(long long)(nh == 4u ? 2 : -2));
          }
          __stcg(out + i, next_attempt(S.next, e, a));
        }
        __syncthreads();
        if (threadIdx.x == 0) {
          total += count;
          fired_s = 0u;
        }
        __syncthreads();
      }
      if (threadIdx.x == 0) {
        if (total) atomicAdd(&sync->fired[round & 3u], total);
        if (blockIdx.x == 0) __stcg(&sync->fired[(round + 2u) & 3u], 0u);   // last read two barriers ago
      }
      if (!barrier()) return;
      made += __ldcg(&sync->fired[round & 3u]);
      // A sweep needs a few dozen rounds; the bound only turns a defect into an error.
      if (r >= (1u << 16)) {
        if (threadIdx.x == 0) atomicExch(&sync->err, 1u);
        return;
      }
    }
  }
  // The last block out resets the counters and advances the sweep count.
  if (threadIdx.x == 0 && gridsync::add_acq_rel(&sync->finished, 1u) == gridDim.x - 1u) {
    sync->arrived = 0u;
    sync->finished = 0u;
    for (int i = 0; i < 4; ++i) sync->fired[i] = 0u;
    *const_cast<uint64_t*>(P.t_dev) += nsweeps;
  }
}

}  // namespace

size_t rsu_scratch_bytes(uint32_t L) { return 5 * (size_t)L * L * sizeof(uint32_t); }

cudaError_t launch_rsu(const SweepParams& P, uint32_t n, void* scratch, GridSync* sync, cudaStream_t st) {
  const size_t N = (size_t)P.g.L * P.g.L;
  uint32_t* w = static_cast<uint32_t*>(scratch);
  Scratch S{{w, w + N}, w + 2 * N, {w + 3 * N, w + 4 * N}};
  int dev = 0, per_sm = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, rsu_kernel, (int)kThreads, 0);
  if (e != cudaSuccess) return e;
  const uint32_t room = (uint32_t)std::max(per_sm * sms, 1);
  const uint32_t grid = (uint32_t)std::min<size_t>(room, (N / 4 + kThreads - 1) / kThreads);
  SweepParams Q = P;
  void* args[] = {&Q, &n, &S, &sync};
  e = cudaLaunchCooperativeKernel((const void*)rsu_kernel, dim3(grid), dim3(kThreads), args, 0, st);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace kpz
