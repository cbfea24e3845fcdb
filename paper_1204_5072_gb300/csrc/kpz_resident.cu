// kpz_resident.cu -- many sweeps of one small or medium lattice in one launch
// (arXiv:1204.5072, Sec. 3 and 3.1; same dynamics and random streams as
// kpz_sweep.cu and kpz_tileset.cu, bit for bit).
//
// What bounds these sizes is latency, not work: at L = 4096 a sweep has 1024
// tiles for 608 warp schedulers, at L = 256 four. So every tile of a step has
// a warp of its own, and the chain a sweep cannot avoid -- window in, 16
// dependent rounds, changes out, everybody done -- is stripped of everything
// else:
//   - one launch runs all sweeps of a kpz_run call; a barrier of the cluster
//     (L <= 1024, lattice in distributed shared memory) or of the grid
//     separates them instead of a launch;
//   - the random numbers do not depend on the surface, so the Philox blocks of
//     the next step are drawn into shared memory by warps of their own or
//     while the barrier is pending, and a round only reads them;
//   - between sweeps the lattice is held in the frame of the last sweep's
//     origin: word (K, p, R) of the layout in kpz_common.cuh then belongs to
//     tile (K, R / 32) alone, so a tile goes back with 16 plain stores (with a
//     fixed frame every word is shared by two tiles and goes back as a
//     read-modify-write; red.xor took 45 cycles each, 1400 to 2400 a tile).
//     Two scratch lattices take turns; the last step writes the fixed frame.
// Microseconds per sweep, p = 1 / p = 0.95, against one launch per sweep with
// runs of 8 tiles (and of one tile, the fastest there): L = 256 1.9 / 3.1
// against 12.4 / 22.8 (10.2 / 15.9), L = 1024 2.7 / 4.3 against 25 / 63 (10.2 /
// 17.7), L = 4096 3.7 / 7.8 against 29 / 80 (14.1 / 25.8); tile sets at L = 2048
// 11.7 / 18.4 against 44 at p = 1. At L = 512 (one tile a block, one tile warp
// a scheduler) the 16 rounds take 2000 / 4300 cycles of a sweep's 3900 / 6400;
// the rest is the window's trip and the barrier. At L = 4096 and general rates
// the seven tiles of an SM bind it (logic and Philox pipes).
#include <algorithm>
#include <mutex>

#include "kpz_resident.h"
#include "kpz_tilemem.cuh"

namespace kpz {
namespace {

using tilemem::QuadTab;
using tilemem::TileMem;

// Random numbers of one tile and sweep, lane = cell row: position blocks of
// the eight round pairs and, at general rates, the acceptance block of each
// round and the outcome of its four deep numbers against both thresholds: bit
// 7 - r % 8 of byte k of deep[r / 8].x (.y) is set when the k-th tie of the row
// in round r is accepted as a minimum (maximum) (streams as in
// kpz_rounds.cuh), the rounds' quadrant offsets (tilemem::QuadTab) and the
// next sweep's origin.
template <bool kGeneral>
struct TileRand {
  uint4 pos[kRounds / 2][32];
  uint4 acc[kGeneral ? kRounds : 1][kGeneral ? 32 : 1];
  uint2 deep[kGeneral ? 2 : 1][kGeneral ? 32 : 1];
  uint4 at[kRounds], sh[kRounds];
  uint32_t origin[4];
};

// Four Philox blocks (counter words c0[i], c1, c2, c3) at once: ten rounds of
// one block are a serial chain, four chains keep the multiplier busy.
__device__ __forceinline__ void philox4(const uint32_t (&ctr)[4], uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                                        uint32_t k1, uint4 (&out)[4]) {
  uint32_t x[4], y[4], z[4], w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) { x[i] = ctr[i]; y[i] = c1; z[i] = c2; w[i] = c3; }
#pragma unroll
  for (int r = 0; r < kPhiloxRounds; ++r) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t hiA = __umulhi(kPhiloxMulA, x[i]), loA = kPhiloxMulA * x[i];
      const uint32_t hiB = __umulhi(kPhiloxMulB, z[i]), loB = kPhiloxMulB * z[i];
      x[i] = hiB ^ y[i] ^ k0;
      z[i] = hiA ^ w[i] ^ k1;
      y[i] = loB;
      w[i] = loA;
    }
    k0 += kPhiloxWeylA;
    k1 += kPhiloxWeylB;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) out[i] = make_uint4(x[i], y[i], z[i], w[i]);
}

// Origin of the tile grid of sweep s.
__device__ __forceinline__ uint2 origin_of(const SweepParams& P, uint32_t s) {
  const uint4 o = philox(kTagOrigin << 28, 0u, s, P.sample, P.k0, P.k1);
  return make_uint2(o.x & (P.g.L - 1u), o.y & (P.g.L - 1u));
}

// Draws part `part` of `parts` (1 or 2) of a tile's blocks.
template <bool kGeneral>
__device__ __forceinline__ void draw_tile(const SweepParams& P, const QuadTab& tab, TileRand<kGeneral>& B,
                                          uint32_t tid, uint32_t s, uint32_t lane, uint32_t part, uint32_t parts) {
  if (part == 0u) {
    const uint32_t w = philox(kTagSet << 28, tid, s, P.sample, P.k0, P.k1).x;
    const uint2 o = origin_of(P, s + 1u);
    if (lane < kRounds) {
      B.at[lane] = tab.at[(w >> (2u * lane)) & 3u];
      B.sh[lane] = tab.sh[(w >> (2u * lane)) & 3u];
    }
    if (lane == 0u) { B.origin[0] = o.x; B.origin[1] = o.y; }
  }
  uint4 o[4];
  if constexpr (kGeneral) {
    const uint32_t n = (kRounds / 2) / parts;
    uint32_t dp = 0u, dq = 0u;   // outcomes of four round pairs
    const uint32_t cp = tilemem::Rates<true>::deep_const(P.Tp), cq = tilemem::Rates<true>::deep_const(P.Tq);
    auto below = [](uint32_t lo, uint32_t hi, uint32_t c) { return tilemem::deep_below(lo, hi, c, ~0u) & 0x80808080u; };
#pragma unroll 1
    for (uint32_t rp = part * n; rp < part * n + n; ++rp) {
      const uint32_t c[4] = {(kTagPos << 28) | (lane << 3) | rp, (kTagAcc << 28) | (lane << 4) | (2u * rp),
                             (kTagAcc << 28) | (lane << 4) | (2u * rp + 1u), (kTagDeep << 28) | (lane << 8) | (rp << 4)};
      philox4(c, tid, s, P.sample, P.k0, P.k1, o);
      B.pos[rp][lane] = o[0];
      B.acc[2u * rp][lane] = o[1];
      B.acc[2u * rp + 1u][lane] = o[2];
      const uint32_t j = 2u * (rp & 3u);
      dp |= (below(o[3].x, o[3].y, cp) >> j) | (below(o[3].z, o[3].w, cp) >> (j + 1u));
      dq |= (below(o[3].x, o[3].y, cq) >> j) | (below(o[3].z, o[3].w, cq) >> (j + 1u));
      if ((rp & 3u) == 3u) {
        B.deep[rp >> 2][lane] = make_uint2(dp, dq);
        dp = dq = 0u;
      }
    }
  } else {
    const uint32_t n = (kRounds / 2) / parts;
#pragma unroll 1
    for (uint32_t rp = part * n; rp < part * n + n; rp += 4u) {
      const uint32_t c0 = (kTagPos << 28) | (lane << 3) | rp;
      const uint32_t c[4] = {c0, c0 + 1u, c0 + 2u, c0 + 3u};
      philox4(c, tid, s, P.sample, P.k0, P.k1, o);
#pragma unroll
      for (uint32_t i = 0; i < 4u; ++i) B.pos[rp + i][lane] = o[i];
    }
  }
}

// The 16 single-hit rounds of the tile in m from its drawn numbers. The
// offsets and numbers of a round are loaded one round ahead, so its chain is
// quadrant in, logic, quadrant out.
template <bool kGeneral, int kPar, bool kTrack>
__device__ __forceinline__ int rounds_from(TileMem& m, const QuadTab& tab, const SweepParams& P, uint32_t tid, uint32_t s,
                                           const tilemem::Origin& og, const TileRand<kGeneral>& B, uint32_t lane) {
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(&m) + lane * 8u;
  const uint32_t one = *(const volatile uint32_t*)&tab.one, neg = *(const volatile uint32_t*)&tab.neg;
  int dh = 0;
  const tilemem::Rates<true> R(P, kPar != 0);
  auto one_round = [&](const uint4& ofs, const uint4& sh, uint32_t X, uint32_t Y, uint32_t r, const uint4& A,
                       uint32_t Wp, uint32_t Wq) {
    if constexpr (kGeneral)
      tilemem::round_general<kTrack>(base, ofs, sh, one, X, Y, kPar != 0, og, dh, [&](uint32_t same, uint32_t any) {
        return tilemem::accept_cells<true>(P, R, tid, s, A, kPar ? Wq : Wp, kPar ? Wp : Wq, lane, r, same, any, one, neg);
      });
    else
      tilemem::round_p1<kPar, kTrack>(base, ofs, sh, one, X, Y, og, dh);
  };
  uint4 at0 = B.at[0], sh0 = B.sh[0], pos = B.pos[0][lane];
  uint4 A0 = B.acc[0][kGeneral ? lane : 0u];
  uint2 W = B.deep[0][kGeneral ? lane : 0u];   // outcomes of the next eight rounds, shifted round by round
#pragma unroll 1
  for (uint32_t rp = 0; rp < kRounds / 2; ++rp) {
    const uint32_t nx = (rp + 1u) & 7u;
    const uint4 at1 = B.at[2u * rp + 1u], sh1 = B.sh[2u * rp + 1u];
    uint4 A1 = A0;
    if constexpr (kGeneral) {
      A1 = B.acc[2u * rp + 1u][lane];
      if (rp == 4u) W = B.deep[1][lane];
    }
    one_round(at0, sh0, pos.x, pos.y, 2u * rp, A0, W.x, W.y);
    at0 = B.at[2u * nx];
    sh0 = B.sh[2u * nx];
    const uint4 pn = B.pos[nx][lane];
    if constexpr (kGeneral) A0 = B.acc[2u * nx][lane];
    one_round(at1, sh1, pos.z, pos.w, 2u * rp + 1u, A1, W.x << 1, W.y << 1);
    pos = pn;
    W.x <<= 2;
    W.y <<= 2;
  }
  return dh;
}

// Lattice words in HBM / L2: other SMs change them between steps, so reads
// bypass L1.
struct GlobalLat {
  uint32_t* p;
  __device__ __forceinline__ uint32_t ld(uint32_t i) const { return __ldcg(p + i); }
  __device__ __forceinline__ void st(uint32_t i, uint32_t v) const { __stcg(p + i, v); }
};
// A tile's words and the sites around it.
struct Window {
  uint32_t T[4][4], hx[4], hy[4], left[4], up[4];
};

// Where a window's words are (word indices of a lattice in global memory, or
// shared addresses over a cluster): they depend on the origins alone, so they
// are worked out while the barrier before the step is pending. For plane row
// y, column x of the window: c the word its bits start in, n the next block
// column's, sh the bit they start at; h the row below (lane 31 needs it), u the
// row above (lane 0) and b3 the block column left of column 3's (kHalo = 2).
struct WinAddr {
  uint32_t c[4][4], n[4][4], h[4][2], u[4][2], b3[4], sh[4];
};

// The window whose site (0,0) is site (X0, Y0) of the frame the lattice is
// held in (geometry as in run::sweep_run, kpz_run.cuh). kHalo: 0 the tile
// alone, 1 with the column right of it (hx) and the row below it (hy), 2 also
// the column left of it and the row above.
template <int kHalo>
__device__ __forceinline__ void window_at(const Geometry& g, uint32_t lane, uint32_t X0, uint32_t Y0, WinAddr& w) {
  const uint32_t NR = g.NR, NB = g.NB;
  X0 &= g.L - 1u;
  Y0 &= g.L - 1u;
  const uint32_t by = Y0 & 3u, Rb = Y0 >> 2, bx = X0 & 3u, a = X0 >> 2;
  uint32_t offY[4];
#pragma unroll
  for (uint32_t yq = 0; yq < 4; ++yq)
    offY[yq] = ((by + yq) & 3u) * 4u * NR + ((Rb + lane + ((by + yq) >> 2)) & (NR - 1u));
  const uint32_t offH = by * 4u * NR + ((Rb + 32u) & (NR - 1u));                                   // row below
  const uint32_t offU = ((by + 3u) & 3u) * 4u * NR + ((Rb - 1u + ((by + 3u) >> 2)) & (NR - 1u));   // row above
#pragma unroll
  for (uint32_t xq = 0; xq < 4; ++xq) {
    const uint32_t st = (a + ((bx + xq) >> 2)) & (g.L / 4u - 1u), kx = st >> 5, offX = ((bx + xq) & 3u) * NR;
    const uint32_t w0 = kx * kPlanes * NR + offX, w1 = ((kx + 1u) & (NB - 1u)) * kPlanes * NR + offX;
    w.sh[xq] = st & 31u;
#pragma unroll
    for (uint32_t yq = 0; yq < 4; ++yq) {
      w.c[yq][xq] = w0 + offY[yq];
      w.n[yq][xq] = w1 + offY[yq];
      if (kHalo == 2 && xq == 3) w.b3[yq] = ((kx + NB - 1u) & (NB - 1u)) * kPlanes * NR + offX + offY[yq];
    }
    if (kHalo >= 1) { w.h[xq][0] = w0 + offH; w.h[xq][1] = w1 + offH; }
    if (kHalo == 2) { w.u[xq][0] = w0 + offU; w.u[xq][1] = w1 + offU; }
  }
}

template <int kHalo, class Load>
__device__ __forceinline__ void fetch_window(const WinAddr& a, Load ld, Window& w) {
  uint32_t C[4][4], N[4][4], H[4][2], U[4][2], B3[4];
#pragma unroll
  for (uint32_t xq = 0; xq < 4; ++xq) {
#pragma unroll
    for (uint32_t yq = 0; yq < 4; ++yq) {
      C[yq][xq] = ld(a.c[yq][xq]);
      N[yq][xq] = ld(a.n[yq][xq]);
      if (kHalo == 2 && xq == 3) B3[yq] = ld(a.b3[yq]);
    }
    if (kHalo >= 1) { H[xq][0] = ld(a.h[xq][0]); H[xq][1] = ld(a.h[xq][1]); }
    if (kHalo == 2) { U[xq][0] = ld(a.u[xq][0]); U[xq][1] = ld(a.u[xq][1]); }
  }
#pragma unroll
  for (uint32_t xq = 0; xq < 4; ++xq) {
#pragma unroll
    for (uint32_t yq = 0; yq < 4; ++yq) {
      w.T[yq][xq] = __funnelshift_r(C[yq][xq], N[yq][xq], a.sh[xq]);
      if (kHalo >= 1 && xq == 0) w.hx[yq] = (N[yq][0] >> a.sh[0]) & 1u;
      if (kHalo == 2 && xq == 3) w.left[yq] = ((a.sh[3] ? C[yq][3] : B3[yq]) >> ((a.sh[3] + 31u) & 31u)) & 1u;
    }
    if (kHalo >= 1) w.hy[xq] = __funnelshift_r(H[xq][0], H[xq][1], a.sh[xq]);
    if (kHalo == 2) w.up[xq] = __funnelshift_r(U[xq][0], U[xq][1], a.sh[xq]);
  }
}

// Tile (tx, ty) of the frame the lattice is held in, with all sites around it.
__device__ __forceinline__ void load_tile(const Geometry& g, const GlobalLat lat, uint32_t lane, uint32_t tx, uint32_t ty,
                                          Window& w) {
  const uint32_t NR = g.NR, NB = g.NB, R = ty * 32u + lane;
  const uint32_t Ru = (ty * 32u + NR - 1u) & (NR - 1u), Rd = (ty * 32u + 32u) & (NR - 1u);
  const uint32_t o = tx * kPlanes * NR, ol = ((tx + NB - 1u) & (NB - 1u)) * kPlanes * NR,
                 orr = ((tx + 1u) & (NB - 1u)) * kPlanes * NR;
#pragma unroll
  for (uint32_t y = 0; y < 4; ++y) {
#pragma unroll
    for (uint32_t x = 0; x < 4; ++x) w.T[y][x] = lat.ld(o + plane(y, x) * NR + R);
    w.left[y] = lat.ld(ol + plane(y, 3) * NR + R) >> 31;
    w.hx[y] = lat.ld(orr + plane(y, 0) * NR + R) & 1u;
  }
#pragma unroll
  for (uint32_t x = 0; x < 4; ++x) {
    w.hy[x] = lat.ld(o + plane(0, x) * NR + Rd);
    w.up[x] = lat.ld(o + plane(3, x) * NR + Ru);
  }
}

__device__ __forceinline__ void store_tile(const Geometry& g, const GlobalLat lat, uint32_t lane, uint32_t tx, uint32_t ty,
                                           const uint32_t (&T)[4][4]) {
  const uint32_t o = tx * kPlanes * g.NR + ty * 32u + lane;
#pragma unroll
  for (uint32_t y = 0; y < 4; ++y)
#pragma unroll
    for (uint32_t x = 0; x < 4; ++x) lat.st(o + plane(y, x) * g.NR, T[y][x]);
}

// The rounds of tile (tx, ty) of the sweep with origin (ox, oy); w.T holds the
// tile before and after. kLive: every site of the tile is live, its neighbours
// are idle (kpz_tileset.cu); otherwise its low row and column are dead.
template <bool kGeneral, bool kLive>
__device__ __forceinline__ void tile_rounds(const SweepParams& P, Window& w, TileMem& m, const QuadTab& tab,
                                            const TileRand<kGeneral>& B, uint32_t lane, uint32_t s, uint32_t ox,
                                            uint32_t oy, uint32_t tx, uint32_t ty) {
  const uint32_t L = P.g.L;
  const uint32_t Y0 = (oy + ty * kTile) & (L - 1u), X0 = (ox + tx * kTile) & (L - 1u);
  const uint32_t tid = ty * P.ntx + tx;
  const uint32_t uo = (0u - X0) & (L - 1u), vo = (0u - Y0) & (L - 1u);
  const bool track = (uo < kTile) && (vo < kTile), odd = (X0 + Y0 + P.g.par) & 1u;
  const tilemem::Origin og(lane, uo, vo);
  tilemem::put_tile<kLive>(m, lane, w.T, w.hx, w.hy, w.left, w.up);
  __syncwarp();
  int dh;
  if (track) dh = odd ? rounds_from<kGeneral, 1, true>(m, tab, P, tid, s, og, B, lane)
                      : rounds_from<kGeneral, 0, true>(m, tab, P, tid, s, og, B, lane);
  else       dh = odd ? rounds_from<kGeneral, 1, false>(m, tab, P, tid, s, og, B, lane)
                      : rounds_from<kGeneral, 0, false>(m, tab, P, tid, s, og, B, lane);
  if (track && dh != 0) atomicAdd(P.h00, (unsigned long long)(long long)dh);
  tilemem::get_tile(m, lane, w.T);
}

// Set swept in phase `phase` of sweep s (the shuffle of kpz_tileset.cu).
__device__ __forceinline__ uint32_t phase_set(const SweepParams& P, uint32_t s, uint32_t phase) {
  const uint4 w = philox(kTagPhase << 28, 0u, s, P.sample, P.k0, P.k1);
  uint32_t perm[4] = {0u, 1u, 2u, 3u};
  const uint32_t r[3] = {w.x, w.y, w.z};
#pragma unroll
  for (uint32_t i = 3; i >= 1; --i) {
    const uint32_t j = r[3 - i] % (i + 1u);
    const uint32_t t = perm[i];
    perm[i] = j == 0u ? perm[0] : j == 1u ? perm[1] : j == 2u ? perm[2] : t;
    if (j == 0u) perm[0] = t; else if (j == 1u) perm[1] = t; else if (j == 2u) perm[2] = t;
  }
  return phase == 0u ? perm[0] : phase == 1u ? perm[1] : phase == 2u ? perm[2] : perm[3];
}

// A step of a tile warp: sweep, set (kSets) and tile.
struct Step {
  uint32_t s, q, tx, ty;
};

// bar.* and barrier.cluster.*.aligned are only defined for a warp whose lanes
// arrive together; divergent code comes before most of them (the atomic add of
// the tile that holds site (0,0), a lane that draws origins), so the lanes are
// brought together here.
__device__ __forceinline__ void bar_sync(uint32_t id, uint32_t n) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t id, uint32_t n) {
  __syncwarp();
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Grid version. A step is a sweep, or one tile set of a sweep (kSets); every
// tile of a step has a tile warp of its own. Warps of a block: wpc tile warps,
// makers * wpc drawing warps (they draw the next step's numbers into the other
// of two buffers while this step runs; with makers = 0 the tile warps draw
// their own numbers while the barrier is pending) and one barrier warp, which
// collects the block (named barrier 1), reports the step to the grid, waits
// for all blocks (bounded in time) and releases the block (named barrier 2).
// A last step brings the lattice back to the fixed frame.
template <bool kGeneral, bool kSets>
__global__ void __launch_bounds__(320, 1) resident_grid_kernel(const SweepParams P, uint32_t n, uint32_t tiles,
                                                               uint32_t wpc, uint32_t makers, uint32_t* scratch,
                                                               GridSync* sync) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TileRand<kGeneral>* rnd = reinterpret_cast<TileRand<kGeneral>*>(smem_raw);   // [1 or 2][wpc]
  TileMem* mem = reinterpret_cast<TileMem*>(rnd + (makers ? 2u : 1u) * wpc);   // [wpc]
  __shared__ QuadTab tab;
  __shared__ uint32_t stop;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const uint32_t nsteps = n * (kSets ? 4u : 1u);   // without the last one
  if (threadIdx.x == 0) stop = 0u;
  if (threadIdx.x < 4u) tilemem::fill_quad_tab(tab, threadIdx.x);
  __syncthreads();
  if (warp == nwarps - 1u) {   // barrier warp
    for (uint32_t k = 1; k <= nsteps; ++k) {
      bar_sync(1, blockDim.x);
      if (lane == 0) {
        gridsync::red_release(&sync->arrived);
        if (!gridsync::wait_for(sync, k * gridDim.x)) stop = 1u;
      }
      __syncwarp();
      bar_sync(2, blockDim.x);
      if (*(volatile uint32_t*)&stop) return;
    }
    bar_sync(1, blockDim.x);
    // The last block out resets the counters and advances the sweep count.
    if (lane == 0) {
      __threadfence();
      if (gridsync::add_acq_rel(&sync->finished, 1u) == gridDim.x - 1u) {
        sync->arrived = 0u;
        sync->finished = 0u;
        *const_cast<uint64_t*>(P.t_dev) += n;
      }
    }
    return;
  }
  const uint32_t t0 = (uint32_t)(*(const volatile uint64_t*)P.t_dev) + P.s_add;
  const bool maker = warp >= wpc;
  const uint32_t slot = maker ? (warp - wpc) % wpc : warp, part = maker ? (warp - wpc) / wpc : 0u;
  const uint32_t c = blockIdx.x * wpc + slot;    // this warp's tile of every step
  const uint32_t across = kSets ? P.ntx / 2u : P.ntx, cy = c / across, cx = c - cy * across;
  const bool live = c < tiles;
  const uint32_t L = P.g.L, words = L * L / 32u;
  Step st;
  // Sweep and tile of step k.
  auto place = [&](uint32_t k) {
    st.s = t0 + (kSets ? k >> 2 : k);
    st.q = kSets ? phase_set(P, st.s, k & 3u) : 0u;
    st.tx = kSets ? 2u * cx + (st.q & 1u) : cx;
    st.ty = kSets ? 2u * cy + (st.q >> 1) : cy;
  };
  if (maker) {
    place(0u);
    if (live) draw_tile<kGeneral>(P, tab, rnd[slot], st.ty * P.ntx + st.tx, st.s, lane, part, makers);
    bar_sync(3, blockDim.x - 32u);
    for (uint32_t k = 0; k <= nsteps; ++k) {
      if (k != 0u) {
        bar_sync(2, blockDim.x);
        if (*(volatile uint32_t*)&stop) return;
      }
      if (k + 1u < nsteps && live) {
        place(k + 1u);
        draw_tile<kGeneral>(P, tab, rnd[((k + 1u) & 1u) * wpc + slot], st.ty * P.ntx + st.tx, st.s, lane, part, makers);
      }
      bar_arrive(1, blockDim.x);
    }
    return;
  }
  // The window's addresses ahead of the barrier: L = 2048, p = 1 2.96 us a sweep
  // against 3.05; general rates gain nothing (L = 4096 7.97 against 7.89).
  constexpr bool kEarly = !kSets && !kGeneral;
  WinAddr at;
  uint32_t ox = 0u, oy = 0u, rx = 0u, ry = 0u;   // origin; its offset in the frame before
  // All that can be known of step k before the barrier in front of it.
  auto plan = [&](uint32_t k) {
    const bool back = k == nsteps;               // the fixed frame again
    place(k);
    if (!kSets || (k & 3u) == 0u) {
      const uint32_t* o = rnd[(makers ? ((k - 1u) & 1u) * wpc : 0u) + slot].origin;
      const uint2 next = back ? make_uint2(0u, 0u) : k == 0u ? origin_of(P, t0) : make_uint2(o[0], o[1]);
      rx = next.x - ox;
      ry = next.y - oy;
      ox = next.x;
      oy = next.y;
    }
    if (!makers) {
      __syncwarp();
      if (live && !back) draw_tile<kGeneral>(P, tab, rnd[slot], st.ty * P.ntx + st.tx, st.s, lane, 0u, 1u);
      __syncwarp();
    }
    if constexpr (kEarly) window_at<1>(P.g, lane, rx + st.tx * kTile, ry + st.ty * kTile, at);
  };
  if (makers) bar_sync(3, blockDim.x - 32u);
  plan(0u);
  for (uint32_t k = 0; k <= nsteps; ++k) {
    const uint32_t sw = kSets ? k >> 2 : k;      // sweeps before this step
    const bool back = k == nsteps;
    const TileRand<kGeneral>& B = rnd[(makers ? (k & 1u) * wpc : 0u) + slot];
    if (k != 0u) {
      bar_sync(2, blockDim.x);
      if (*(volatile uint32_t*)&stop) return;
    }
    const GlobalLat from{sw == 0u ? P.lat : scratch + ((sw - 1u) & 1u) * words};
    const GlobalLat to{back ? P.lat : scratch + (sw & 1u) * words};
    auto ld = [&](uint32_t i) { return from.ld(i); };
    if (live) {
      Window w;
      if (kSets && (back || (k & 3u) == 0u)) {   // the four tiles of this warp change frames
#pragma unroll 1
        for (uint32_t q = 0; q < 4u; ++q) {
          if (!back && q == st.q) continue;
          const uint32_t qx = 2u * cx + (q & 1u), qy = 2u * cy + (q >> 1);
          WinAddr aq;
          window_at<0>(P.g, lane, rx + qx * kTile, ry + qy * kTile, aq);
          fetch_window<0>(aq, ld, w);
          store_tile(P.g, to, lane, qx, qy, w.T);
        }
      }
      if (!(kSets && back)) {
        if constexpr (!kSets) {
          if constexpr (!kEarly) window_at<1>(P.g, lane, rx + st.tx * kTile, ry + st.ty * kTile, at);
          fetch_window<1>(at, ld, w);
        } else if ((k & 3u) == 0u) {
          window_at<2>(P.g, lane, rx + st.tx * kTile, ry + st.ty * kTile, at);
          fetch_window<2>(at, ld, w);
        } else {
          load_tile(P.g, to, lane, st.tx, st.ty, w);
        }
        if (!back) tile_rounds<kGeneral, kSets>(P, w, mem[slot], tab, B, lane, st.s, ox, oy, st.tx, st.ty);
        store_tile(P.g, to, lane, st.tx, st.ty, w.T);
      }
    }
    bar_arrive(1, blockDim.x);
    if (k < nsteps) plan(k + 1u);
  }
}

// Cluster version (up to 64 tiles at a time): one cluster of 1 to 16 blocks
// holds the whole lattice in its shared memory, two frames of it by turns;
// windows are read over distributed shared memory and the hardware's cluster
// barrier ends a step; between arriving and waiting the tile warps work out the
// next window's addresses (L = 512, p = 1: 2.18 -> 1.95 us a sweep; an mbarrier
// in each block, raised by every tile warp of the cluster, took 2.06). Warps of a block: a tile warp for each of its units,
// `makers` drawing warps for each.
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t map_to(uint32_t addr, uint32_t cta) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(cta));
  return r;
}
__device__ __forceinline__ uint32_t ld_cluster(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync() {
  cluster_arrive();
  cluster_wait();
}

// The lattice over the cluster: a block's frame holds 1 << lg units of one
// tile, or (kSets) of 2 x 2 tiles, one of each set, each tile as [16 planes][32
// cell rows] words.
template <bool kSets>
struct ClusterLat {
  uint32_t frame;   // shared address of the frame in every block
  uint32_t lg, NR, NB, ntx;
  // Address of plane 0 of block column K at cell row R (both wrapped).
  __device__ __forceinline__ uint32_t at(uint32_t K, uint32_t R) const {
    K &= NB - 1u;
    R &= NR - 1u;
    const uint32_t ty = R >> 5;
    const uint32_t unit = kSets ? (ty >> 1) * (ntx >> 1) + (K >> 1) : ty * ntx + K;
    const uint32_t q = kSets ? (K & 1u) + 2u * (ty & 1u) : 0u;
    const uint32_t slot = (unit & ((1u << lg) - 1u)) * (kSets ? 4u : 1u) + q;
    return map_to(frame + slot * (kPlanes * 128u) + (R & 31u) * 4u, unit >> lg);
  }
};

// window_at over the cluster.
template <int kHalo, bool kSets>
__device__ __forceinline__ void window_at_cluster(const ClusterLat<kSets>& lat, uint32_t lane, uint32_t X0, uint32_t Y0,
                                                  WinAddr& w) {
  const uint32_t L = lat.NR * 4u;
  X0 &= L - 1u;
  Y0 &= L - 1u;
  const uint32_t by = Y0 & 3u, Rb = Y0 >> 2, bx = X0 & 3u, a = X0 >> 2, K = a >> 5;
  // Plane 0 of block columns K, K + 1, K + 2 at cell rows Rb + lane, Rb + lane
  // + 1, of the row below the tile and the one above.
  uint32_t at[4][3];
#pragma unroll
  for (uint32_t i = 0; i < (kHalo == 2 ? 4u : kHalo ? 3u : 2u); ++i) {
    const uint32_t R = i == 3u ? Rb - 1u + ((by + 3u) >> 2) : Rb + (i == 2u ? 32u : lane + i);
#pragma unroll
    for (uint32_t j = 0; j < 3u; ++j) at[i][j] = lat.at(K + j, R);
  }
#pragma unroll
  for (uint32_t xq = 0; xq < 4; ++xq) {
    const uint32_t st = a + ((bx + xq) >> 2), x4 = (bx + xq) & 3u;
    w.sh[xq] = st & 31u;
    const bool next = (st >> 5) != K;   // carried into the next block column
#pragma unroll
    for (uint32_t yq = 0; yq < 4; ++yq) {
      const uint32_t p = plane((by + yq) & 3u, x4) * 128u;
      const bool wrap = by + yq >= 4u;
      w.c[yq][xq] = (wrap ? (next ? at[1][1] : at[1][0]) : (next ? at[0][1] : at[0][0])) + p;
      w.n[yq][xq] = (wrap ? (next ? at[1][2] : at[1][1]) : (next ? at[0][2] : at[0][1])) + p;
      if (kHalo == 2 && xq == 3) w.b3[yq] = lat.at((st >> 5) - 1u, Rb + lane + (wrap ? 1u : 0u)) + p;
    }
    if (kHalo) {
      const uint32_t p = plane(by, x4) * 128u;
      w.h[xq][0] = (next ? at[2][1] : at[2][0]) + p;
      w.h[xq][1] = (next ? at[2][2] : at[2][1]) + p;
    }
    if (kHalo == 2) {
      const uint32_t p = plane((by + 3u) & 3u, x4) * 128u;
      w.u[xq][0] = (next ? at[3][1] : at[3][0]) + p;
      w.u[xq][1] = (next ? at[3][2] : at[3][1]) + p;
    }
  }
}

// load_tile over the cluster; own: this lane's words of the tile, 32 apart.
__device__ __forceinline__ void load_tile_cluster(const ClusterLat<true>& lat, uint32_t lane, uint32_t tx, uint32_t ty,
                                                  const uint32_t* own, Window& w) {
  const uint32_t R = ty * 32u + lane;
  const uint32_t l = lat.at(tx - 1u, R), r = lat.at(tx + 1u, R);
  const uint32_t u = lat.at(tx, ty * 32u - 1u), d = lat.at(tx, ty * 32u + 32u);
#pragma unroll
  for (uint32_t y = 0; y < 4; ++y) {
    w.left[y] = ld_cluster(l + plane(y, 3) * 128u) >> 31;
    w.hx[y] = ld_cluster(r + plane(y, 0) * 128u) & 1u;
  }
#pragma unroll
  for (uint32_t x = 0; x < 4; ++x) {
    w.hy[x] = ld_cluster(d + plane(0, x) * 128u);
    w.up[x] = ld_cluster(u + plane(3, x) * 128u);
  }
#pragma unroll
  for (uint32_t p = 0; p < kPlanes; ++p) w.T[p >> 2][p & 3u] = own[p * 32u];
}

template <bool kGeneral, bool kSets>
__global__ void __launch_bounds__(384, 1) resident_cluster_kernel(const SweepParams P, uint32_t n, uint32_t lg,
                                                                  uint32_t makers) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr uint32_t kTiles = kSets ? 4u : 1u, kTileWords = kPlanes * 32u;   // tiles of a unit
  const uint32_t units = 1u << lg;
  TileRand<kGeneral>* rnd = reinterpret_cast<TileRand<kGeneral>*>(smem_raw);   // [2][units]
  TileMem* mem = reinterpret_cast<TileMem*>(rnd + 2u * units);                 // [units]
  uint32_t* frame = reinterpret_cast<uint32_t*>(mem + units);                  // [2][units][tiles][16][32]
  __shared__ QuadTab tab;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t t0 = (uint32_t)(*(const volatile uint64_t*)P.t_dev) + P.s_add;
  if (threadIdx.x < 4u) tilemem::fill_quad_tab(tab, threadIdx.x);
  const bool maker = warp >= units;
  const uint32_t slot = maker ? (warp - units) & (units - 1u) : warp, part = maker ? (warp - units) >> lg : 0u;
  const uint32_t unit = blockIdx.x * units + slot, across = P.ntx / (kSets ? 2u : 1u);
  const uint32_t uy = unit / across, ux = unit - uy * across;
  __syncthreads();
  uint32_t* own = frame + slot * kTiles * kTileWords + lane;   // this lane's words, 32 apart; + the frame's and the tile's offset
  const uint32_t half = units * kTiles * kTileWords;           // words of one frame in this block
  const uint32_t nsteps = n * kTiles;
  Step st;
  auto place = [&](uint32_t k) {
    st.s = t0 + k / kTiles;
    st.q = kSets ? phase_set(P, st.s, k & 3u) : 0u;
    st.tx = kSets ? 2u * ux + (st.q & 1u) : ux;
    st.ty = kSets ? 2u * uy + (st.q >> 1) : uy;
  };
  if (maker) {
    place(0u);
    draw_tile<kGeneral>(P, tab, rnd[slot], st.ty * P.ntx + st.tx, st.s, lane, part, makers);
    cluster_sync();
    for (uint32_t k = 0; k < nsteps; ++k) {
      if (k + 1u < nsteps) {
        place(k + 1u);
        draw_tile<kGeneral>(P, tab, rnd[((k + 1u) & 1u) * units + slot], st.ty * P.ntx + st.tx, st.s, lane, part, makers);
      }
      cluster_sync();
    }
    cluster_sync();
    return;
  }
#pragma unroll 1
  for (uint32_t i = 0; i < kTiles; ++i) {
    const uint32_t x = kSets ? 2u * ux + (i & 1u) : ux, y = kSets ? 2u * uy + (i >> 1) : uy;
    const uint32_t o = x * kPlanes * P.g.NR + y * 32u + lane;
#pragma unroll
    for (uint32_t p = 0; p < kPlanes; ++p) own[i * kTileWords + p * 32u] = __ldcg(P.lat + o + p * P.g.NR);
  }
  Window w;
  WinAddr at;
  uint32_t ox = 0u, oy = 0u, rx = 0u, ry = 0u;   // origin; its offset in the frame before
  auto lattice = [&](uint32_t sweep) {   // as it stands after `sweep` sweeps of this launch
    return ClusterLat<kSets>{smem_u32(frame + (sweep & 1u) * half), lg, P.g.NR, P.g.NB, P.ntx};
  };
  auto put = [&](uint32_t* to) {
#pragma unroll
    for (uint32_t p = 0; p < kPlanes; ++p) to[p * 32u] = w.T[p >> 2][p & 3u];
  };
  // All that can be known of step k before the barrier in front of it; next:
  // the origin of its sweep.
  auto plan = [&](uint32_t k, const uint2 next) {
    place(k);
    if (!kSets || (k & 3u) == 0u) {
      rx = next.x - ox;
      ry = next.y - oy;
      ox = next.x;
      oy = next.y;
      if constexpr (!kSets) window_at_cluster<1>(lattice(k), lane, rx + st.tx * kTile, ry + st.ty * kTile, at);
    }
  };
  auto ld = [](uint32_t a) { return ld_cluster(a); };
  cluster_sync();
  plan(0u, origin_of(P, t0));
  for (uint32_t k = 0; k < nsteps; ++k) {
    const uint32_t sw = k / kTiles;
    const TileRand<kGeneral>& B = rnd[(k & 1u) * units + slot];
    uint32_t* to = own + ((sw + 1u) & 1u) * half;
    if (!kSets || (k & 3u) == 0u) {   // the sweep's first step: the frame changes
      if (kSets) {
#pragma unroll 1
        for (uint32_t i = 0; i < 4u; ++i) {
          if (i == st.q) continue;
          WinAddr aq;
          window_at_cluster<0>(lattice(sw), lane, rx + (2u * ux + (i & 1u)) * kTile, ry + (2u * uy + (i >> 1)) * kTile, aq);
          fetch_window<0>(aq, ld, w);
          put(to + i * kTileWords);
        }
      }
      if (kSets) window_at_cluster<2>(lattice(sw), lane, rx + st.tx * kTile, ry + st.ty * kTile, at);
      fetch_window<kSets ? 2 : 1>(at, ld, w);
    } else if constexpr (kSets) {
      load_tile_cluster(lattice(sw + 1u), lane, st.tx, st.ty, to + st.q * kTileWords, w);
    }
    tile_rounds<kGeneral, kSets>(P, w, mem[slot], tab, B, lane, st.s, ox, oy, st.tx, st.ty);
    put(to + st.q * kTileWords);
    // Once every warp has arrived, the drawing warp may go on to overwrite this
    // step's numbers, so the origin they hold is read before.
    const uint2 next = make_uint2(B.origin[0], B.origin[1]);
    cluster_arrive();
    if (k + 1u < nsteps) plan(k + 1u, next);
    cluster_wait();
  }
#pragma unroll 1
  for (uint32_t i = 0; i < kTiles; ++i) {   // the fixed frame again
    const uint32_t x = kSets ? 2u * ux + (i & 1u) : ux, y = kSets ? 2u * uy + (i >> 1) : uy;
    window_at_cluster<0>(lattice(n), lane, x * kTile - ox, y * kTile - oy, at);
    fetch_window<0>(at, ld, w);
    store_tile(P.g, GlobalLat{P.lat}, lane, x, y, w.T);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *const_cast<uint64_t*>(P.t_dev) += n;
  cluster_sync();   // no block leaves while its shared memory is read
}

struct Shape {
  bool cluster;             // cluster version
  uint32_t wpc, grid;       // tile warps per block, blocks
  uint32_t tiles, makers;   // tiles per step, drawing warps per tile
  size_t smem;
};

constexpr uint32_t kSms = 152;   // GB300; where fewer are to be had, fits() says no

// How a lattice is laid over the chip (wpc = 0: not served). p = 1 draws 8
// blocks a tile and sweep, general rates 32; one warp draws a block in about
// 120 cycles, an SM's quarter in 80 (the wide multiplies), so drawing warps
// pay while an SM has at most two tiles; with seven or eight they take the issue slots
// the tile warps need (L = 4096 at p = 0.95: 9.0 us a sweep with them, 7.9
// without). The cluster has 16 SMs: at p = 1 it serves four tiles each (L =
// 1024 2.7 us a sweep, 2.9 on a grid; tile sets at L = 2048 11.6, 13.4), at
// general rates one (L = 512 3.15, on a grid 4.2; L = 1024 4.5 against 4.3; tile
// sets at L = 1024 13.5 against 18.1, at L = 2048 20.2 against 18.6). Beyond 1024
// tiles an SM would have more than two tiles a scheduler, and work, not
// latency, is the bound. 1024 tiles go to 147 blocks of seven tile warps: with
// eight on 128 of the 152 SMs L = 4096 took 3.94 us a sweep at p = 1 against 3.73
// (the tiles of an SM share its LSU), tile sets at L = 8192 17.8 against 17.0.
Shape shape_of(const SweepParams& P, bool tilesets, bool general, bool cluster) {
  Shape h{};
  const size_t rnd = general ? sizeof(TileRand<true>) : sizeof(TileRand<false>);
  const uint32_t all = P.ntx * P.nty;
  if (cluster) {
    h.tiles = tilesets ? all / 4u : all;
    if (h.tiles > (general ? 16u : 64u)) return Shape{};
    h.cluster = true;
    h.grid = std::min(h.tiles, 16u);
    h.wpc = h.tiles / h.grid;
    h.makers = general ? 2u : 1u;
    h.smem = h.wpc * (2u * rnd + sizeof(TileMem) + (tilesets ? 8u : 2u) * kPlanes * 32u * sizeof(uint32_t));
    return h;
  }
  h.tiles = tilesets ? all / 4u : all;
  if (h.tiles > 1024u) return h;
  h.wpc = std::max(1u, (h.tiles + kSms - 1u) / kSms);   // blocks of 1 to 7 tile warps, one on an SM
  h.grid = (h.tiles + h.wpc - 1u) / h.wpc;
  h.makers = h.wpc > 2u ? 0u : (general ? 2u : 1u);
  h.smem = h.wpc * ((h.makers ? 2u : 1u) * rnd + sizeof(TileMem));
  return h;
}

const void* kernel_of(const Shape& h, bool tilesets, bool general) {
  if (h.cluster && tilesets)
    return general ? (const void*)resident_cluster_kernel<true, true> : (const void*)resident_cluster_kernel<false, true>;
  if (h.cluster)
    return general ? (const void*)resident_cluster_kernel<true, false>
                   : (const void*)resident_cluster_kernel<false, false>;
  if (tilesets)
    return general ? (const void*)resident_grid_kernel<true, true> : (const void*)resident_grid_kernel<false, true>;
  return general ? (const void*)resident_grid_kernel<true, false> : (const void*)resident_grid_kernel<false, false>;
}

uint32_t threads_of(const Shape& h) { return 32u * (h.wpc * (1u + h.makers) + (h.cluster ? 0u : 1u)); }

cudaLaunchConfig_t config_of(const Shape& h, cudaLaunchAttribute* attr, cudaStream_t st) {
  if (h.cluster) {
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = h.grid;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1u;
  } else {
    attr->id = cudaLaunchAttributeCooperative;
    attr->val.cooperative = 1;
  }
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(h.grid);
  c.blockDim = dim3(threads_of(h));
  c.dynamicSmemBytes = h.smem;
  c.stream = st;
  c.attrs = attr;
  c.numAttrs = 1;
  return c;
}

// Whether the current device holds all blocks of the kernel at once.
bool fits(const Shape& h, bool tilesets, bool general) {
  if (h.wpc == 0u) return false;
  int dev = 0, per_sm = 0, sms = 0, coop = 0, most = 0;
  const void* f = kernel_of(h, tilesets, general);
  cudaFuncAttributes fa{};
  // The kernel's limit is the device's, not this shape's: it stays for every
  // later launch, and lattices of other sizes share the kernel.
  bool ok = cudaGetDevice(&dev) == cudaSuccess && cudaFuncGetAttributes(&fa, f) == cudaSuccess &&
            cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
            (most -= (int)fa.sharedSizeBytes) >= (int)h.smem &&
            cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most) == cudaSuccess;
  if (ok && h.cluster) {
    if (h.grid > 8u) ok = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t c = config_of(h, &attr, nullptr);
    int clusters = 0;
    ok = ok && cudaOccupancyMaxActiveClusters(&clusters, f, &c) == cudaSuccess && clusters > 0;
  } else if (ok) {
    ok = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
         cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop &&
         cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, (int)threads_of(h), h.smem) == cudaSuccess &&
         (uint32_t)(per_sm * sms) >= h.grid;
  }
  if (!ok) cudaGetLastError();
  return ok;
}

bool is_general(const SweepParams& P) { return !(P.Tp == 65536u && P.Tq == 0u); }

}  // namespace

uint32_t resident_kind(const SweepParams& P, bool tilesets) {
  if (P.cell == 2u || P.nty * kTile != P.g.L) return 0u;
  const bool general = is_general(P);
  // The answer for a device, size and kernel is kept (the queries take 10 us).
  constexpr int kMaxDev = 64;
  static std::mutex mu;
  static uint8_t known[kMaxDev][32][2][2] = {};   // kind + 1
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0u;
  std::lock_guard<std::mutex> lock(mu);
  uint8_t other = 0u;
  uint8_t& k = dev < kMaxDev ? known[dev][__builtin_ctz(P.g.L)][tilesets][general] : other;
  if (k) return k - 1u;
  const uint32_t kind = fits(shape_of(P, tilesets, general, true), tilesets, general)    ? 2u
                        : fits(shape_of(P, tilesets, general, false), tilesets, general) ? 1u
                                                                                          : 0u;
  k = (uint8_t)(kind + 1u);
  return kind;
}

cudaError_t launch_resident(const SweepParams& P, bool tilesets, uint32_t kind, uint32_t n, uint32_t* scratch,
                            GridSync* sync, cudaStream_t st) {
  const bool general = is_general(P);
  const Shape h = shape_of(P, tilesets, general, kind == 2u);
  if (h.wpc == 0u) return cudaErrorInvalidValue;
  SweepParams Q = P;
  uint32_t nn = n, makers = h.makers, tiles = h.tiles, wpc = h.wpc, lg = 0u;
  while ((1u << lg) < h.wpc) ++lg;
  void* cluster_args[] = {&Q, &nn, &lg, &makers};
  void* grid_args[] = {&Q, &nn, &tiles, &wpc, &makers, &scratch, &sync};
  cudaLaunchAttribute attr;
  const cudaLaunchConfig_t c = config_of(h, &attr, st);
  const cudaError_t e =
      cudaLaunchKernelExC(&c, kernel_of(h, tilesets, general), h.cluster ? cluster_args : grid_args);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace kpz
