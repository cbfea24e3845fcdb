// kpz_observe.cu -- flat start, packed import/export, heights and exact W^2.
//
// Sec. 2.1 of arXiv:1204.5072: flat start with periodic boundaries, heights
// reconstructed from the slopes, squared interface width eq. (Wdef).
// The lattice holds one bit per site, b = (h >> 1) & 1 (kpz_common.cuh); the
// slopes follow from neighbouring bits and the site parity (i + j + par) & 1.
// Heights are built in the gauge h(0,0) = 0: first down column 0,
//   h(0,j) = sum_{k<j} sigma_y(0,k),
// then along each row, h(i,j) = h(0,j) + sum_{l<i} sigma_x(l,j); on a valid
// (curl-free) surface this equals any other path sum.
#include <algorithm>
#include <mutex>

#include "kpz_observe.h"
#include "kpz_w2.cuh"

namespace kpz {
namespace {

// Bit b of site (i, j) (i < L, j < L).
__device__ __forceinline__ uint32_t site_bit(const uint32_t* lat, const Geometry& g, uint32_t i,
                                             uint32_t j) {
  return (lat[g.word(i >> 7, plane(j & 3u, i & 3u), j >> 2)] >> ((i >> 2) & 31u)) & 1u;
}

// Flat start h = (i+j) & 1: h >> 1 = 0 everywhere.
__global__ void init_flat_kernel(uint4* lat4, size_t n4) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4;
       i += (size_t)gridDim.x * blockDim.x)
    lat4[i] = make_uint4(0u, 0u, 0u, 0u);
}

// Bits of 4 consecutive cells (starting at cell c0) of a plane, spread to
// positions 4*jc (jc = cell offset): the row-major order of sites 4jc + x4.
__device__ __forceinline__ uint32_t spread4(uint32_t n) {
  return (n & 1u) | ((n & 2u) << 3) | ((n & 4u) << 6) | ((n & 8u) << 9);
}

// Interleave: bit k of a -> bit 2k, for a < 2^16.
__device__ __forceinline__ uint32_t part1by1(uint32_t a) {
  a = (a | (a << 8)) & 0x00FF00FFu;
  a = (a | (a << 4)) & 0x0F0F0F0Fu;
  a = (a | (a << 2)) & 0x33333333u;
  a = (a | (a << 1)) & 0x55555555u;
  return a;
}

// Block columns of one import/export block: warp w of a block takes block
// columns [w KS, (w + 1) KS), KS = NB / min(kIoSegs, NB).
constexpr uint32_t kIoSegs = 16;

// Rows j = 4R + y4 of a band for 32 consecutive cell rows R (lane = R - R0)
// and one y4 (blockIdx.x = 4 group + y4): a warp's loads of one plane word are
// 128 contiguous bytes, and each lane writes its row's 8 packed words of a
// block column (32 contiguous bytes).
__global__ void __launch_bounds__(32 * kIoSegs) export_kernel(const uint32_t* __restrict__ lat, Geometry g,
                                                              uint32_t j0, uint32_t nrows,
                                                              uint32_t* __restrict__ packed) {
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
  const uint32_t S = min(kIoSegs, g.NB), KS = g.NB / S;
  const uint32_t y4 = blockIdx.x & 3u, rr = 32u * (blockIdx.x >> 2) + lane;
  if (w >= S || 4u * rr >= nrows) return;
  const uint32_t R = j0 / 4u + rr, j = 4u * R + y4;
  const uint32_t y4n = (y4 + 1u) & 3u, Rn = (y4 == 3u) ? ((R + 1u) & (g.NR - 1u)) : R;   // row j + 1
  // parity of site 16 wi + k is (k + j + par) & 1; a neighbour is higher iff
  // the bits differ by that parity, so sigma = +1 <=> b(next) ^ b ^ parity == 0
  const uint32_t odd = ((j + g.par) & 1u) ? 0x5555u : 0xAAAAu;
  uint4* out = reinterpret_cast<uint4*>(packed + (size_t)(4u * rr + y4) * (g.L / 16u));
  for (uint32_t K = w * KS; K < (w + 1u) * KS; ++K) {
    uint32_t A[4], B[4];
#pragma unroll
    for (uint32_t x4 = 0; x4 < 4; ++x4) {
      A[x4] = lat[g.word(K, plane(y4, x4), R)];
      B[x4] = lat[g.word(K, plane(y4n, x4), Rn)];
    }
    const uint32_t nxt = lat[g.word((K + 1u) & (g.NB - 1u), plane(y4, 0), R)] & 1u;   // site 128(K+1)
    uint32_t o[8];
#pragma unroll
    for (uint32_t q = 0; q < 8; ++q) {   // packed word q: sites 16q + k = cells 4q + k/4, x4 = k%4
      uint32_t r0 = 0, r1 = 0;
#pragma unroll
      for (uint32_t x4 = 0; x4 < 4; ++x4) {
        r0 |= spread4((A[x4] >> (4u * q)) & 0xFu) << x4;
        r1 |= spread4((B[x4] >> (4u * q)) & 0xFu) << x4;
      }
      r0 |= (q < 7u ? (A[0] >> (4u * q + 4u)) & 1u : nxt) << 16;
      const uint32_t sx = ~((r0 >> 1) ^ r0 ^ odd) & 0xFFFFu;
      const uint32_t sy = ~(r1 ^ r0 ^ odd) & 0xFFFFu;
      o[q] = part1by1(sx) | (part1by1(sy) << 1);
    }
    out[2u * K] = make_uint4(o[0], o[1], o[2], o[3]);
    out[2u * K + 1u] = make_uint4(o[4], o[5], o[6], o[7]);
  }
}

// Absolute heights modulo 4 down column 0 for rows [j0, j0 + nrows) of a
// packed band; hcar holds h(0, j0) mod 4 on entry and h(0, j0 + nrows) mod 4
// on exit. One block.
__global__ void import_col_kernel(const uint32_t* __restrict__ packed, Geometry g, uint32_t nrows,
                                  uint32_t* __restrict__ hcar, int32_t* __restrict__ hcol) {
  __shared__ int32_t part[1024];
  const uint32_t nt = blockDim.x, t = threadIdx.x, wpr = g.L / 16;
  const uint32_t chunk = (nrows + nt - 1) / nt;
  const uint32_t r0 = min(nrows, t * chunk), r1 = min(nrows, r0 + chunk);
  int32_t sum = 0;
  for (uint32_t r = r0; r < r1; ++r) sum += ((packed[(size_t)r * wpr] >> 1) & 1u) ? 1 : -1;
  part[t] = sum;
  __syncthreads();
  for (uint32_t off = 1; off < nt; off <<= 1) {
    const int32_t v = (t >= off) ? part[t - off] : 0;
    __syncthreads();
    part[t] += v;
    __syncthreads();
  }
  const int32_t base = (int32_t)*hcar;
  int32_t h = base + ((t == 0) ? 0 : part[t - 1]);
  for (uint32_t r = r0; r < r1; ++r) {
    hcol[r] = h & 3;
    h += ((packed[(size_t)r * wpr] >> 1) & 1u) ? 1 : -1;
  }
  __syncthreads();
  if (t == nt - 1) *hcar = (uint32_t)((base + part[nt - 1]) & 3);
}

// The 16 x-slopes of a packed word (its even bits) at bits 0..15.
__device__ __forceinline__ uint32_t even_bits(uint32_t a) {
  a &= 0x55555555u;
  a = (a | (a >> 1)) & 0x33333333u;
  a = (a | (a >> 2)) & 0x0F0F0F0Fu;
  a = (a | (a >> 4)) & 0x00FF00FFu;
  return (a | (a >> 8)) & 0x0000FFFFu;
}

// Bits 0, 4, 8, 12 of v at bits 0..3.
__device__ __forceinline__ uint32_t gather4(uint32_t v) {
  v &= 0x1111u;
  v = (v | (v >> 3)) & 0x0303u;
  return (v | (v >> 6)) & 0xFu;
}

// Bits of the rows of a packed band, laid out as in export_kernel. Along row
// j, h(i,j) = h(0,j) - i + 2 U(i,j) with U(i,j) the number of +1 x-slopes
// left of i, so b(i,j) = bit 1 of (h(0,j) - i) mod 4, XOR U(i,j) mod 2: a
// prefix XOR of the x-slope bits. Each warp first takes the parity of its
// block columns' x-slopes; the parities of the segments before it give its
// carry.
__global__ void __launch_bounds__(32 * kIoSegs) import_rows_kernel(uint32_t* __restrict__ lat, Geometry g,
                                                                   uint32_t j0, uint32_t nrows,
                                                                   const uint32_t* __restrict__ packed,
                                                                   const int32_t* __restrict__ hcol) {
  __shared__ uint32_t seg_par[kIoSegs][32];
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
  const uint32_t S = min(kIoSegs, g.NB), KS = g.NB / S;
  const uint32_t y4 = blockIdx.x & 3u, rr = 32u * (blockIdx.x >> 2) + lane;
  const bool live = w < S && 4u * rr < nrows;
  const uint32_t r = 4u * rr + y4;   // row within the band
  const uint4* row = reinterpret_cast<const uint4*>(packed + (size_t)(live ? r : 0u) * (g.L / 16u));
  uint32_t x = 0;
  if (live)
    for (uint32_t K = w * KS; K < (w + 1u) * KS; ++K) {
      const uint4 a = row[2u * K], b = row[2u * K + 1u];
      x ^= a.x ^ a.y ^ a.z ^ a.w ^ b.x ^ b.y ^ b.z ^ b.w;
    }
  seg_par[w][lane] = __popc(x & 0x55555555u) & 1u;
  __syncthreads();
  if (!live) return;
  uint32_t carry = 0;   // parity of the +1 x-slopes left of the segment
  for (uint32_t v = 0; v < w; ++v) carry ^= seg_par[v][lane];
  // bit 1 of (h(0,j) - k) mod 4 for k = 0..15 (period 4; 16 wi = 0 mod 4)
  const uint32_t pat = ((0x39C6u >> (4u * ((uint32_t)hcol[r] & 3u))) & 0xFu) * 0x1111u;
  const uint32_t R = j0 / 4u + rr;
  for (uint32_t K = w * KS; K < (w + 1u) * KS; ++K) {
    const uint4 a = row[2u * K], b = row[2u * K + 1u];
    const uint32_t pw[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    uint32_t W[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (uint32_t q = 0; q < 8; ++q) {   // sites 128K + 16q + k = cell 4q + k/4, x4 = k%4
      uint32_t e = even_bits(pw[q]);
      e ^= e << 1;
      e ^= e << 2;
      e ^= e << 4;
      e ^= e << 8;                       // bit k: parity of the x-slopes 0..k of the word
      const uint32_t bits = (((e << 1) ^ (0u - carry)) & 0xFFFFu) ^ pat;
      carry ^= (e >> 15) & 1u;
#pragma unroll
      for (uint32_t x4 = 0; x4 < 4; ++x4) W[x4] |= gather4(bits >> x4) << (4u * q);
    }
#pragma unroll
    for (uint32_t x4 = 0; x4 < 4; ++x4) lat[g.word(K, plane(y4, x4), R)] = W[x4];
  }
}

// h(0,j) for all rows j, gauge h(0,0) = 0: one block; thread t owns rows
// [t chunk, (t+1) chunk) in pieces of 32. A piece's 32 bits b(0, j) are loaded
// at once into a mask; its steps sigma_y(0, j) = +1 where b(0,j) ^ b(0,j+1)
// equals the parity of j + par, so the piece's height change is
// 2 popc(E) - 32; a block scan of the chunk sums gives each chunk's start.
constexpr uint32_t kCol0Threads = 1024;

__global__ void __launch_bounds__(kCol0Threads) col0_kernel(const uint32_t* __restrict__ lat, Geometry g,
                                                           int32_t* __restrict__ col0) {
  __shared__ int32_t part[kCol0Threads];
  const uint32_t nt = blockDim.x, t = threadIdx.x;
  const uint32_t chunk = g.L / nt;                 // multiple of 32
  const uint32_t j0 = t * chunk, pieces = chunk / 32u;
  const uint32_t parpat = ((g.par & 1u) ? 0x55555555u : 0xAAAAAAAAu);  // bit i: (j0+32p+i+par) odd
  auto piece_steps = [&](uint32_t jp) -> uint32_t {   // E bits of rows jp .. jp+31
    // Rows jp + 4r + y4 (r < 8): words R0 + r of plane (y4, 0), R0 = jp/4 a
    // multiple of 8, read as two 16-byte vectors per plane.
    uint32_t b = 0;
#pragma unroll
    for (uint32_t y4 = 0; y4 < 4u; ++y4) {
      const uint4* v = reinterpret_cast<const uint4*>(lat + g.word(0, plane(y4, 0), jp >> 2));
      const uint4 lo = __ldcg(v), hi = __ldcg(v + 1);
      const uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
      for (uint32_t r = 0; r < 8u; ++r) b |= (w[r] & 1u) << (4u * r + y4);
    }
    const uint32_t jn = (jp + 32u) & (g.L - 1u);
    const uint32_t bn = __ldcg(lat + g.word(0, plane(jn & 3u, 0), jn >> 2)) & 1u;
    return ~(b ^ ((b >> 1) | (bn << 31)) ^ parpat);
  };
  int32_t sum = 0;
  for (uint32_t p = 0; p < pieces; ++p) sum += 2 * __popc(piece_steps(j0 + 32u * p)) - 32;
  part[t] = sum;
  __syncthreads();
  for (uint32_t off = 1; off < nt; off <<= 1) {   // inclusive Hillis-Steele scan
    const int32_t v = (t >= off) ? part[t - off] : 0;
    __syncthreads();
    part[t] += v;
    __syncthreads();
  }
  int32_t h = (t == 0) ? 0 : part[t - 1];
  for (uint32_t p = 0; p < pieces; ++p) {
    const uint32_t E = piece_steps(j0 + 32u * p);
    int32_t* o = col0 + j0 + 32u * p;
#pragma unroll 8
    for (uint32_t i = 0; i < 32u; ++i) {
      o[i] = h;
      h += ((E >> i) & 1u) ? 1 : -1;
    }
  }
}

// Exact W^2. A band is 32 rows (8 cell rows); a block takes bands by turns and
// leaves of each the column-0 height change D over it and the sums S1, S2 of
// its heights relative to its first site; the last block to finish chains the
// bands (band k starts at the sum of the D above it). One launch: no memset,
// no column-0 kernel, no atomics on the sums.
//
// Warp w of a block takes the rows y4 = w & 3 of the band's cell rows (lane &
// 7) and the segments 4 (w >> 2) + (lane >> 3) of 8 (a lane reads 8
// consecutive cell rows' words with its neighbours: full 32-byte sectors).
// Along a segment a run of 8 sites (kpz_w2.cuh) that starts at height h has
// the height sum m = 8h + A1 and the square sum (m^2 + V) / 8 with V = 8 A2 -
// A1^2, so a run costs one table entry {8D << 16 | V, A1}, whose first word is
// also the running height: m from one shift-add, m and m^2 accumulated.
// The per-run unpacking of D, A1, A2 and the three-term update it replaces
// took 2.57 instructions a site (0.43 ms at L = 2^16 and 0.05 for the column;
// now 0.27 ms, 2.0 TB/s, waiting for loads; 0.33 with 3 blocks an SM, 0.32 with 5).
constexpr uint32_t kBandRows = 32, kBandCells = kBandRows / 4u, kBandThreads = 256, kBandBlocks = 4, kSegs = 8;
// One copy for lanes l and l + 16: 8-byte loads go by half warps.
constexpr size_t kRunTab2Bytes = 256u * 16u * sizeof(uint2);

// Table entry of run byte b (kpz_w2.cuh): {8 D << 16 | V, A1}.
__device__ __forceinline__ uint2 run_entry2(uint32_t b) {
  const uint32_t e = w2::run_entry(b);
  const int32_t A2 = (int32_t)(e & 0xFFu), A1 = (int32_t)((e >> 8) & 0xFFu) - 28, D = (int32_t)(e >> 16) - 8;
  return make_uint2((uint32_t)(8 * D * 65536 + 8 * A2 - A1 * A1), (uint32_t)A1);
}

__global__ void __launch_bounds__(kBandThreads, kBandBlocks) roughness_kernel(const uint32_t* __restrict__ lat, Geometry g,
                                                                    long long* __restrict__ part, RoughOut out) {
  extern __shared__ __align__(16) uint2 tab2[];   // [256][16]
  __shared__ long long seg_s1[kBandRows][kSegs], seg_s2[kBandRows][kSegs];
  __shared__ int seg_dh[kBandRows][kSegs];
  __shared__ bool last;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  {
    const uint2 e = run_entry2(threadIdx.x);   // kBandThreads = 256 entries; a warp writes its 32 side by side
#pragma unroll 8
    for (uint32_t i = 0; i < 16u; ++i) {
      const uint32_t k = 2u * i + (lane >> 4);
      const uint2 v = make_uint2(__shfl_sync(0xffffffffu, e.x, k), __shfl_sync(0xffffffffu, e.y, k));
      tab2[(warp * 32u + k) * 16u + (lane & 15u)] = v;
    }
  }
  __syncthreads();
  const char* tl = reinterpret_cast<const char*>(tab2);
  const uint32_t lane8 = (lane & 15u) * 8u;
  const uint32_t y4 = warp & 3u, rr = lane & 7u, q = (warp >> 2) * 4u + (lane >> 3);
  const uint32_t seg = (g.NB + kSegs - 1u) / kSegs, K0 = min(g.NB, q * seg), K1 = min(g.NB, K0 + seg);
  const uint32_t nb = g.L / kBandRows;
  for (uint32_t band = blockIdx.x; band < nb; band += gridDim.x) {
    const uint32_t R = band * kBandCells + rr, j = 4u * R + y4;
    long long s1 = 0, s2 = 0;   // relative to the segment's first site
    int dH = 0;
    if (K0 < K1) {
      uint32_t Pl[4], Pn[4];
#pragma unroll
      for (uint32_t x4 = 0; x4 < 4; ++x4) {
        Pl[x4] = __ldcg(lat + g.word(K0, plane(y4, x4), R));
        Pn[x4] = __ldcg(lat + g.word((K0 + 1u) & (g.NB - 1u), plane(y4, x4), R));
      }
      for (uint32_t K = K0; K < K1; ++K) {
        uint32_t Pnn[4];   // two blocks ahead
        const uint32_t K2 = (K + 2u) & (g.NB - 1u);
#pragma unroll
        for (uint32_t x4 = 0; x4 < 4; ++x4) Pnn[x4] = __ldcg(lat + g.word(K2, plane(y4, x4), R));
        uint32_t S[4], u[4];
        w2::sigma_x_planes(Pl, Pn[0] & 1u, j, g.par, S);
        w2::run_bytes(S, u);
        int32_t run = 0, sm = 0, sq = 0;
#pragma unroll
        for (uint32_t m = 0; m < 4; ++m)
#pragma unroll
          for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t v = m == 0u ? u[k] << 7 : u[k] >> (8u * m - 7u);
            const uint2 e = *reinterpret_cast<const uint2*>(tl + ((v & 0x7F80u) | lane8));
            const int32_t mm = (run >> 16) + (int32_t)e.y;
            sm += mm;
            sq += mm * mm;
            run += (int32_t)e.x;
          }
        const int32_t a2 = (sq + (run & 0xFFFF)) >> 3;
        s1 += 128ll * dH + sm;
        s2 += (long long)dH * (128ll * dH + 2ll * sm) + a2;
        dH += run >> 19;
#pragma unroll
        for (uint32_t x4 = 0; x4 < 4; ++x4) { Pl[x4] = Pn[x4]; Pn[x4] = Pnn[x4]; }
      }
    }
    seg_s1[4u * rr + y4][q] = s1;
    seg_s2[4u * rr + y4][q] = s2;
    seg_dh[4u * rr + y4][q] = dH;
    __syncthreads();
    if (warp == 0u) {   // lane = row of the band
      const uint32_t jr = band * kBandRows + lane;
      const uint32_t b0 = site_bit(lat, g, 0u, jr), b1 = site_bit(lat, g, 0u, (jr + 1u) & (g.L - 1u));
      const uint32_t upm = __ballot_sync(0xffffffffu, (b0 ^ b1) == ((jr + g.par) & 1u));   // sigma_y(0, jr) = +1
      long long H = 2 * (int)__popc(upm & ((1u << lane) - 1u)) - (int)lane, t1 = 0, t2 = 0;
      for (uint32_t k = 0; k < kSegs; ++k) {
        const long long n = 128ll * (min(g.NB, (k + 1u) * seg) - min(g.NB, k * seg));
        const long long a = seg_s1[lane][k];
        t1 += n * H + a;
        t2 += H * (n * H + 2 * a) + seg_s2[lane][k];
        H += seg_dh[lane][k];
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        t1 += __shfl_xor_sync(0xffffffffu, t1, off);
        t2 += __shfl_xor_sync(0xffffffffu, t2, off);
      }
      if (lane == 0u) {
        part[3u * band] = 2 * (int)__popc(upm) - 32;
        part[3u * band + 1u] = t1;
        part[3u * band + 2u] = t2;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(out.ticket, 1u) == gridDim.x - 1u;
  }
  __syncthreads();
  if (!last) return;
  // Chain the bands: thread t takes bands [t per, (t + 1) per), at most 32. A
  // height is at most the distance from (0,0) along the axes, both ways round,
  // so at L = 2^18 a band's sum of squares is at most 7/3 2^57 (a tent in each
  // direction, at the crest) and a thread's 32 bands stay below 2^64, unsigned;
  // the block adds the threads' 32-bit halves.
  __threadfence();
  __shared__ long long scan[kBandThreads];
  const uint32_t per = (nb + kBandThreads - 1u) / kBandThreads, k0 = min(nb, threadIdx.x * per), k1 = min(nb, k0 + per);
  long long d = 0;
  for (uint32_t k = k0; k < k1; ++k) d += __ldcg(part + 3u * k);
  scan[threadIdx.x] = d;
  __syncthreads();
  for (uint32_t off = 1; off < kBandThreads; off <<= 1) {   // inclusive scan
    const long long v = threadIdx.x >= off ? scan[threadIdx.x - off] : 0;
    __syncthreads();
    scan[threadIdx.x] += v;
    __syncthreads();
  }
  long long H = scan[threadIdx.x] - d, t1 = 0;
  unsigned long long t2 = 0;
  const long long n = (long long)kBandRows * g.L;
  for (uint32_t k = k0; k < k1; ++k) {
    const long long a = __ldcg(part + 3u * k + 1u);
    t1 += n * H + a;
    t2 += (unsigned long long)(H * (n * H + 2 * a) + __ldcg(part + 3u * k + 2u));
    H += __ldcg(part + 3u * k);
  }
  unsigned long long lo = t2 & 0xffffffffull, hi = t2 >> 32;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    t1 += __shfl_xor_sync(0xffffffffu, t1, off);
    lo += __shfl_xor_sync(0xffffffffu, lo, off);
    hi += __shfl_xor_sync(0xffffffffu, hi, off);
  }
  __syncthreads();
  if (lane == 0u) { scan[warp] = t1; scan[8u + warp] = (long long)lo; scan[16u + warp] = (long long)hi; }
  __syncthreads();
  if (threadIdx.x == 0) {
    long long a = 0;
    unsigned long long l = 0, h = 0;
    for (uint32_t k = 0; k < kBandThreads / 32u; ++k) {
      a += scan[k];
      l += (unsigned long long)scan[8u + k];
      h += (unsigned long long)scan[16u + k];
    }
    const unsigned long long s2lo = (h << 32) + l, s2hi = (h >> 32) + (s2lo < l ? 1ull : 0ull);
    *out.ticket = 0u;
    out.sums[0] = a;
    out.sums[1] = (long long)s2lo;
    out.sums[2] = (long long)s2hi;
    if (out.h00) out.sums[3] = *(volatile const long long*)out.h00;
    if (out.err) out.sums[4] = *(volatile const uint32_t*)out.err;
    __threadfence_system();
  }
}

// Heights of the rows of a band, one warp per row and segment of kHeightSeg
// block columns: the segment's start height is col0 plus the height changes of
// the block columns before it (a lane each), then lane c writes the four
// sites of cell c, 32 bytes beside its neighbours'. One thread per row with
// 8-byte stores a row apart took 0.3 ms for a 64-row band at L = 2048.
constexpr uint32_t kHeightSeg = 4;

__global__ void __launch_bounds__(256) heights_kernel(const uint32_t* __restrict__ lat, Geometry g,
                                                      const int32_t* __restrict__ col0, uint32_t j0, uint32_t nrows,
                                                      const unsigned long long* __restrict__ h00,
                                                      int64_t* __restrict__ out) {
  const uint32_t lane = threadIdx.x & 31u, gw = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const uint32_t nseg = (g.NB + kHeightSeg - 1u) / kHeightSeg, r = gw / nseg, q = gw - r * nseg;
  if (r >= nrows) return;
  const uint32_t j = j0 + r, R = j >> 2, y4 = j & 3u, K0 = q * kHeightSeg, K1 = min(g.NB, K0 + kHeightSeg);
  auto steps = [&](uint32_t K, uint32_t (&S)[4]) {
    uint32_t P[4];
#pragma unroll
    for (uint32_t x4 = 0; x4 < 4; ++x4) P[x4] = __ldg(lat + g.word(K, plane(y4, x4), R));
    w2::sigma_x_planes(P, __ldg(lat + g.word((K + 1u) & (g.NB - 1u), plane(y4, 0), R)) & 1u, j, g.par, S);
  };
  int before = 0;
  for (uint32_t K = lane; K < K0; K += 32u) {
    uint32_t S[4];
    steps(K, S);
    before += 2 * (__popc(S[0]) + __popc(S[1]) + __popc(S[2]) + __popc(S[3])) - 128;
  }
  before = __reduce_add_sync(0xffffffffu, before);
  int64_t H = (int64_t)col0[j] + (h00 ? (int64_t)*h00 : 0) + before;
  int64_t* o = out + (size_t)r * g.L + 4u * lane;
  const uint32_t below = (1u << lane) - 1u;
  for (uint32_t K = K0; K < K1; ++K) {
    uint32_t S[4];
    steps(K, S);
    const int up = __popc(S[0] & below) + __popc(S[1] & below) + __popc(S[2] & below) + __popc(S[3] & below);
    int64_t h[4];
    h[0] = H + 2 * up - 4 * (int)lane;
#pragma unroll
    for (int x = 0; x < 3; ++x) h[x + 1] = h[x] + 2 * (int)((S[x] >> lane) & 1u) - 1;
    longlong2* v = reinterpret_cast<longlong2*>(o + 128u * K);
    v[0] = make_longlong2(h[0], h[1]);
    v[1] = make_longlong2(h[2], h[3]);
    H += 2 * (__popc(S[0]) + __popc(S[1]) + __popc(S[2]) + __popc(S[3])) - 128;
  }
}

unsigned grid_for(size_t n, unsigned block) {
  size_t b = (n + block - 1) / block;
  if (b > 152u * 64u) b = 152u * 64u;
  return (unsigned)(b ? b : 1);
}

}  // namespace

cudaError_t launch_init_flat(uint32_t* lat, Geometry g, cudaStream_t st) {
  const size_t n4 = (size_t)g.L * g.L / 128;   // L^2 bits = L^2/128 uint4
  init_flat_kernel<<<grid_for(n4, 256), 256, 0, st>>>(reinterpret_cast<uint4*>(lat), n4);
  count_launch();
  return cudaGetLastError();
}

// Both conversions take j0 and nrows as multiples of 4 (whole cell rows) and a
// 16-byte aligned packed band.
cudaError_t launch_export_packed(const uint32_t* lat, Geometry g, uint32_t j0, uint32_t nrows,
                                 uint32_t* packed, cudaStream_t st) {
  export_kernel<<<4u * ((nrows / 4u + 31u) / 32u), 32u * kIoSegs, 0, st>>>(lat, g, j0, nrows, packed);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_import_packed(uint32_t* lat, Geometry g, uint32_t j0, uint32_t nrows,
                                 const uint32_t* packed, uint32_t* hcar, int32_t* hcol,
                                 cudaStream_t st) {
  import_col_kernel<<<1, 1024, 0, st>>>(packed, g, nrows, hcar, hcol);
  count_launch();
  import_rows_kernel<<<4u * ((nrows / 4u + 31u) / 32u), 32u * kIoSegs, 0, st>>>(lat, g, j0, nrows, packed, hcol);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_col0(const uint32_t* lat, Geometry g, int32_t* col0, cudaStream_t st) {
  col0_kernel<<<1, std::min(kCol0Threads, g.L / 32u), 0, st>>>(lat, g, col0);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_roughness(const uint32_t* lat, Geometry g, void* scratch, const RoughOut& out, cudaStream_t st) {
  constexpr int kMaxDev = 64;
  static std::mutex mu;
  static uint32_t blocks[kMaxDev] = {};   // resident blocks of the device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  uint32_t room = 0;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (dev < kMaxDev) room = blocks[dev];
    if (!room) {
      int per_sm = 0, sms = 0;
      e = cudaFuncSetAttribute(roughness_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRunTab2Bytes);
      if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, roughness_kernel, (int)kBandThreads, kRunTab2Bytes);
      if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      if (e != cudaSuccess) return e;
      room = (uint32_t)std::max(per_sm, 1) * (uint32_t)std::max(sms, 1);
      if (dev < kMaxDev) blocks[dev] = room;
    }
  }
  roughness_kernel<<<std::min(room, g.L / kBandRows), kBandThreads, kRunTab2Bytes, st>>>(
      lat, g, static_cast<long long*>(scratch), out);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_heights(const uint32_t* lat, Geometry g, const int32_t* col0, uint32_t j0,
                           uint32_t nrows, const unsigned long long* h00, int64_t* out,
                           cudaStream_t st) {
  const uint32_t warps = nrows * ((g.NB + kHeightSeg - 1u) / kHeightSeg);
  heights_kernel<<<(warps + 7u) / 8u, 256, 0, st>>>(lat, g, col0, j0, nrows, h00, out);
  count_launch();
  return cudaGetLastError();
}

}  // namespace kpz
