// kpz_tilemem.cuh -- the 16 single-hit rounds of one 128 x 128 tile held by a
// warp in shared memory (arXiv:1204.5072, Sec. 3.1; update rule eq. rule,
// Sec. 2.1; same moves as rounds::tile_rounds, bit for bit).
//
// Lane = cell row of the tile, word bit = cell of the row, as in
// kpz_rounds.cuh, but the 16 words of a lane sit in shared memory as pairs of
// columns (2 px, 2 px + 1) of a row y, one 8-byte slot per lane. The active
// quadrant of a round is then four byte offsets, so a round is one straight
// piece of code for all four quadrants: no dispatch on the set (four copies
// of the round, a divergent-looking branch each and their instruction-cache
// misses cost more than the round's logic), no shuffles (the rows above and
// below are the neighbouring slots) and few registers.
//
// Sites outside the tile: slot 33 of row 0 is the row below the tile, slot 0
// of row 3 the row above it, and the columns left and right of it are bits
// shifted in from `ghost`. A dead site (tile row or column 0) has two
// neighbours in the dead border that never change during the sweep; its
// neighbour outside the tile is given the opposite of one of them, so its
// four neighbours are never all equal and it is never a candidate: the dead
// border costs no instruction in a round.
#pragma once
#include "kpz_internal.h"

namespace kpz {
namespace tilemem {

constexpr uint32_t kSlots = 34;                          // slots of a (row, pair): lanes -1 .. 32
constexpr uint32_t kPairBytes = kSlots * 8u;             // one (row, pair)
constexpr uint32_t kRowBytes = 2u * kPairBytes;

struct TileMem {
  uint2 w[4][2][kSlots];   // [row y of the cell row][columns 2 px, 2 px + 1][1 + lane]
};

// Per quadrant set k = QX + 2 QY: byte offsets (lane 0) of the active pair of
// row 2 QY, of the other pair of that row, of the pair above and the one
// below; then QX, 1 - QX, 8 QY (shift amounts).
struct QuadTab {
  uint4 at[4], sh[4];
};
__device__ __forceinline__ void fill_quad_tab(QuadTab& t, uint32_t k) {
  const uint32_t qx = k & 1u, qy = (k >> 1) & 1u;
  auto off = [](uint32_t y, uint32_t px, uint32_t slot) { return y * kRowBytes + px * kPairBytes + slot * 8u; };
  t.at[k] = make_uint4(off(2u * qy, qx, 1u), off(2u * qy, qx ^ 1u, 1u), qy ? off(1u, qx, 1u) : off(3u, qx, 0u),
                       qy ? off(0u, qx, 2u) : off(2u, qx, 1u));
  t.sh[k] = make_uint4(qx, qx ^ 1u, 8u * qy, 0u);
}

// Site (0,0) in the tile (kTrack): at.x of its quadrant, its cell in its
// lane (0 elsewhere), and masks that turn the position bits into "is its
// site": all ones for column (row) 0 of the quadrant.
struct Origin {
  uint32_t at, mask, nx, ny;
  __device__ __forceinline__ Origin(uint32_t lane, uint32_t u, uint32_t v) {
    at = ((v & 2u) * 2u + (u & 2u) / 2u) * kPairBytes + 8u;
    mask = lane == (v >> 2) ? 1u << ((u >> 2) & 31u) : 0u;
    nx = (u & 1u) ? 0u : ~0u;
    ny = (v & 1u) ? 0u : ~0u;
  }
  // The cell of site (0,0) if it moved: m = cells that moved this round.
  __device__ __forceinline__ uint32_t hit(const uint4& a, uint32_t X, uint32_t Y, uint32_t m) const {
    return a.x == at ? mask & m & (X ^ nx) & (Y ^ ny) : 0u;
  }
};

__device__ __forceinline__ uint2 ld2(const char* p) { return *reinterpret_cast<const uint2*>(p); }
__device__ __forceinline__ void st2(char* p, uint32_t a, uint32_t b) { *reinterpret_cast<uint2*>(p) = make_uint2(a, b); }

// Puts the tile's words, the row below it (hy, lane 31) and, kLive, the row
// above it (up, lane 0) and the bits left of it (left[y] bit 0) into shared
// memory and returns the ghost word: bit 31 - 4 y the site left of row y, bit
// (32 - 4 y) mod 32 the one right of it (hx[y] bit 0).
template <bool kLive>
__device__ __forceinline__ uint32_t put_tile(TileMem& m, uint32_t lane, const uint32_t (&T)[4][4],
                                             const uint32_t (&hx)[4], const uint32_t (&hy)[4],
                                             const uint32_t (&left)[4], const uint32_t (&up)[4]) {
#pragma unroll
  for (int y = 0; y < 4; ++y)
#pragma unroll
    for (int px = 0; px < 2; ++px) m.w[y][px][1 + lane] = make_uint2(T[y][2 * px], T[y][2 * px + 1]);
  if (lane == 31u) {
    m.w[0][0][33] = make_uint2(hy[0], hy[1]);
    m.w[0][1][33] = make_uint2(hy[2], hy[3]);
  }
  if (lane == 0u) {
    const uint32_t nR = __funnelshift_r(T[0][0], hx[0], 1);   // right neighbours of column 3 in the dead row
    m.w[3][0][0] = kLive ? make_uint2(up[0], up[1]) : make_uint2(~T[0][1], ~T[0][2]);
    m.w[3][1][0] = kLive ? make_uint2(up[2], up[3]) : make_uint2(~T[0][3], ~nR);
  }
  uint32_t g = 0u, l[4];
  if (kLive) {
#pragma unroll
    for (int y = 0; y < 4; ++y) l[y] = left[y];
  } else {   // the opposite of the site below, which is in the dead column as well
    uint32_t below = __shfl_down_sync(0xffffffffu, T[0][0], 1);
    if (lane == 31u) below = hy[0];
    l[0] = ~T[1][0]; l[1] = ~T[2][0]; l[2] = ~T[3][0]; l[3] = ~below;
  }
#pragma unroll
  for (int y = 0; y < 4; ++y) g |= ((l[y] & 1u) << (31 - 4 * y)) | ((hx[y] & 1u) << ((32 - 4 * y) & 31));
  __syncwarp();
  return g;
}

// The words around the active quadrant of one round: centre rows c0, c1 (.x,
// .y = its two columns), left / right neighbours l, r of each row, the rows
// above (u) and below (d).
struct Quad {
  uint2 c0, c1, u, d;
  uint32_t l0, r0, l1, r1;
  __device__ __forceinline__ Quad(const char* base, const uint4& at, const uint4& sh, uint32_t ghost) {
    c0 = ld2(base + at.x);
    c1 = ld2(base + at.x + kRowBytes);
    const uint2 o0 = ld2(base + at.y), o1 = ld2(base + at.y + kRowBytes);
    u = ld2(base + at.z);
    d = ld2(base + at.w);
    const uint32_t g0 = __funnelshift_l(ghost, ghost, sh.z), g1 = __funnelshift_l(g0, g0, 4);
    l0 = __funnelshift_l(g0, o0.y, sh.y);   // column 3 of cell c - 1 (QX = 0), else column 1
    l1 = __funnelshift_l(g1, o1.y, sh.y);
    r0 = __funnelshift_r(o0.x, g0, sh.x);   // column 0 of cell c + 1 (QX = 1), else column 2
    r1 = __funnelshift_r(o1.x, g1, sh.x);
  }
};

// All four neighbours higher than a site of parity kOdd: each equals v = s
// (even) or ~s (odd).
template <bool kOdd>
__device__ __forceinline__ uint32_t is_min(uint32_t s, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  return kOdd ? ((a ^ s) & (b ^ s)) & ((c ^ s) & (d ^ s)) : (~(a ^ s) & ~(b ^ s)) & (~(c ^ s) & ~(d ^ s));
}
__device__ __forceinline__ uint32_t all_equal(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  const uint32_t e = ~(a ^ b) & ~(a ^ c);
  return e & ~(c ^ d);
}

// One p = 1, q = 0 round. X, Y: position bits.
template <int kPar, bool kTrack>
__device__ __forceinline__ void round_p1(char* base, const uint4& at, const uint4& sh, uint32_t ghost, uint32_t X,
                                         uint32_t Y, const Origin& og, int& dh) {
  const Quad q(base, at, sh, ghost);
  const uint32_t f00 = is_min<kPar != 0>(q.c0.x, q.l0, q.c0.y, q.u.x, q.c1.x) & ~X & ~Y;
  const uint32_t f01 = is_min<kPar == 0>(q.c0.y, q.c0.x, q.r0, q.u.y, q.c1.y) & X & ~Y;
  const uint32_t f10 = is_min<kPar == 0>(q.c1.x, q.l1, q.c1.y, q.c0.x, q.d.x) & ~X & Y;
  const uint32_t f11 = is_min<kPar != 0>(q.c1.y, q.c1.x, q.r1, q.c0.y, q.d.y) & X & Y;
  if (kTrack && og.hit(at, X, Y, (f00 | f01) | (f10 | f11))) dh += 2;
  st2(base + at.x, q.c0.x ^ f00, q.c0.y ^ f01);
  st2(base + at.x + kRowBytes, q.c1.x ^ f10, q.c1.y ^ f11);
  __syncwarp();
}

// One general-rate round: `accept(up, uq)` returns the cells whose candidate
// (up: a minimum, uq: a maximum) moves.
template <int kPar, bool kTrack, class Accept>
__device__ __forceinline__ void round_general(char* base, const uint4& at, const uint4& sh, uint32_t ghost, uint32_t X,
                                              uint32_t Y, const Origin& og, int& dh, Accept accept) {
  const Quad q(base, at, sh, ghost);
  const uint32_t k00 = all_equal(q.l0, q.c0.y, q.u.x, q.c1.x) & ~X & ~Y;
  const uint32_t k01 = all_equal(q.c0.x, q.r0, q.u.y, q.c1.y) & X & ~Y;
  const uint32_t k10 = all_equal(q.l1, q.c1.y, q.c0.x, q.d.x) & ~X & Y;
  const uint32_t k11 = all_equal(q.c1.x, q.r1, q.c0.y, q.d.y) & X & Y;
  // A candidate is a minimum when a neighbour's bit marks it higher (= v).
  const uint32_t a = (k00 & ~(q.c1.x ^ q.c0.x)) | (k11 & ~(q.c0.y ^ q.c1.y));
  const uint32_t b = (k01 & (q.c1.y ^ q.c0.y)) | (k10 & (q.c0.x ^ q.c1.x));
  const uint32_t even = k00 | k11, odd = k01 | k10, any = even | odd;
  const uint32_t up = kPar ? (even & ~a) | (odd & ~b) : a | b;
  const uint32_t acc = accept(up, any & ~up);
  if (kTrack) {
    const uint32_t h = og.hit(at, X, Y, any & acc);
    if (h) dh += (h & up) ? 2 : -2;
  }
  st2(base + at.x, q.c0.x ^ (k00 & acc), q.c0.y ^ (k01 & acc));
  st2(base + at.x + kRowBytes, q.c1.x ^ (k10 & acc), q.c1.y ^ (k11 & acc));
  __syncwarp();
}

}  // namespace tilemem
}  // namespace kpz
