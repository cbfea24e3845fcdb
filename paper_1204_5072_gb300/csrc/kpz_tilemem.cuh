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

struct alignas(16) TileMem {
  uint2 w[4][2][kSlots];   // [row y of the cell row][columns 2 px, 2 px + 1][1 + lane]
  uint2 ghost[2][32];      // [QY][lane]: ghost words of rows 2 QY, 2 QY + 1 (put_tile)
  uint4 at[kRounds], sh[kRounds];   // of each round's quadrant set (QuadTab)
};
constexpr uint32_t kGhostOff = 4u * kRowBytes;

// Per quadrant set k = QX + 2 QY: at = byte offsets (lane 0) of the active
// pair of row 2 QY, of the other pair of that row, of the pair above and the
// one below; sh = QX, 1 - QX, offset of the ghost words. one, neg: 1 and -1 as
// values the compiler cannot see through (add_fma).
struct QuadTab {
  uint4 at[4], sh[4];
  uint32_t one, neg;
};
__device__ __forceinline__ void fill_quad_tab(QuadTab& t, uint32_t k) {
  const uint32_t qx = k & 1u, qy = (k >> 1) & 1u;
  auto off = [](uint32_t y, uint32_t px, uint32_t slot) { return y * kRowBytes + px * kPairBytes + slot * 8u; };
  t.at[k] = make_uint4(off(2u * qy, qx, 1u), off(2u * qy, qx ^ 1u, 1u), qy ? off(1u, qx, 1u) : off(3u, qx, 0u),
                       qy ? off(0u, qx, 2u) : off(2u, qx, 1u));
  t.sh[k] = make_uint4(qx, qx ^ 1u, kGhostOff + qy * 256u, 0u);
  if (k == 0u) { t.one = 1u; t.neg = ~0u; }
}

// a * m + b on the FMA pipe. With m = one or neg from shared memory it is an
// addition or subtraction that does not load the ALU pipe, which bounds the
// general-rate rounds: all their logic, shifts and compares run on it.
__device__ __forceinline__ uint32_t add_fma(uint32_t a, uint32_t m, uint32_t b) {
  uint32_t r;
  asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(m), "r"(b));
  return r;
}

// The rounds' offsets of a tile with quadrant sets setw (two bits a round).
__device__ __forceinline__ void put_rounds(TileMem& m, const QuadTab& tab, uint32_t lane, uint32_t setw) {
  if (lane < kRounds) {
    const uint32_t k = (setw >> (2u * lane)) & 3u;
    m.at[lane] = tab.at[k];
    m.sh[lane] = tab.sh[k];
  }
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

// Shared-memory access by 32-bit address and constant offset.
template <int kOff = 0>
__device__ __forceinline__ uint2 ld2(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2+%3];" : "=r"(v.x), "=r"(v.y) : "r"(a), "n"(kOff));
  return v;
}
template <int kOff = 0>
__device__ __forceinline__ void st2(uint32_t a, uint32_t x, uint32_t y) {
  asm volatile("st.shared.v2.u32 [%0+%1], {%2, %3};" ::"r"(a), "n"(kOff), "r"(x), "r"(y) : "memory");
}
template <int kOff = 0>
__device__ __forceinline__ uint4 ld4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4+%5];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(a), "n"(kOff));
  return v;
}

// Puts the tile's words, the row below it (hy, lane 31), the bits right of it
// (hx[y] bit 0) and, kLive, the row above it (up, lane 0) and the bits left of
// it (left[y] bit 0) into shared memory. A ghost word holds the site left of
// its row at bit 31 and the one right of it at bit 0: it is shifted in beside
// the row's outer column. The caller synchronises the warp.
template <bool kLive>
__device__ __forceinline__ void put_tile(TileMem& m, uint32_t lane, const uint32_t (&T)[4][4],
                                         const uint32_t (&hx)[4], const uint32_t (&hy)[4], const uint32_t (&left)[4],
                                         const uint32_t (&up)[4]) {
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
  uint32_t l[4];
  if (kLive) {
#pragma unroll
    for (int y = 0; y < 4; ++y) l[y] = left[y];
  } else {   // the opposite of the site below, which is in the dead column as well
    uint32_t below = __shfl_down_sync(0xffffffffu, T[0][0], 1);
    if (lane == 31u) below = hy[0];
    l[0] = ~T[1][0]; l[1] = ~T[2][0]; l[2] = ~T[3][0]; l[3] = ~below;
  }
  uint32_t g[4];
#pragma unroll
  for (int y = 0; y < 4; ++y) g[y] = (l[y] << 31) | (hx[y] & 1u);
  m.ghost[0][lane] = make_uint2(g[0], g[1]);
  m.ghost[1][lane] = make_uint2(g[2], g[3]);
}

// The tile's words after the rounds.
__device__ __forceinline__ void get_tile(const TileMem& m, uint32_t lane, uint32_t (&T)[4][4]) {
#pragma unroll
  for (int y = 0; y < 4; ++y)
#pragma unroll
    for (int px = 0; px < 2; ++px) {
      const uint2 v = m.w[y][px][1u + lane];
      T[y][2 * px] = v.x;
      T[y][2 * px + 1] = v.y;
    }
}

// The words around the active quadrant of one round: centre rows c0, c1 (.x,
// .y = its two columns), left / right neighbours l, r of each row, the rows
// above (u) and below (d).
struct Quad {
  uint32_t at;             // address of the active pair of row 2 QY
  uint2 c0, c1, u, d;
  uint32_t l0, r0, l1, r1;
  __device__ __forceinline__ Quad(uint32_t base, const uint4& ofs, const uint4& sh, uint32_t one) {
    at = add_fma(ofs.x, one, base);
    const uint32_t o = add_fma(ofs.y, one, base);
    c0 = ld2(at);
    c1 = ld2<kRowBytes>(at);
    const uint2 o0 = ld2(o), o1 = ld2<kRowBytes>(o), g = ld2(add_fma(sh.z, one, base));
    u = ld2(add_fma(ofs.z, one, base));
    d = ld2(add_fma(ofs.w, one, base));
    l0 = __funnelshift_l(g.x, o0.y, sh.y);   // column 3 of cell c - 1 (QX = 0), else column 1
    l1 = __funnelshift_l(g.y, o1.y, sh.y);
    r0 = __funnelshift_r(o0.x, g.x, sh.x);   // column 0 of cell c + 1 (QX = 1), else column 2
    r1 = __funnelshift_r(o1.x, g.y, sh.x);
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
__device__ __forceinline__ void round_p1(uint32_t base, const uint4& ofs, const uint4& sh, uint32_t one, uint32_t X,
                                         uint32_t Y, const Origin& og, int& dh) {
  const Quad q(base, ofs, sh, one);
  const uint32_t f00 = is_min<kPar != 0>(q.c0.x, q.l0, q.c0.y, q.u.x, q.c1.x) & ~X & ~Y;
  const uint32_t f01 = is_min<kPar == 0>(q.c0.y, q.c0.x, q.r0, q.u.y, q.c1.y) & X & ~Y;
  const uint32_t f10 = is_min<kPar == 0>(q.c1.x, q.l1, q.c1.y, q.c0.x, q.d.x) & ~X & Y;
  const uint32_t f11 = is_min<kPar != 0>(q.c1.y, q.c1.x, q.r1, q.c0.y, q.d.y) & X & Y;
  if (kTrack && og.hit(ofs, X, Y, (f00 | f01) | (f10 | f11))) dh += 2;
  st2(q.at, q.c0.x ^ f00, q.c0.y ^ f01);
  st2<kRowBytes>(q.at, q.c1.x ^ f10, q.c1.y ^ f11);
  __syncwarp();
}

// Thresholds of a tile at general rates. A candidate's four neighbours carry
// one bit; class A are the candidates where, counted on even sites, it equals
// the site's own: the minima of a tile whose site (0,0) is even, the maxima of
// an odd one. So Ta = Tp, Tb = Tq on even tiles and the reverse on odd ones,
// and a round needs no parity. kEdge: a rate is 0 or 1 (all or none accepted
// without drawing); otherwise those terms drop out.
template <bool kEdge>
struct Rates {
  uint32_t Ta, Tb, ca, cb, ba[4], bb[4];
  uint32_t draw_a, draw_b, all_a, all_b;
  __device__ __forceinline__ Rates(const SweepParams& P, bool odd) {
    Ta = odd ? P.Tq : P.Tp;
    Tb = odd ? P.Tp : P.Tq;
    ca = deep_const(Ta);
    cb = deep_const(Tb);
#pragma unroll
    for (uint32_t n = 0; n < 4u; ++n) {
      ba[n] = 0u - ((Ta >> (15u - n)) & 1u);
      bb[n] = 0u - ((Tb >> (15u - n)) & 1u);
    }
    draw_a = (Ta != 0u && Ta < 65536u) ? ~0u : 0u;
    draw_b = (Tb != 0u && Tb < 65536u) ? ~0u : 0u;
    all_a = (Ta >> 16) ? ~0u : 0u;
    all_b = (Tb >> 16) ? ~0u : 0u;
  }
  // Both 16-bit halves t + 0x7FFF for t = T's low twelve bits: minus a 12-bit
  // number h the top bit of a half is set exactly when h < t.
  static __device__ __forceinline__ uint32_t deep_const(uint32_t T) { return ((T & 0xFFFu) + 0x7FFFu) * 0x10001u; }
};
// The four 12-bit numbers of lo, hi (16-bit halves) against the threshold of
// constant c: the outcome of number k in the top bit of byte k.
__device__ __forceinline__ uint32_t deep_below(uint32_t lo, uint32_t hi, uint32_t c, uint32_t neg) {
  return __byte_perm(add_fma(lo & 0x0FFF0FFFu, neg, c), add_fma(hi & 0x0FFF0FFFu, neg, c), 0x7531);
}

// All ones where the top bit of byte k of w is set.
template <int k>
__device__ __forceinline__ uint32_t byte_mask(uint32_t w) {
  uint32_t r;
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(w), "n"(0x8888 + 0x1111 * k));
  return r;
}
// Acceptance of a general-rate round (the rule of rounds::one_round) of cell
// row `lane`: the candidates' (any; same: class A) top four bits (block A)
// against their threshold by a majority chain; the k-th tie from below takes
// the k-th deep outcome, the top bits of the bytes of Wa (as class A) and Wb.
template <bool kEdge>
__device__ __forceinline__ uint32_t accept_cells(const SweepParams& P, const Rates<kEdge>& R, uint32_t tid, uint32_t s,
                                                 const uint4& A, uint32_t Wa, uint32_t Wb, uint32_t lane, uint32_t r,
                                                 uint32_t same, uint32_t any, uint32_t one, uint32_t neg) {
  const uint32_t dm = kEdge ? any & ((same & R.draw_a) | (~same & R.draw_b)) : any;   // need random bits
  const uint32_t w[4] = {A.x, A.y, A.z, A.w};
  uint32_t b[4];
#pragma unroll
  for (uint32_t n = 0; n < 4u; ++n) b[n] = (same & R.ba[n]) | (~same & R.bb[n]);
  uint32_t lt = ~w[3] & b[3];
#pragma unroll
  for (int n = 2; n >= 0; --n) lt = (~w[n] & lt) | (~w[n] & b[n]) | (lt & b[n]);
  uint32_t tie = dm;
#pragma unroll
  for (int n = 0; n < 4; ++n) tie &= ~(w[n] ^ b[n]);
  uint32_t acc = lt & dm;
  if (kEdge) acc |= any & ((same & R.all_a) | (~same & R.all_b));
  // The k-th tie from below takes the k-th outcome; a row has a fourth one in
  // seven rounds of a thousand, so three are taken without a branch.
  const uint32_t g0 = (same & byte_mask<0>(Wa)) | (~same & byte_mask<0>(Wb));
  const uint32_t g1 = (same & byte_mask<1>(Wa)) | (~same & byte_mask<1>(Wb));
  const uint32_t g2 = (same & byte_mask<2>(Wa)) | (~same & byte_mask<2>(Wb));
  const uint32_t m1 = tie & add_fma(tie, one, neg), m2 = m1 & add_fma(m1, one, neg), m3 = m2 & add_fma(m2, one, neg);
  acc |= (tie & ~m1 & g0) | (m1 & ~m2 & g1);
  acc |= m2 & ~m3 & g2;
  if (m3 != 0u) {   // the fourth, and from the fifth on the overflow blocks of the round
    const uint32_t m4 = m3 & (m3 - 1u);
    acc |= m3 & ~m4 & ((same & byte_mask<3>(Wa)) | (~same & byte_mask<3>(Wb)));
    uint4 X = make_uint4(0u, 0u, 0u, 0u);
    uint32_t m = m4;
    for (uint32_t k = 0u; m != 0u; ++k) {
      const uint32_t bit = m & (0u - m);
      m ^= bit;
      if ((k & 7u) == 0u)
        X = philox((kTagDeep << 28) | (lane << 8) | (r << 3) | (1u + (k >> 3)), tid, s, P.sample, P.k0, P.k1);
      const uint32_t x = (k & 4u) ? ((k & 2u) ? X.w : X.z) : ((k & 2u) ? X.y : X.x);
      const uint32_t h = ((k & 1u) ? (x >> 16) : x) & 0xFFFu;
      acc |= (h < (((bit & same) ? R.Ta : R.Tb) & 0xFFFu)) ? bit : 0u;
    }
  }
  return acc;
}

// One general-rate round: `accept(same, any)` returns the cells whose
// candidate (any; same: class A) moves. odd: parity of the tile's site (0,0).
template <bool kTrack, class Accept>
__device__ __forceinline__ void round_general(uint32_t base, const uint4& ofs, const uint4& sh, uint32_t one, uint32_t X,
                                              uint32_t Y, bool odd, const Origin& og, int& dh, Accept accept) {
  const Quad q(base, ofs, sh, one);
  const uint32_t k00 = all_equal(q.l0, q.c0.y, q.u.x, q.c1.x) & ~X & ~Y;
  const uint32_t k01 = all_equal(q.c0.x, q.r0, q.u.y, q.c1.y) & X & ~Y;
  const uint32_t k10 = all_equal(q.l1, q.c1.y, q.c0.x, q.d.x) & ~X & Y;
  const uint32_t k11 = all_equal(q.c1.x, q.r1, q.c0.y, q.d.y) & X & Y;
  const uint32_t e = q.c0.x ^ q.c1.x, f = q.c0.y ^ q.c1.y;   // neighbour against own bit, by column
  const uint32_t same = ((k00 & ~e) | (k10 & e)) | ((k11 & ~f) | (k01 & f));
  const uint32_t any = (k00 | k01 | k10) | k11;
  const uint32_t acc = accept(same, any);
  if (kTrack) {
    const uint32_t h = og.hit(ofs, X, Y, any & acc);
    if (h) dh += ((h & same) != 0u) != odd ? 2 : -2;
  }
  st2(q.at, q.c0.x ^ (k00 & acc), q.c0.y ^ (k01 & acc));
  st2<kRowBytes>(q.at, q.c1.x ^ (k10 & acc), q.c1.y ^ (k11 & acc));
  __syncwarp();
}

// The 16 single-hit rounds of the tile in m (put_tile, put_rounds) at general
// rates, its numbers drawn on the way (draw(c0): Philox block of counter word
// 0 = c0 for this tile and sweep). Returns the height change of site (0,0).
//
// Bound: the ALU pipe (logic, shifts, compares: two cycles a warp instruction)
// beside the wide multiplies of Philox (3.5 cycles each, 640 a tile). Measured
// at L = 2^16, p = 0.95: 1.27 ms a sweep against 1.58 ms with the tile in
// registers and a four-way dispatch on the set (2190 against 2600 ALU
// instructions a tile); additions on the FMA pipe 1.27 against 1.32, no terms
// for rates of 0 and 1 1.32 against 1.37. Slower: 20 or 24 resident warps at 96
// or 80 registers (1.50, 1.58), one copy of the round in a loop of 16 (1.46),
// Philox rounds of the next pair between the rounds of this one (1.39). At
// p = 1 the same rounds are bound by the 16 shared-memory wavefronts a round
// (0.56 ms against 0.47 in registers), so that path keeps its registers.
template <bool kEdge, bool kTrack, class Draw>
__device__ __forceinline__ int rounds_drawn(TileMem& m, const QuadTab& tab, const SweepParams& P, uint32_t tid,
                                            uint32_t s, bool odd, const Origin& og, uint32_t lane, Draw draw) {
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(&m) + lane * 8u;
  uint32_t rt = (uint32_t)__cvta_generic_to_shared(m.at);
  const uint32_t one = *(const volatile uint32_t*)&tab.one, neg = *(const volatile uint32_t*)&tab.neg;
  constexpr int kSh = (int)sizeof(m.at);
  int dh = 0;
  const Rates<kEdge> R(P, odd);
#pragma unroll 1
  for (uint32_t rp = 0; rp < kRounds / 2; ++rp) {
    const uint4 pos = draw((kTagPos << 28) | (lane << 3) | rp);
    const uint4 D = draw((kTagDeep << 28) | (lane << 8) | (rp << 4));
    const uint4 A0 = draw((kTagAcc << 28) | (lane << 4) | (2u * rp));
    const uint4 A1 = draw((kTagAcc << 28) | (lane << 4) | (2u * rp + 1u));
    round_general<kTrack>(base, ld4(rt), ld4<kSh>(rt), one, pos.x, pos.y, odd, og, dh, [&](uint32_t same, uint32_t any) {
      return accept_cells<kEdge>(P, R, tid, s, A0, deep_below(D.x, D.y, R.ca, neg), deep_below(D.x, D.y, R.cb, neg), lane,
                                 2u * rp, same, any, one, neg);
    });
    round_general<kTrack>(base, ld4<16>(rt), ld4<kSh + 16>(rt), one, pos.z, pos.w, odd, og, dh,
                          [&](uint32_t same, uint32_t any) {
                            return accept_cells<kEdge>(P, R, tid, s, A1, deep_below(D.z, D.w, R.ca, neg),
                                                       deep_below(D.z, D.w, R.cb, neg), lane, 2u * rp + 1u, same, any, one,
                                                       neg);
                          });
    rt += 32u;
  }
  return dh;
}

}  // namespace tilemem
}  // namespace kpz
