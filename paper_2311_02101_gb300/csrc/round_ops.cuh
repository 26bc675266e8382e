// Device pieces of a round on formulas of at most 3 literals per clause, shared
// by the two-launch, resident (sparse.cu) and local (local.cu) rounds: hidden
// draws of one clause for eight chains, and sums of contributions selected by
// 4-bit hidden patterns.
#pragma once

#include <cstdint>

#include "internal.h"
#include "philox.cuh"

namespace rbmsat {

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}

// acc |= BIT when x < w (unsigned): one compare and one predicated OR
template <uint32_t BIT>
__device__ __forceinline__ void or_if_below(uint32_t& acc, uint32_t x, uint32_t w) {
  asm("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %1, %2;\n\t@p or.b32 %0, %0, %3;\n\t}"
      : "+r"(acc)
      : "r"(x), "r"(w), "n"(BIT));
}

// Unit H's draw for chain Q of the octet against threshold word w: bit
// 4 Q + H of hw (NIB), else bit 8 (Q & 3) + H.
template <bool SAT, bool NIB, int Q, int H>
__device__ __forceinline__ void unit_draw(const uint4 (&R)[3], uint32_t w, uint32_t& hw) {
  const uint32_t word = word_of(R[H], Q >> 1);
  const uint32_t x = (Q & 1) ? (SAT ? (word & 0xFFFF0000u) : word) : (word << 16);
  or_if_below<(1u << ((NIB ? 4 * Q : 8 * (Q & 3)) + H))>(hw, x, w);
}

// Chain Q of the octet: its record (free energy, thresholds of units 0..2)
// and its three draws.
template <bool SAT, bool NIB, int Q>
__device__ __forceinline__ void chain_draws(uint32_t addr_bytes, uint32_t rb, const uint4 (&R)[3],
                                            float& fe, uint32_t& hw) {
  const uint4 r = lds128(__byte_perm(addr_bytes, rb, 0x7650u | (Q & 3)));
  fe += __uint_as_float(r.x);
  unit_draw<SAT, NIB, Q, 0>(R, r.y, hw);
  unit_draw<SAT, NIB, Q, 1>(R, r.z, hw);
  unit_draw<SAT, NIB, Q, 2>(R, r.w, hw);
}

// The octet's hidden pattern: with NIB all 8 chains in h_lo, 4 bits each;
// else chains 0..3 in the bytes of h_lo and 4..7 in those of h_hi.
template <bool SAT, bool NIB>
__device__ __forceinline__ void octet_draws(uint32_t a_lo, uint32_t a_hi, uint32_t rb,
                                            const uint4 (&R)[3], float (&fe)[8], uint32_t& h_lo,
                                            uint32_t& h_hi) {
  chain_draws<SAT, NIB, 0>(a_lo, rb, R, fe[0], h_lo);
  chain_draws<SAT, NIB, 1>(a_lo, rb, R, fe[1], h_lo);
  chain_draws<SAT, NIB, 2>(a_lo, rb, R, fe[2], h_lo);
  chain_draws<SAT, NIB, 3>(a_lo, rb, R, fe[3], h_lo);
  chain_draws<SAT, NIB, 4>(a_hi, rb, R, fe[4], NIB ? h_lo : h_hi);
  chain_draws<SAT, NIB, 5>(a_hi, rb, R, fe[5], NIB ? h_lo : h_hi);
  chain_draws<SAT, NIB, 6>(a_hi, rb, R, fe[6], NIB ? h_lo : h_hi);
  chain_draws<SAT, NIB, 7>(a_hi, rb, R, fe[7], NIB ? h_lo : h_hi);
}

// The hidden draws' Philox4x32-10 blocks, counter (clause, octet | unit << 24, t,
// phase). What a thread needs of rounds 0 and 1 for its octet: round 0's product
// of word z = t (u1 is word x of round 1 without octet and unit, u2 word y), and
// per unit round 1's product of word x.
struct HiddenThread {
  uint32_t u1, u2, th[3], sh[3];
};

__device__ __forceinline__ HiddenThread hidden_thread(uint32_t octet, uint32_t t,
                                                      const RoundKeys& K) {
  HiddenThread Q;
  const uint64_t pt = (uint64_t)kPhiloxM1 * t;
  Q.u1 = (uint32_t)(pt >> 32) ^ K.k0[0];
  Q.u2 = (uint32_t)pt;
#pragma unroll
  for (int h = 0; h < 3; ++h) {
    const uint64_t p = (uint64_t)kPhiloxM0 * ((octet | ((uint32_t)h << 24)) ^ Q.u1);
    Q.th[h] = (uint32_t)(p >> 32) ^ K.k1[1];
    Q.sh[h] = (uint32_t)p;
  }
  return Q;
}

// The clause's share of rounds 0..2: word x of round 2 without the unit is c4,
// the other words of round 3 c5 (to be joined with the unit's) and c6.
struct HiddenClause {
  uint32_t c2, c4, c5, c6;
};

__device__ __forceinline__ HiddenClause hidden_clause(uint32_t u2, uint32_t clause, uint32_t phase,
                                                      const RoundKeys& K) {
  HiddenClause H;
  const uint64_t p0 = (uint64_t)kPhiloxM0 * clause;
  const uint32_t c1 = (uint32_t)(p0 >> 32) ^ phase ^ K.k1[0];
  H.c2 = (uint32_t)p0;
  const uint64_t p1 = (uint64_t)kPhiloxM1 * c1;
  const uint32_t c3 = (uint32_t)(p1 >> 32) ^ u2 ^ K.k0[1];
  H.c4 = (uint32_t)p1;
  const uint64_t p2 = (uint64_t)kPhiloxM0 * c3;
  H.c5 = (uint32_t)(p2 >> 32) ^ K.k1[2];
  H.c6 = (uint32_t)p2;
  return H;
}

// A unit's own part, from round 2's product of word z on.
__device__ __forceinline__ uint4 hidden_unit(const HiddenClause& H, uint32_t th, uint32_t sh,
                                             const RoundKeys& K) {
  const uint64_t pz = (uint64_t)kPhiloxM1 * (th ^ H.c2);
  return philox_rounds<3>(
      make_uint4((uint32_t)(pz >> 32) ^ H.c4 ^ K.k0[2], (uint32_t)pz, H.c5 ^ sh, H.c6), K);
}

__device__ __forceinline__ void hidden_blocks3(const HiddenThread& Q, uint32_t clause,
                                               uint32_t phase, const RoundKeys& K, uint4 (&R)[3]) {
  const HiddenClause H = hidden_clause(Q.u2, clause, phase, K);
#pragma unroll
  for (int h = 0; h < 3; ++h) R[h] = hidden_unit(H, Q.th[h], Q.sh[h], K);
}

// byte permute by a register selector: bits 0..2 of each 4-bit field pick one of
// 8 bytes (bit 3 is never set in a pattern; __byte_perm would mask it first)
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t s) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(s));
  return r;
}

// the contributions of four chains (selector s, low 16 bits) as pairs
__device__ __forceinline__ void nib_pairs(const uint4& tb, uint32_t s, uint32_t& p01,
                                          uint32_t& p23) {
  const uint32_t lo = prmt(tb.x, tb.y, s), hi = prmt(tb.z, tb.w, s);
  p01 = __byte_perm(lo, hi, 0x5140u);
  p23 = __byte_perm(lo, hi, 0x7362u);
}

// adds the contributions of the octet's 8 chains (pattern word h)
__device__ __forceinline__ void nib_add(const uint4& tb, uint32_t h, uint32_t (&acc)[4]) {
  uint32_t a, b;
  nib_pairs(tb, h, a, b);
  acc[0] += a;
  acc[1] += b;
  nib_pairs(tb, h >> 16, a, b);
  acc[2] += a;
  acc[3] += b;
}

// as nib_add for an octet across two temperatures: table ta, and tb for the
// chains of mask mk (one 16-bit half per chain)
__device__ __forceinline__ void nib_add2(const uint4& ta, const uint4& tb, uint32_t h,
                                         const uint32_t (&mk)[4], uint32_t (&acc)[4]) {
#pragma unroll
  for (int w = 0; w < 4; w += 2) {
    uint32_t a, b, a1, b1;
    nib_pairs(ta, w ? h >> 16 : h, a, b);
    nib_pairs(tb, w ? h >> 16 : h, a1, b1);
    acc[w] += (a & ~mk[w]) | (a1 & mk[w]);
    acc[w + 1] += (b & ~mk[w + 1]) | (b1 & mk[w + 1]);
  }
}

// the masks of the chains from `split` on
__device__ __forceinline__ void nib_masks(int split, uint32_t (&mk)[4]) {
#pragma unroll
  for (int w = 0; w < 4; ++w)
    mk[w] = (2 * w >= split ? 0x0000FFFFu : 0u) | (2 * w + 1 >= split ? 0xFFFF0000u : 0u);
}

// the octet's temperatures: tab at the first chain's; returns the first chain
// of the next temperature (8: none; octets have at most two)
__device__ __forceinline__ int nib_split(const DevTables& T, const DevChains& C, int b0,
                                         uint32_t tab0, uint32_t& tab) {
  const int gb0 = C.g8_off * 8 + b0;
  const int e0 = temp_of(gb0, T.n_temps, C.B_total, C.inv_B_total);
  tab = tab0 + (uint32_t)(e0 * T.ptab_stride);
  if (e0 == temp_of(gb0 + 7, T.n_temps, C.B_total, C.inv_B_total)) return 8;
  return (int)(((long long)(e0 + 1) * C.B_total + T.n_temps - 1) / T.n_temps) - gb0;
}

// moves a window's sums (with cw biases) to 32 bits
__device__ __forceinline__ void nib_flush(const uint32_t (&acc)[4], int bias, int (&z)[8]) {
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    z[2 * w] += (int)(acc[w] & 0xFFFFu) - bias;
    z[2 * w + 1] += (int)(acc[w] >> 16) - bias;
  }
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// A window of a variable's incidences (lane k holds incidence k in win): copies
// the 256 chains' pattern rows (128 bytes each, from H, hstride words apart, H
// at the lane's 16 bytes of the tile) to `rows` and the contribution offsets to
// s_off, as one cp.async group. lane / 8 picks one of four rows, lane % 8 its 16
// bytes.
__device__ __forceinline__ void nib_copy_rows(const int2& win, int cnt, const uint32_t* H,
                                              size_t hstride, uint32_t rows, uint32_t* s_off,
                                              int lane) {
  s_off[lane] = (uint32_t)win.y;
  for (int u = 0; u < cnt; u += 4) {
    const int row = u + (lane >> 3);
    const int c = __shfl_sync(0xFFFFFFFFu, win.x, row & 31);
    if (row < cnt)
      cp_async16(rows + (uint32_t)(row * 128 + (lane & 7) * 16), H + (size_t)c * hstride);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// loads of shared memory that changes during the kernel (lds128 reads tables)
__device__ __forceinline__ uint4 lds128_now(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}

// adds a copied window's contributions for the lane's octet; off, hr: shared
// addresses of the offsets and of the lane's word of row 0. `two`: some octet of the warp lies across two temperatures (mk:
// its chains at the second, tab1: that temperature's rows).
__device__ __forceinline__ void nib_sum_rows(uint32_t tab, uint32_t tab1, bool two, int split,
                                             uint32_t off, uint32_t hr, int cnt,
                                             uint32_t (&acc)[4]) {
  const uint32_t end = off + 4u * (uint32_t)cnt;
  if (!two) {
#pragma unroll 1
    for (; off < end; off += 16u, hr += 512u) {
      const uint4 of = lds128_now(off);
      const uint32_t h0 = lds32(hr), h1 = lds32(hr + 128u), h2 = lds32(hr + 256u),
                     h3 = lds32(hr + 384u);
      nib_add(lds128(tab + of.x), h0, acc);
      nib_add(lds128(tab + of.y), h1, acc);
      nib_add(lds128(tab + of.z), h2, acc);
      nib_add(lds128(tab + of.w), h3, acc);
    }
  } else {
    uint32_t mk[4];
    nib_masks(split, mk);
#pragma unroll 1
    for (; off < end; off += 4u, hr += 128u) {
      const uint32_t of = lds32(off);
      nib_add2(lds128(tab + of), lds128(tab1 + of), lds32(hr), mk, acc);
    }
  }
}

}  // namespace rbmsat
