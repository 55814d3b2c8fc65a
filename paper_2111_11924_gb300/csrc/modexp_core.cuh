// Warp-cooperative Montgomery exponentiation for sm_103a.
//
// One exponentiation ("instance") is held by TPI consecutive lanes of a warp;
// lane r keeps limbs [r L, r L + L) of every S-limb value in registers
// (L = S / TPI).  The multiplication is Algorithm 3 (Montgomery) in its
// word-serial CIOS form (Koc, Acar, Kaliski 1996), R = 2^(32 S), two words of
// the multiplier a step:
//     for i in 0, 2, .. S-2:  T += a (y_i + 2^32 y_{i+1});  T = (T + q N) / 2^64
// with q so that T + q N is divisible (how q is found: PairSum), followed by
// one conditional subtraction, so that a product of operands below N is
// canonical (< N).  Exponentiation is Algorithm 2's square-and-multiply
// generalised to a left-to-right sliding window of odd powers (schedules built
// on the host).
//
// Cost model on this GPU (measured with row-shaped loops, MAC per clock per SM
// at 4 / 8 / 16 warps per SM): a wide multiply-add with carry in and out
// (mad.lo.cc + madc.hi.cc of one 64-bit pair) 19 / 26 / 27, a wide multiply
// whose halves are then added into 64-bit columns 16 / 20 / 20, mad.lo 58 /
// 63 / 64.  The multiplier's high half bounds every form, and the adds are
// free only inside the multiply-add, so a row is built of carry chains over
// 64-bit pairs: one instruction per MAC and nothing but the chain ends on the
// ALU pipe.  (Forming each cross product of a squaring once was built on top
// of this and left out: 804 instead of 1,024 multiply-adds a lane at 64 limbs
// on 8 lanes, but 400 more adds and moves; the same speed with two warps per
// scheduler, 4% faster with three, and 6% slower at 32 limbs on 4 lanes.)
// Lane-to-lane carries are deferred: a lane keeps small pending words above
// its L limbs; after the last row a ballot carry-lookahead resolves them in
// O(1) warp operations.
#pragma once

#include <cstdint>
#include <type_traits>

#include "pmk_internal.h"

namespace pmk {
namespace dev {

constexpr int kThreads = 128;   // threads per block (4 warps)
constexpr int kTableMax = 1 << (kWindowFull - 1);  // odd powers x^1 .. x^(2 kTableMax - 1)
// Rows of the odd-power table of each size (kTableFull, kTableSmall).
__host__ __device__ constexpr int table_rows(int table) { return table == kTableSmall ? kTableMax / 2 : kTableMax; }
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ void add_cc(uint32_t &r, uint32_t a, uint32_t b) {
  asm volatile("add.cc.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
}
__device__ __forceinline__ void addc_cc(uint32_t &r, uint32_t a, uint32_t b) {
  asm volatile("addc.cc.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
}
__device__ __forceinline__ void addc(uint32_t &r, uint32_t a, uint32_t b) {
  asm volatile("addc.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
}
__device__ __forceinline__ void sub_cc(uint32_t &r, uint32_t a, uint32_t b) {
  asm volatile("sub.cc.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
}
__device__ __forceinline__ void subc_cc(uint32_t &r, uint32_t a, uint32_t b) {
  asm volatile("subc.cc.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
}
__device__ __forceinline__ void subc(uint32_t &r, uint32_t a, uint32_t b) {
  asm volatile("subc.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
}

// Shared-memory layout in words.  Rows of S limbs stand without padding: the
// lanes of a warp read one row index at a time, so only the stride between
// instances matters.  Rows padded to S + 4 left room for 10 warps of the
// 32-limb, 4-lane geometry on an SM instead of 12, and for 8 of the 16-limb,
// 2-lane one instead of 12: CRT took 25.9 instead of 24.7 ms on 41,121 chunks
// of 2048 bits (6.17 instead of 4.77 on 7,000) and 3.54 instead of 2.94 ms on
// 33,000 of 1024 bits.
template <int S>
struct Layout {
  static constexpr int kRow = S;
  // Per-instance block (a table of `rows` rows + one operand buffer), padded
  // to 4 mod 32 words so the 32/TPI instances of a warp read distinct
  // 16-byte bank groups.
  static __host__ __device__ constexpr int inst(int rows) {
    return (rows + 1) * kRow + ((4 - ((rows + 1) * kRow) % 32) + 32) % 32;
  }
  // One operand row per instance, with the same effect.
  static constexpr int kLoneRow = inst(0);
  static constexpr int kInst = inst(kTableMax);
  static constexpr int kConstRows = 3;  // R^2, one, R^3
};

// (t, c0, c1) += a * y, where t is this lane's L limbs and (c0, c1) the
// pending words above them.
template <int L>
__device__ __forceinline__ void row_mac(uint32_t (&t)[L], uint32_t &c0, uint32_t &c1, const uint32_t (&a)[L],
                                        uint32_t y) {
  uint32_t lo[L], hi[L];
#pragma unroll
  for (int j = 0; j < L; j++) {
    const uint64_t p = (uint64_t)a[j] * y;
    lo[j] = (uint32_t)p;
    hi[j] = (uint32_t)(p >> 32);
  }
  add_cc(t[0], t[0], lo[0]);
#pragma unroll
  for (int j = 1; j < L; j++) addc_cc(t[j], t[j], lo[j]);
  addc_cc(c0, c0, 0u);
  addc(c1, c1, 0u);
  if constexpr (L > 1) {
    add_cc(t[1], t[1], hi[0]);
#pragma unroll
    for (int j = 1; j < L - 1; j++) addc_cc(t[j + 1], t[j + 1], hi[j]);
    addc_cc(c0, c0, hi[L - 1]);
  } else {
    add_cc(c0, c0, hi[0]);
  }
  addc(c1, c1, 0u);
}

// Carry-lookahead over the lanes of every TPI-lane group of the warp.
// gen: this lane's word-block overflowed into the next lane; prop: this
// lane's block is all ones (all zeros for borrows) and passes a carry on.
// Returns the carry (0/1) entering this lane.  Top lanes of a group neither
// generate nor propagate into the next group.
__device__ __forceinline__ uint32_t lookahead(bool gen, bool prop, bool top) {
  const uint32_t G = __ballot_sync(kFull, gen && !top);
  const uint32_t P = __ballot_sync(kFull, prop && !top);
  const uint32_t cin = ((G | P) + G) ^ P;  // carry into each bit of (G|P) + G
  return (cin >> (threadIdx.x & 31)) & 1u;
}

// Resolve the pending word c0 of every lane (lane r's belongs at lane r+1's
// limb 0) into t.  Returns the value's word above limb S - 1 (top lane only).
template <int L, int TPI>
__device__ __forceinline__ uint32_t resolve(uint32_t (&t)[L], uint32_t c0, uint32_t r) {
  const bool top = (r == TPI - 1);
  uint32_t topw = top ? c0 : 0u;
  if constexpr (TPI > 1) {
    uint32_t inc = __shfl_up_sync(kFull, c0, 1, TPI);
    if (r == 0) inc = 0;
    uint32_t g;
    add_cc(t[0], t[0], inc);
#pragma unroll
    for (int j = 1; j < L; j++) addc_cc(t[j], t[j], 0u);
    addc(g, 0u, 0u);
    // A pending word is small, so a lane overflows only when its limbs are all
    // but ones and the lookahead is rarely needed.  Leaving it out is 1-3%
    // faster with few limbs per lane (16 limbs on 8 lanes 1.084 and 1.050 ms,
    // 64 on 32 13.15 and 13.07), and up to 1.5% slower with 8.
    if (L > 4 || __any_sync(kFull, g != 0)) {
      uint32_t all1 = t[0];
#pragma unroll
      for (int j = 1; j < L; j++) all1 &= t[j];
      const uint32_t cin = lookahead(g != 0, all1 == 0xffffffffu, top);
      uint32_t g2;
      add_cc(t[0], t[0], cin);
#pragma unroll
      for (int j = 1; j < L; j++) addc_cc(t[j], t[j], 0u);
      addc(g2, 0u, 0u);
      if (top) topw += g + g2;
    }
  }
  return topw;
}

// Subtract N once if the value (topw above t, topw in the top lane) is at
// least N.  Returns whether it was, and the new word above limb S - 1 in topw
// (top lane only).
template <int L, int TPI>
__device__ __forceinline__ bool reduce_once(uint32_t (&t)[L], uint32_t &topw, const uint32_t (&nn)[L], uint32_t r) {
  const bool top = (r == TPI - 1);
  uint32_t d[L], b;
  sub_cc(d[0], t[0], nn[0]);
#pragma unroll
  for (int j = 1; j < L; j++) subc_cc(d[j], t[j], nn[j]);
  subc(b, 0u, 0u);
  b &= 1u;
  if constexpr (TPI > 1) {
    uint32_t any = d[0];
#pragma unroll
    for (int j = 1; j < L; j++) any |= d[j];
    const uint32_t bin = lookahead(b != 0, any == 0, top);
    uint32_t b2;
    sub_cc(d[0], d[0], bin);
#pragma unroll
    for (int j = 1; j < L; j++) subc_cc(d[j], d[j], 0u);
    subc(b2, 0u, 0u);
    b |= b2 & 1u;
  }
  // value - N = (topw - b) 2^(32 S) + d: keep d iff topw >= b (decided by the top lane)
  uint32_t ge = (topw >= b) ? 1u : 0u;
  if constexpr (TPI > 1) ge = __shfl_sync(kFull, ge, TPI - 1, TPI);
  if (ge) {
#pragma unroll
    for (int j = 0; j < L; j++) t[j] = d[j];
    topw -= b;
  }
  return ge;
}

// Resolve pending words and reduce the value once by N, leaving the canonical
// result (< N) in t.  Requires the value < 2N.
template <int L, int TPI>
__device__ __forceinline__ void finalize(uint32_t (&t)[L], uint32_t c0, const uint32_t (&nn)[L], uint32_t r) {
  uint32_t topw = resolve<L, TPI>(t, c0, r);
  reduce_once<L, TPI>(t, topw, nn, r);
}

// Store / load this lane's L limbs of a value at row + r L.
template <int L>
__device__ __forceinline__ void store_slice(uint32_t *row, const uint32_t (&a)[L], uint32_t r) {
  uint32_t *p = row + r * L;
  if constexpr (L % 4 == 0) {
#pragma unroll
    for (int j = 0; j < L; j += 4) *reinterpret_cast<uint4 *>(p + j) = make_uint4(a[j], a[j + 1], a[j + 2], a[j + 3]);
  } else {
#pragma unroll
    for (int j = 0; j < L; j++) p[j] = a[j];
  }
}
template <int L>
__device__ __forceinline__ void load_slice(uint32_t (&a)[L], const uint32_t *row, uint32_t r) {
  const uint32_t *p = row + r * L;
  if constexpr (L % 4 == 0) {
#pragma unroll
    for (int j = 0; j < L; j += 4) {
      const uint4 v = *reinterpret_cast<const uint4 *>(p + j);
      a[j] = v.x; a[j + 1] = v.y; a[j + 2] = v.z; a[j + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < L; j++) a[j] = p[j];
  }
}
template <int L>
__device__ __forceinline__ void load_slice_global(uint32_t (&a)[L], const uint32_t *__restrict__ row, uint32_t r) {
  const uint32_t *p = row + r * L;
  if constexpr (L % 4 == 0) {
#pragma unroll
    for (int j = 0; j < L; j += 4) {
      const uint4 v = __ldg(reinterpret_cast<const uint4 *>(p + j));
      a[j] = v.x; a[j + 1] = v.y; a[j + 2] = v.z; a[j + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < L; j++) a[j] = __ldg(p + j);
  }
}

// Whether the top lane takes lane 0's words in the place of a zero (see
// PairSum).  It spares two of about 15 instructions a step beside the
// multiply-adds, which counts where a lane has few limbs: 2 limbs per lane
// 38.6 against 36.5 ms (2048-bit full d, 12,000 chunks) and 35.5 against 33.0
// (CRT, 41,121 chunks), 3 limbs 3.41 against 3.35 (3072-bit CRT, 685 chunks);
// with 4 limbs or more it measured the same to 3% slower, but on two lanes
// 2% faster (16 limbs, CRT at 1024 bits, 33,000 chunks: 3.00 and 2.93 ms).
template <int L, int TPI>
__host__ __device__ constexpr bool ring() {
  return L <= 3 || TPI == 2;
}

// A modulus N as the products use it: this lane's limbs of N, and for the form
// of PairSum of f = F, or F - 2^(32 (S - 2)) mod N with ring(), where
// F = (k N + 1) / 2^64 and k = -N^-1 mod 2^64.  tight: N is so near 2^(32 S)
// that a product can reach 2N before its last subtraction.
template <int L>
struct Modulus {
  uint32_t n[L], f[L];
  uint32_t k0, k1;
  bool tight;
};

// a <- MontMul(a, y) = a y R^-1 mod N.  a: this lane's limbs (any value < R);
// ys: y's S limbs in shared or global memory (y < N).
// One row at a time, one add-with-carry chain per lane: the form for one limb
// per lane and for four limbs on two (see pair_form).
template <int S, int TPI>
__device__ __forceinline__ void mont_mul_chain(uint32_t (&a)[S / TPI], const uint32_t *ys, const Modulus<S / TPI> &m,
                                               uint32_t r) {
  constexpr int L = S / TPI;
  uint32_t t[L];
#pragma unroll
  for (int j = 0; j < L; j++) t[j] = 0;
  uint32_t c0 = 0, c1 = 0;
  constexpr int kStep = (S % 4 == 0) ? 4 : 2;  // rows per 16- or 8-byte read of y
#pragma unroll 1
  for (int i0 = 0; i0 < S; i0 += kStep) {
    uint32_t yv[kStep];
    load_slice<kStep>(yv, ys + i0, 0);
#pragma unroll
    for (int u = 0; u < kStep; u++) {
      row_mac<L>(t, c0, c1, a, yv[u]);
      uint32_t q = t[0] * m.k0;
      if constexpr (TPI > 1) q = __shfl_sync(kFull, q, 0, TPI);
      row_mac<L>(t, c0, c1, m.n, q);
      // T /= 2^32: limb 0 of lane 0 is now zero; every lane takes the next
      // lane's limb 0 as its new top limb and folds its pending word into it.
      uint32_t in = 0;
      if constexpr (TPI > 1) {
        in = __shfl_down_sync(kFull, t[0], 1, TPI);
        if (r == TPI - 1) in = 0;
      }
#pragma unroll
      for (int j = 0; j < L - 1; j++) t[j] = t[j + 1];
      add_cc(t[L - 1], in, c0);
      addc(c0, c1, 0u);
      c1 = 0;
    }
  }
  finalize<L, TPI>(t, c0, m.n, r);
#pragma unroll
  for (int j = 0; j < L; j++) a[j] = t[j];
}

// (lo, hi) += a y, a 64-bit pair, with the carry out (and in, for madc) in the
// condition code; each compiles to one wide multiply-add.
__device__ __forceinline__ void mad_wide_cc(uint32_t &lo, uint32_t &hi, uint32_t a, uint32_t y) {
  asm volatile("mad.lo.cc.u32 %0, %2, %3, %0;\n\tmadc.hi.cc.u32 %1, %2, %3, %1;" : "+r"(lo), "+r"(hi) : "r"(a), "r"(y));
}
__device__ __forceinline__ void madc_wide_cc(uint32_t &lo, uint32_t &hi, uint32_t a, uint32_t y) {
  asm volatile("madc.lo.cc.u32 %0, %2, %3, %0;\n\tmadc.hi.cc.u32 %1, %2, %3, %1;" : "+r"(lo), "+r"(hi) : "r"(a), "r"(y));
}

// (w[OFF + 2 i], w[OFF + 2 i + 1]) += m[PAR + 2 i] y over the limbs of one
// parity (PAR) in one carry chain.  CIN: the chain takes the condition code's
// carry.  The carry out is left in the condition code.
template <int L, int PAR, int OFF, bool CIN = false, int W>
__device__ __forceinline__ void pair_chain(uint32_t (&w)[W], const uint32_t (&m)[L], uint32_t y) {
  if constexpr (CIN) {
    madc_wide_cc(w[OFF], w[OFF + 1], m[PAR], y);
  } else {
    mad_wide_cc(w[OFF], w[OFF + 1], m[PAR], y);
  }
#pragma unroll
  for (int i = 1; i < (L + 1 - PAR) / 2; i++) madc_wide_cc(w[OFF + 2 * i], w[OFF + 2 * i + 1], m[PAR + 2 * i], y);
}

// pair_chain whose last pair starts from zero.
template <int L, int PAR, int W>
__device__ __forceinline__ void pair_chain_new_top(uint32_t (&w)[W], const uint32_t (&m)[L], uint32_t y) {
#pragma unroll
  for (int i = 0; i < L / 2 - 1; i++) madc_wide_cc(w[2 * i], w[2 * i + 1], m[PAR + 2 * i], y);
  asm volatile("madc.lo.cc.u32 %0, %2, %3, 0;\n\tmadc.hi.cc.u32 %1, %2, %3, 0;"
               : "=r"(w[L - 2]), "=r"(w[L - 1])
               : "r"(m[PAR + L - 2]), "r"(y));
}

__device__ __forceinline__ void mul_wide(uint32_t &lo, uint32_t &hi, uint32_t a, uint32_t y) {
  const uint64_t p = (uint64_t)a * y;
  lo = (uint32_t)p;
  hi = (uint32_t)(p >> 32);
}

// The running sum T of a Montgomery product for an even number of limbs per
// lane, two rows (64 bits of y) a step.
//
// A lane's part of T is two sums of 64-bit pairs: e, whose word j has weight
// 2^(32 j), and o, whose word j has weight 2^(32 (j + 1)).  The even limbs
// times y_i and the odd limbs times y_{i+1} land on e's pairs, the other two
// products on o's, so each of the four is one carry chain of L / 2 wide
// multiply-adds, and T / 2^64 moves whole pairs: e and o keep their roles.
// (Separate sums for even and odd products are common practice; their spread
// over lanes, the order of the chains and the ring are this library's own.)
//
// Reduction (quotients by Orup 1995, "Simplifying quotient determination in
// high-radix modular multiplication").  F = (k N + 1) / 2^64 with
// k = -N^-1 mod 2^64 makes
// k N = F 2^64 - 1, so adding T mod 2^64 times k N clears the low 64 bits:
//     T <- floor(T / 2^64) + (T mod 2^64) F.
// The quotient is lane 0's two low words as they stand, with no product by k
// on the way, and F has no more limbs than N.  Every lane passes its two low
// words to the lane below.  With ring() lane 0 passes them to the top lane,
// which so adds the quotient times 2^(32 (S - 2)), and
// f = F - 2^(32 (S - 2)) mod N makes up for it; else the top lane takes zeros
// and f = F.  T stays below (2^64 + 2) N + a; the last two steps therefore
// reduce by N itself (q = T k mod 2^64: lane 0's low words become zero), which
// brings T below 2N, or below 3N when the top 64 bits of N are all but ones
// (Modulus::tight).
//
// Chains are ordered so that each one's carry out falls on a word that holds
// only carries yet.  The two words a lane passes down and the next quotient
// are sent before a step's last two chains, which hide the shuffles.
template <int L, int TPI>
struct PairSum {
  uint32_t e[L + 2], o[L], c2;  // c2: weight 2^(32 (L + 2))
  uint32_t x0, x1, q0, q1;      // from the lane above (its words 0, 1), and the quotient
  int above;                    // the lane above; lane 0 for the top lane
  uint32_t keep;                // zero in the top lane, unless ring()

  __device__ __forceinline__ explicit PairSum(uint32_t r)
      : above((int)((r + 1) % TPI)), keep(!ring<L, TPI>() && r == TPI - 1 ? 0u : kFull) {}

  __device__ __forceinline__ uint32_t from_above(uint32_t x) const {
    return ring<L, TPI>() ? __shfl_sync(kFull, x, above, TPI) : __shfl_down_sync(kFull, x, 1, TPI);
  }
  __device__ __forceinline__ uint32_t in(uint32_t x) const { return ring<L, TPI>() ? x : x & keep; }

  template <bool QUOTIENT>
  __device__ __forceinline__ void send() {
    x0 = e[0];
    x1 = e[1] + o[0];
    if constexpr (TPI > 1) {
      if constexpr (QUOTIENT) {
        q0 = __shfl_sync(kFull, x0, 0, TPI);
        q1 = __shfl_sync(kFull, x1, 0, TPI);
      }
      x0 = from_above(x0);
      x1 = from_above(x1);
    } else {
      q0 = x0;
      q1 = x1;
      x0 = x1 = 0;
    }
  }

  // T = a (y0 + 2^32 y1)
  __device__ __forceinline__ void start(const uint32_t (&a)[L], uint32_t y0, uint32_t y1) {
#pragma unroll
    for (int j = 0; j < L; j += 2) {
      mul_wide(e[j], e[j + 1], a[j], y0);
      mul_wide(o[j], o[j + 1], a[j + 1], y0);
    }
    pair_chain<L, 0, 0>(o, a, y1);
    addc(e[L + 1], 0u, 0u);
    e[L] = 0;
    send<true>();
    pair_chain<L, 1, 2>(e, a, y1);
    c2 = 0;
  }

  // T = T / 2^64 + a (y0 + 2^32 y1), and with REDUCE + (q0 + 2^32 q1) f.
  template <bool REDUCE>
  __device__ __forceinline__ void step(const uint32_t (&a)[L], uint32_t y0, uint32_t y1, const uint32_t (&f)[L]) {
    uint32_t d, drop;  // d: weight L + 1
    // o's first pair ends in weight 2, the new weight 0; the carry of that
    // sum has the new weight 1, where o's next chain starts (and ends in a
    // pair that was zero: no carry out).
    add_cc(drop, e[1], o[0]);
    addc_cc(e[2], e[2], o[1]);
#pragma unroll
    for (int j = 0; j < L - 2; j++) o[j] = o[j + 2];
    pair_chain_new_top<L, 1>(o, a, y0);
#pragma unroll
    for (int j = 0; j < L; j++) e[j] = e[j + 2];
    pair_chain<L, 0, 0>(e, a, y0);
    addc(e[L], c2, 0u);
    pair_chain<L, 0, 0>(o, a, y1);
    addc(d, 0u, 0u);
    add_cc(e[L - 2], e[L - 2], in(x0));
    addc_cc(e[L - 1], e[L - 1], in(x1));
    addc(e[L], e[L], 0u);
    if constexpr (REDUCE) {
      pair_chain<L, 0, 0>(e, f, q0);
      addc(e[L], e[L], 0u);
      pair_chain<L, 1, 0>(o, f, q0);
      addc(d, d, 0u);
      const uint32_t p1 = q1;
      pair_chain<L, 0, 0>(o, f, p1);
      addc(e[L + 1], d, 0u);
      send<true>();
      pair_chain<L, 1, 2>(e, a, y1);
      addc(c2, 0u, 0u);
      pair_chain<L, 1, 2>(e, f, p1);
      addc(c2, c2, 0u);
    } else {
      e[L + 1] = d;
      pair_chain<L, 1, 2>(e, a, y1);
      addc(c2, 0u, 0u);
    }
  }

  // T += q N with q = T (-N^-1) mod 2^64
  __device__ __forceinline__ void reduce(const Modulus<L> &m) {
    const uint64_t w = (uint64_t)e[0] * m.k0;
    uint32_t p0 = (uint32_t)w;
    uint32_t p1 = (uint32_t)(w >> 32) + e[0] * m.k1 + (e[1] + o[0]) * m.k0;
    if constexpr (TPI > 1) {
      p0 = __shfl_sync(kFull, p0, 0, TPI);
      p1 = __shfl_sync(kFull, p1, 0, TPI);
    }
    uint32_t c0, c1;  // carries of weight L and L + 1, whose words are full here
    pair_chain<L, 0, 0>(e, m.n, p0);
    addc(c0, 0u, 0u);
    pair_chain<L, 1, 0>(o, m.n, p0);
    addc(c1, 0u, 0u);
    pair_chain<L, 0, 0>(o, m.n, p1);
    addc(c1, c1, 0u);
    send<false>();
    pair_chain<L, 1, 2>(e, m.n, p1);
    addc(c2, c2, 0u);
    add_cc(e[L], e[L], c0);
    addc_cc(e[L + 1], e[L + 1], c1);
    addc(c2, c2, 0u);
  }

  // t = T / 2^64 (rounded down); returns the lane's pending word.
  __device__ __forceinline__ uint32_t shift_out(uint32_t (&t)[L]) {
    uint32_t drop, c;
    add_cc(e[L], e[L], in(x0));
    addc_cc(e[L + 1], e[L + 1], in(x1));
    addc(c, c2, 0u);
    add_cc(drop, e[1], o[0]);
#pragma unroll
    for (int j = 0; j < L; j++) addc_cc(t[j], e[j + 2], (j + 1 < L) ? o[j + 1] : 0u);
    addc(c, c, 0u);
    return c;
  }
};

// PairSum for an odd number of limbs per lane: three, always with ring().  The
// even limbs are one more than the odd ones, so e ends in weight L and o in
// weight L + 1, and the words that hold only carries are others: the chains'
// order differs.
template <int L, int TPI>
struct OddPairSum {
  static_assert(L % 2 == 1 && L > 1 && ring<L, TPI>(), "every lane takes the words of the next one");
  uint32_t e[L + 1], o[L + 1], c1, c2;  // c1, c2: weights 2^(32 (L + 1)), 2^(32 (L + 2))
  uint32_t x0, x1, q0, q1;
  int above;  // the lane above; lane 0 for the top lane

  __device__ __forceinline__ explicit OddPairSum(uint32_t r) : above((int)((r + 1) % TPI)) {}

  template <bool QUOTIENT>
  __device__ __forceinline__ void send() {
    x0 = e[0];
    x1 = e[1] + o[0];
    if constexpr (QUOTIENT) {
      q0 = __shfl_sync(kFull, x0, 0, TPI);
      q1 = __shfl_sync(kFull, x1, 0, TPI);
    }
    x0 = __shfl_sync(kFull, x0, above, TPI);
    x1 = __shfl_sync(kFull, x1, above, TPI);
  }

  __device__ __forceinline__ void start(const uint32_t (&a)[L], uint32_t y0, uint32_t y1) {
#pragma unroll
    for (int j = 0; j < L; j += 2) mul_wide(e[j], e[j + 1], a[j], y0);
#pragma unroll
    for (int j = 1; j < L; j += 2) mul_wide(o[j - 1], o[j], a[j], y0);
    o[L - 1] = o[L] = 0;
    pair_chain<L, 0, 0>(o, a, y1);
    c2 = 0;  // a (y0 + 2^32 y1) ends below weight L + 2
    send<true>();
    pair_chain<L, 1, 2>(e, a, y1);
    addc(c1, 0u, 0u);
  }

  template <bool REDUCE>
  __device__ __forceinline__ void step(const uint32_t (&a)[L], uint32_t y0, uint32_t y1, const uint32_t (&f)[L]) {
    uint32_t drop, d;  // d: weight L + 1
    add_cc(drop, e[1], o[0]);
    addc_cc(e[2], e[2], o[1]);
#pragma unroll
    for (int j = 0; j < L - 1; j++) o[j] = o[j + 2];
    pair_chain<L, 1, 0, true>(o, a, y0);
    addc(o[L - 1], 0u, 0u);
#pragma unroll
    for (int j = 0; j < L - 1; j++) e[j] = e[j + 2];
    e[L - 1] = c1;
    e[L] = c2;
    pair_chain<L, 0, 0>(e, a, y0);
    addc(d, 0u, 0u);
    add_cc(e[L - 2], e[L - 2], x0);
    addc_cc(e[L - 1], e[L - 1], x1);
    addc_cc(e[L], e[L], 0u);
    addc(d, d, 0u);
    if constexpr (REDUCE) {
      pair_chain<L, 0, 0>(e, f, q0);
      addc(d, d, 0u);
      pair_chain<L, 1, 0>(o, f, q0);
      addc(o[L - 1], o[L - 1], 0u);
    }
    o[L] = d;
    pair_chain<L, 0, 0>(o, a, y1);
    addc(c2, 0u, 0u);
    if constexpr (REDUCE) {
      const uint32_t p1 = q1;
      pair_chain<L, 0, 0>(o, f, p1);
      addc(c2, c2, 0u);
      send<true>();
      pair_chain<L, 1, 2>(e, a, y1);
      addc(c1, 0u, 0u);
      pair_chain<L, 1, 2>(e, f, p1);
      addc(c1, c1, 0u);
    } else {
      pair_chain<L, 1, 2>(e, a, y1);
      addc(c1, 0u, 0u);
    }
  }

  __device__ __forceinline__ void reduce(const Modulus<L> &m) {
    const uint64_t w = (uint64_t)e[0] * m.k0;
    uint32_t p0 = (uint32_t)w;
    uint32_t p1 = (uint32_t)(w >> 32) + e[0] * m.k1 + (e[1] + o[0]) * m.k0;
    p0 = __shfl_sync(kFull, p0, 0, TPI);
    p1 = __shfl_sync(kFull, p1, 0, TPI);
    uint32_t c0;  // weight L, whose words are full here
    pair_chain<L, 0, 0>(e, m.n, p0);
    addc(c1, c1, 0u);
    pair_chain<L, 1, 0>(o, m.n, p0);
    addc(c0, 0u, 0u);
    pair_chain<L, 0, 0>(o, m.n, p1);
    addc(c2, c2, 0u);
    send<false>();
    pair_chain<L, 1, 2>(e, m.n, p1);
    addc(c1, c1, 0u);
    add_cc(o[L - 1], o[L - 1], c0);
    addc_cc(o[L], o[L], 0u);
    addc(c2, c2, 0u);
  }

  __device__ __forceinline__ uint32_t shift_out(uint32_t (&t)[L]) {
    uint32_t drop, c;
    add_cc(e[L], e[L], x0);
    addc_cc(o[L], o[L], x1);
    addc(c, c2, 0u);
    add_cc(o[L], o[L], c1);
    addc(c, c, 0u);
    add_cc(drop, e[1], o[0]);
#pragma unroll
    for (int j = 0; j < L; j++) addc_cc(t[j], (j + 2 <= L) ? e[j + 2] : 0u, o[j + 1]);
    addc(c, c, 0u);
    return c;
  }
};

// Whether products of S limbs on TPI lanes take the form of PairSum: not with
// one limb per lane, which has no pairs, nor at four limbs, where making F and
// the last two reductions cost more than the rows (256-bit CRT, 1,700 chunks:
// 72.5 us in pairs and 67.3 by rows; 8 limbs on 2 lanes, 512-bit CRT, 168 in
// pairs and 183 by rows).
template <int S, int TPI>
__host__ __device__ constexpr bool pair_form() {
  return S / TPI > 1 && S > 4;
}

template <int S, int TPI>
__device__ __forceinline__ void make_modulus(Modulus<S / TPI> &m, const uint32_t *N, uint32_t n0, uint32_t r) {
  constexpr int L = S / TPI;
  load_slice_global<L>(m.n, N, r);
  m.k0 = n0;
  m.tight = false;
  if constexpr (pair_form<S, TPI>()) {
    // -N^-1 mod 2^64 from its low word by one Newton step, in lane 0
    const uint64_t n01 = ((uint64_t)m.n[1] << 32) | m.n[0];
    m.k1 = (uint32_t)(((uint64_t)n0 * (2 + n01 * n0)) >> 32);
    if constexpr (TPI > 1) m.k1 = __shfl_sync(kFull, m.k1, 0, TPI);
    std::conditional_t<L % 2 == 0, PairSum<L, TPI>, OddPairSum<L, TPI>> t(r);
    t.start(m.n, m.k0, m.k1);
    if (r == TPI - 1) t.x0 = t.x1 = 0;
    const uint32_t c = t.shift_out(m.f);
    // k N = -1 mod 2^64: the + 1 carries out of the dropped words into lane 0
    uint32_t g;
    add_cc(m.f[0], m.f[0], r == 0 ? 1u : 0u);
#pragma unroll
    for (int j = 1; j < L; j++) addc_cc(m.f[j], m.f[j], 0u);
    addc(g, c, 0u);
    resolve<L, TPI>(m.f, g, r);
    if constexpr (ring<L, TPI>()) {
      // f = F + (N - 2^(32 (S - 2))) mod N; N has exactly 32 S bits
      uint32_t n1 = m.n[L - 2], n2 = m.n[L - 1];
      if (r == TPI - 1) {
        sub_cc(n1, n1, 1u);
        subc(n2, n2, 0u);
      }
      add_cc(m.f[0], m.f[0], L == 2 ? n1 : m.n[0]);
#pragma unroll
      for (int j = 1; j < L; j++) addc_cc(m.f[j], m.f[j], j == L - 1 ? n2 : j == L - 2 ? n1 : m.n[j]);
      addc(g, 0u, 0u);
      uint32_t topw = resolve<L, TPI>(m.f, g, r);
      reduce_once<L, TPI>(m.f, topw, m.n, r);
    }
    uint32_t t1 = m.n[L - 1], t0 = m.n[L - 2];
    if constexpr (TPI > 1) {
      t1 = __shfl_sync(kFull, t1, TPI - 1, TPI);
      t0 = __shfl_sync(kFull, t0, TPI - 1, TPI);
    }
    m.tight = t1 == 0xffffffffu && t0 >= 0xfffffff0u;  // T < 2N needs the top 64 bits of N below 2^64 - 5
  }
}

// Steps of a product unrolled together.  HOT is the exponentiation's own
// product (one site per kernel), unrolled whole where that still measured
// faster; elsewhere as many steps as bring a lane's words back to the
// registers they started from.  Clocks per product with 1 / 2 / 3 warps per
// scheduler, L / 2 steps against the whole product: 64 limbs on 32 lanes
// 3,316 / 4,765 / 6,913 and 2,504 / 3,763 / 5,197, on 16 lanes 4,581 / 6,572 /
// 9,568 and 3,835 / 5,684 / 8,433, on 8 lanes 7,279 / 10,376 / 16,009 and
// 6,860 / 9,863 / 15,620; 32 limbs on 4 lanes 3,917 / 5,511 and 3,711 / 5,245.
template <int S, int L, bool HOT>
__host__ __device__ constexpr int unrolled_steps() {
  return !HOT                                                ? (L == 2 ? 2 : L % 2 ? L : L / 2)
         : (S <= 96 && L <= 12) || (S == 128 && L <= 4)      ? S / 2 - 2
         : L % 2 == 0 && 12 % (L / 2) == 0                   ? 12
                                                             : L / 2;
}

// a <- MontMul(a, y) = a y R^-1 mod N for two or more limbs per lane.
// ys: y's S limbs in shared or global memory.
//
// Range.  The steps add Q N with Q < R (1 + d), d = 2.01 / 2^64 (the quotients
// of F stand for products with k < 2^64, or k + 2^64 with ring()), so
// T < a y / R + N (1 + d).  For a, y < N that is below 2N, or below 3N when
// tight, and the result is canonical.  For a in [N, R) T is below N (1 + d) + y:
// the result is congruent but, with y that close to N and N not tight, can be
// N or just above, below N (1 + d).  CRT pieces and chunks >= N are such
// operands; the products that follow see values below N (1 + 2 d), after
// mod_add, and 5 d < 16 / 2^64 keeps them below 2N, so the next result is
// canonical again, and so is the last one, with 1.  Whoever looks at a value
// before that takes N for zero (k_blind_crt).
//
// Bound: the wide multiply-add, 4 L per lane and step at 4 clocks of the
// fma-heavy pipe each, against about 20 other instructions a step (64 limbs
// on 8 lanes: 1,028 instructions on that pipe and 680 others a product).  A
// single warp issues one per 6.6 clocks; two warps per scheduler take 9,700
// clocks for a product each, 85% of the pipe, three or more 4,650 per product.
// Measured, 2048-bit keys, default geometry, in ms with 64-bit columns / pairs
// and a quotient by product / now: full d 1 MiB 17.63 / 12.66 / 11.40, 10 MiB
// 142.3 / 104.1 / 93.1; CRT 1 MiB 4.63 / 3.34 / 3.08.
template <int S, int TPI, bool HOT>
__device__ __forceinline__ void mont_mul_pairs(uint32_t (&a)[S / TPI], const uint32_t *ys, const Modulus<S / TPI> &m,
                                               uint32_t r) {
  constexpr int L = S / TPI;
  constexpr int kReduced = S / 2 - 2;  // steps between the first pair of rows and the last
  constexpr int G = unrolled_steps<S, L, HOT>() > 0 ? unrolled_steps<S, L, HOT>() : 1;
  constexpr int kHead = kReduced % G;
  const uint2 *yp = reinterpret_cast<const uint2 *>(ys);
  std::conditional_t<L % 2 == 0, PairSum<L, TPI>, OddPairSum<L, TPI>> t(r);
  uint2 y = yp[0], next = yp[1];  // y is read one step ahead
  t.start(a, y.x, y.y);
#pragma unroll
  for (int i = 1; i <= kHead; i++) {
    y = next;
    next = yp[i + 1];
    t.template step<true>(a, y.x, y.y, m.f);
  }
  if constexpr (kReduced >= G) {
#pragma unroll 1
    for (int i0 = kHead + 1; i0 <= kReduced; i0 += G) {
#pragma unroll
      for (int i = 0; i < G; i++) {
        y = next;
        next = yp[i0 + i + 1];
        t.template step<true>(a, y.x, y.y, m.f);
      }
    }
  }
  t.reduce(m);
  t.template step<false>(a, next.x, next.y, m.f);
  t.reduce(m);
  const uint32_t pending = t.shift_out(a);
  uint32_t topw = resolve<L, TPI>(a, pending, r);
  reduce_once<L, TPI>(a, topw, m.n, r);
  if (m.tight) reduce_once<L, TPI>(a, topw, m.n, r);
}

template <int S, int TPI, bool HOT = false>
__device__ __forceinline__ void mont(uint32_t (&a)[S / TPI], const uint32_t *ys, const Modulus<S / TPI> &m, uint32_t r) {
  if constexpr (pair_form<S, TPI>()) {
    mont_mul_pairs<S, TPI, HOT>(a, ys, m, r);
  } else {
    mont_mul_chain<S, TPI>(a, ys, m, r);
  }
}

// a <- (a + b) mod N for a, b < N (distributed add, lookahead, one reduction).
template <int L, int TPI>
__device__ __forceinline__ void mod_add(uint32_t (&a)[L], const uint32_t (&b)[L], const uint32_t (&nn)[L], uint32_t r) {
  uint32_t c;
  add_cc(a[0], a[0], b[0]);
#pragma unroll
  for (int j = 1; j < L; j++) addc_cc(a[j], a[j], b[j]);
  addc(c, 0u, 0u);
  // c is this lane's carry into the next lane: reuse finalize, whose first
  // step moves a lane's pending word into the next lane's limb 0.
  finalize<L, TPI>(a, c, nn, r);
}

// Table of odd powers and the exponent walk.  On entry a = x in Montgomery
// form; on exit a = MontMul(x^E in Montgomery form, last), that is, for any
// x < N, x^E R^-E last mod N.  tbl: the instance's odd-power table (at least
// maxidx + 1 rows: the table size the schedule was built for), ybuf: one row
// of this instance.  sched: steps of make_schedule() (warp-uniform).
// Squarings and multiplications share one product in the code, so that it can
// be unrolled whole.
template <int S, int TPI>
__device__ __forceinline__ void exp_window(uint32_t (&a)[S / TPI], uint32_t *tbl, uint32_t *ybuf,
                                           const uint32_t *__restrict__ sched, uint32_t nsteps, uint32_t maxidx,
                                           const uint32_t *last, const Modulus<S / TPI> &m, uint32_t r) {
  constexpr int L = S / TPI;
  constexpr int ROW = Layout<S>::kRow;
  store_slice<L>(tbl, a, r);  // T[0] = x
  if (maxidx > 0) {
    store_slice<L>(ybuf, a, r);
    // k = 0: x^2; k > 0: T[k] = T[k-1] x^2 = x^(2k+1)
#pragma unroll 1
    for (uint32_t k = 0; k <= maxidx; k++) {
      __syncwarp();
      mont<S, TPI>(a, ybuf, m, r);
      if (k == 0) {
        __syncwarp();
        store_slice<L>(ybuf, a, r);
        load_slice<L>(a, tbl, r);
      } else {
        store_slice<L>(tbl + k * ROW, a, r);
      }
    }
    __syncwarp();
  }
  load_slice<L>(a, tbl + __ldg(sched) * ROW, r);
  uint32_t si = 0, nsq = 0, idx = 0xffu;  // squarings and multiplication left of step si
  for (;;) {
    const uint32_t *y;
    if (nsq > 0) {
      nsq--;
      __syncwarp();
      store_slice<L>(ybuf, a, r);
      __syncwarp();
      y = ybuf;
    } else if (idx != 0xffu) {
      y = tbl + idx * ROW;
      idx = 0xffu;
    } else if (++si < nsteps) {
      const uint32_t step = __ldg(sched + si);
      nsq = step >> 8;
      idx = step & 0xffu;
      continue;
    } else if (si == nsteps) {
      y = last;
    } else {
      break;
    }
    mont<S, TPI, true>(a, y, m, r);
  }
}

}  // namespace dev
}  // namespace pmk
