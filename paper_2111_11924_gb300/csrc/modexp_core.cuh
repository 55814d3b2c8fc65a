// Warp-cooperative Montgomery exponentiation for sm_103a.
//
// One exponentiation ("instance") is held by TPI consecutive lanes of a warp;
// lane r keeps limbs [r L, r L + L) of every S-limb value in registers
// (L = S / TPI).  The multiplication is Algorithm 3 (Montgomery) in its
// word-serial CIOS form (Koc, Acar, Kaliski 1996) with r = 2^32 per row and
// R = 2^(32 S) overall:
//     for i in 0..S-1:  T += a * y_i;  q = T_0 * n0 mod 2^32;  T += q N;  T /= 2^32
// followed by one conditional subtraction, so every product is canonical
// (< N).  Exponentiation is Algorithm 2's square-and-multiply generalised to a
// left-to-right sliding window of odd powers (schedules built on the host).
//
// Cost model on this GPU (measured with row-shaped loops, MAC per clock per SM
// at 4 / 8 / 16 warps per SM): a wide multiply-add with carry in and out
// (mad.lo.cc + madc.hi.cc of one 64-bit pair) 19 / 26 / 27, a wide multiply
// whose halves are then added into 64-bit columns 16 / 20 / 20, mad.lo 58 /
// 63 / 64.  The multiplier's high half bounds every form, and the adds are
// free only inside the multiply-add, so a row is built of carry chains over
// 64-bit pairs: one instruction per MAC and nothing but the chain ends on the
// ALU pipe.
// Lane-to-lane carries are deferred: a lane keeps small pending words above
// its L limbs; after the last row a ballot carry-lookahead resolves them in
// O(1) warp operations.
#pragma once

#include <cstdint>

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

// Words of shared memory per stored S-limb value: S + 4 keeps 16-byte rows.
template <int S>
struct Layout {
  static constexpr int kRow = S + 4;
  // Per-instance block (a table of `rows` rows + one operand buffer), padded
  // to 4 mod 32 words so the 32/TPI instances of a warp read distinct
  // 16-byte bank groups.
  static __host__ __device__ constexpr int inst(int rows) {
    return (rows + 1) * kRow + ((4 - ((rows + 1) * kRow) % 32) + 32) % 32;
  }
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

// Resolve the pending word c0 (lane r's belongs at lane r+1's limb 0; the top
// lane's is the value's top word) and reduce the value once by N, leaving the
// canonical result (< N) in t.  Requires the value < 2N.
template <int L, int TPI>
__device__ __forceinline__ void finalize(uint32_t (&t)[L], uint32_t c0, const uint32_t (&nn)[L], uint32_t r) {
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
  }
}

// Rows of a product per unrolled group.  A group of L rows (or 2 L, for whole
// 16-byte reads of y) brings the per-row shift of the lane's words back to
// the starting registers, so no register moves remain.
template <int S, int L>
__host__ __device__ constexpr int row_group() {
  return (L % 4 == 0) ? L : (L % 2 == 0 && S % (2 * L) == 0) ? 2 * L : (L % 2 == 0) ? L : (S % 4 == 0) ? 4 : 2;
}

template <int K>
__device__ __forceinline__ void load_y(uint32_t (&yv)[K], const uint32_t *ys) {
  if constexpr (K % 4 == 0) {
#pragma unroll
    for (int q = 0; q < K; q += 4) {
      const uint4 v = *reinterpret_cast<const uint4 *>(ys + q);
      yv[q] = v.x; yv[q + 1] = v.y; yv[q + 2] = v.z; yv[q + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < K; q += 2) {
      const uint2 v = *reinterpret_cast<const uint2 *>(ys + q);
      yv[q] = v.x; yv[q + 1] = v.y;
    }
  }
}

// a <- MontMul(a, y) = a y R^-1 mod N.  a: this lane's limbs (any value < R);
// ys: y's S limbs in shared memory (y < N), read as 16-byte broadcasts.
// One row at a time, one add-with-carry chain per lane: the form for an odd
// number of limbs per lane, which has no pairs.
template <int S, int TPI>
__device__ __forceinline__ void mont_mul(uint32_t (&a)[S / TPI], const uint32_t *ys, const uint32_t (&nn)[S / TPI],
                                         uint32_t n0, uint32_t r) {
  constexpr int L = S / TPI;
  constexpr int kStep = row_group<S, L>();
  uint32_t t[L];
#pragma unroll
  for (int j = 0; j < L; j++) t[j] = 0;
  uint32_t c0 = 0, c1 = 0;
#pragma unroll 1
  for (int i0 = 0; i0 < S; i0 += kStep) {
    uint32_t yv[kStep];
    load_y<kStep>(yv, ys + i0);
#pragma unroll
    for (int u = 0; u < kStep; u++) {
      row_mac<L>(t, c0, c1, a, yv[u]);
      uint32_t q = t[0] * n0;
      if constexpr (TPI > 1) q = __shfl_sync(kFull, q, 0, TPI);
      row_mac<L>(t, c0, c1, nn, q);
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
  finalize<L, TPI>(t, c0, nn, r);
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

// (w[OFF + 2 i], w[OFF + 2 i + 1]) += m[PAR + 2 i] y for i < L / 2 in one
// carry chain.  CIN: the chain takes the condition code's carry.  The carry
// out is left in the condition code.
template <int L, int PAR, int OFF, bool CIN, int W>
__device__ __forceinline__ void pair_chain(uint32_t (&w)[W], const uint32_t (&m)[L], uint32_t y) {
  if constexpr (CIN) {
    madc_wide_cc(w[OFF], w[OFF + 1], m[PAR], y);
  } else {
    mad_wide_cc(w[OFF], w[OFF + 1], m[PAR], y);
  }
#pragma unroll
  for (int i = 1; i < L / 2; i++) madc_wide_cc(w[OFF + 2 * i], w[OFF + 2 * i + 1], m[PAR + 2 * i], y);
}

// a <- MontMul(a, y) for an even number of limbs per lane: two rows per step.
//
// The lane's part of T is kept as two sums of 64-bit pairs: e, whose word j
// has weight 2^(32 j), and o, whose word j has weight 2^(32 (j + 1)).  The
// even limbs times y_i and the odd limbs times y_{i+1} land on e's pairs, the
// other two products on o's, so each of the four is one carry chain of L / 2
// wide multiply-adds.  The quotient of both rows is one 64-bit value,
// q = T (-N^-1) mod 2^64 of lane 0, and T /= 2^64 moves whole pairs: e and o
// keep their roles and a step needs one broadcast of q and one shift between
// lanes.  A chain's carry out is held back (c0, c1, c2: weights L, L + 1,
// L + 2) and joins the words that the shift brings in.
//
// Bound: the wide multiply-add, 4 L per lane and step against about 26 other
// instructions on other pipes.  Measured against the column form that it
// replaces (2048-bit keys, full d): 12.76 vs 17.67 ms at 1 MiB, 104.9 vs
// 142.7 ms at 10 MiB; CRT 3.41 vs 4.64 ms at 1 MiB.
template <int S, int TPI>
__device__ __forceinline__ void mont_mul_pairs(uint32_t (&a)[S / TPI], const uint32_t *ys,
                                               const uint32_t (&nn)[S / TPI], uint32_t n0, uint32_t r) {
  constexpr int L = S / TPI;
  static_assert(L % 2 == 0, "pairs of limbs");
  constexpr int kStep = row_group<S, L>();
  // -N^-1 mod 2^64 from its low word by one Newton step (lane 0's is used).
  const uint64_t n01 = ((uint64_t)nn[1] << 32) | nn[0];
  const uint32_t k1 = (uint32_t)(((uint64_t)n0 * (2 + n01 * n0)) >> 32);
  const uint32_t below_top = (r == TPI - 1) ? 0u : kFull;
  uint32_t e[L + 2], o[L];
#pragma unroll
  for (int j = 0; j < L; j++) e[j] = o[j] = 0;
  e[L] = e[L + 1] = 0;
  uint32_t c0 = 0, c1 = 0, c2 = 0;
  // The words of weight 0 and 1 go to the lane below (lane 0's are zero).
  auto shifted_out = [&](uint32_t &x0, uint32_t &x1) {
    x0 = e[0];
    x1 = e[1] + o[0];
    if constexpr (TPI > 1) {
      x0 = __shfl_down_sync(kFull, x0, 1, TPI) & below_top;
      x1 = __shfl_down_sync(kFull, x1, 1, TPI) & below_top;
    } else {
      x0 = x1 = 0;
    }
  };
#pragma unroll 1
  for (int i0 = 0; i0 < S; i0 += kStep) {
    uint32_t yv[kStep];
    load_y<kStep>(yv, ys + i0);
#pragma unroll
    for (int u = 0; u < kStep; u += 2) {
      // T /= 2^64.  o's first pair ends in weight 2; the carry of that sum has
      // weight 3, the first word of the new o, where the next chain starts.
      uint32_t x0, x1, drop;
      shifted_out(x0, x1);
      add_cc(drop, e[1], o[0]);
      addc_cc(e[2], e[2], o[1]);
      uint32_t f[L + 2], p[L];
#pragma unroll
      for (int j = 0; j < L; j++) f[j] = e[j + 2];
#pragma unroll
      for (int j = 0; j < L - 2; j++) p[j] = o[j + 2];
      p[L - 2] = p[L - 1] = 0;
      pair_chain<L, 1, 0, true>(p, a, yv[u]);
      uint32_t d1;
      addc(d1, 0u, 0u);
      add_cc(f[L - 2], f[L - 2], c0);
      addc_cc(f[L - 1], f[L - 1], c1);
      addc(c2, c2, 0u);
      add_cc(f[L - 2], f[L - 2], x0);
      addc_cc(f[L - 1], f[L - 1], x1);
      addc(f[L], c2, 0u);
      // T += a (y_i + 2^32 y_{i+1})
      pair_chain<L, 0, 0, false>(f, a, yv[u]);
      addc(f[L], f[L], 0u);
      pair_chain<L, 0, 0, false>(p, a, yv[u + 1]);
      addc(f[L + 1], d1, 0u);
      uint32_t q0 = f[0] * n0;
      uint32_t q1 = __umulhi(f[0], n0) + f[0] * k1 + (f[1] + p[0]) * n0;
      if constexpr (TPI > 1) {
        q0 = __shfl_sync(kFull, q0, 0, TPI);
        q1 = __shfl_sync(kFull, q1, 0, TPI);
      }
      pair_chain<L, 1, 2, false>(f, a, yv[u + 1]);
      addc(c2, 0u, 0u);
      // T += N (q_0 + 2^32 q_1)
      pair_chain<L, 0, 0, false>(f, nn, q0);
      addc(c0, 0u, 0u);
      pair_chain<L, 1, 0, false>(p, nn, q0);
      addc(c1, 0u, 0u);
      pair_chain<L, 0, 0, false>(p, nn, q1);
      addc(c1, c1, 0u);
      pair_chain<L, 1, 2, false>(f, nn, q1);
      addc(c2, c2, 0u);
#pragma unroll
      for (int j = 0; j < L + 2; j++) e[j] = f[j];
#pragma unroll
      for (int j = 0; j < L; j++) o[j] = p[j];
    }
  }
  // The last shift, then e and o in one carry chain.
  uint32_t x0, x1, drop;
  shifted_out(x0, x1);
  add_cc(e[L], e[L], c0);
  addc_cc(e[L + 1], e[L + 1], c1);
  addc(c2, c2, 0u);
  add_cc(e[L], e[L], x0);
  addc_cc(e[L + 1], e[L + 1], x1);
  addc(c2, c2, 0u);
  add_cc(drop, e[1], o[0]);
#pragma unroll
  for (int j = 0; j < L; j++) addc_cc(a[j], e[j + 2], (j + 1 < L) ? o[j + 1] : 0u);
  addc(c2, c2, 0u);
  finalize<L, TPI>(a, c2, nn, r);
}

template <int S, int TPI>
__device__ __forceinline__ void mont(uint32_t (&a)[S / TPI], const uint32_t *ys, const uint32_t (&nn)[S / TPI],
                                     uint32_t n0, uint32_t r) {
  if constexpr ((S / TPI) % 2 == 0) {
    mont_mul_pairs<S, TPI>(a, ys, nn, n0, r);
  } else {
    mont_mul<S, TPI>(a, ys, nn, n0, r);
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

// Table of odd powers and the exponent walk.  On entry a = x in Montgomery
// form; on exit a = x^E in Montgomery form.  tbl: the instance's odd-power
// table (at least maxidx + 1 rows: the table size the schedule was built
// for), ybuf: one row of this instance.  sched: steps of make_schedule()
// (block-uniform).
template <int S, int TPI>
__device__ __forceinline__ void exp_window(uint32_t (&a)[S / TPI], uint32_t *tbl, uint32_t *ybuf,
                                           const uint32_t *__restrict__ sched, uint32_t nsteps, uint32_t maxidx,
                                           const uint32_t (&nn)[S / TPI], uint32_t n0, uint32_t r) {
  constexpr int L = S / TPI;
  constexpr int ROW = Layout<S>::kRow;
  store_slice<L>(tbl, a, r);  // T[0] = x
  if (maxidx > 0) {
    store_slice<L>(ybuf, a, r);
    __syncwarp();
    mont<S, TPI>(a, ybuf, nn, n0, r);  // x^2
    __syncwarp();
    store_slice<L>(ybuf, a, r);
    load_slice<L>(a, tbl, r);
    __syncwarp();
#pragma unroll 1
    for (uint32_t k = 1; k <= maxidx; k++) {  // T[k] = T[k-1] x^2 = x^(2k+1)
      mont<S, TPI>(a, ybuf, nn, n0, r);
      store_slice<L>(tbl + k * ROW, a, r);
    }
    __syncwarp();
  }
  load_slice<L>(a, tbl + __ldg(sched) * ROW, r);
#pragma unroll 1
  for (uint32_t si = 1; si < nsteps; si++) {
    const uint32_t step = __ldg(sched + si);
    const uint32_t nsq = step >> 8, idx = step & 0xffu;
#pragma unroll 1
    for (uint32_t k = 0; k < nsq; k++) {
      __syncwarp();
      store_slice<L>(ybuf, a, r);
      __syncwarp();
      mont<S, TPI>(a, ybuf, nn, n0, r);
    }
    if (idx != 0xffu) mont<S, TPI>(a, tbl + idx * ROW, nn, n0, r);
  }
}

}  // namespace dev
}  // namespace pmk
