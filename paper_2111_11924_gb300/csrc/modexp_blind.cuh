// Blinded CRT decryption in one pass per prime (Algorithm 1 "Decryption"
// with the random matrix R, in the Section 2.1 CRT form).
//
// Algorithm 1 recovers m' = m* r'^-1 with m* = c*^d and r' = c_r^d (mod N).
// Modulo each prime r_i of N, and for c_r a unit mod r_i, that residue is
//     (c* c_r^-1)^d = c*^(d_i) * c_r^(r_i - 1 - d_i)   (mod r_i),
// with d_i = d mod (r_i - 1) (Fermat: c_r^(r_i - 1) = 1).  Both powers run
// in one squaring chain (simultaneous exponentiation with interleaved
// sliding windows, Straus / Shamir): about n/b squarings plus the windows
// of the two exponents, instead of a Fermat inversion, a product and a
// second exponentiation.  The residues are recombined by k_crt_sum.
#pragma once

#include "modexp_grid.cuh"

namespace pmk {
namespace dev {

static_assert(kTableMax >= 16, "the joint tables use rows 0-7 (A) and 8-15 (B)");

// a <- A^eA B^eB in Montgomery form.  On entry rows 0 and 8 of tbl hold A
// and B (Montgomery form, this instance); tbl gets A's odd powers in rows
// 0..maxa and B's in rows 8..8+maxb; ybuf is the squaring buffer.  sched is
// a Schedule2 (block-uniform).
template <int S, int TPI>
__device__ __forceinline__ void exp2_window(uint32_t (&a)[S / TPI], uint32_t *tbl, uint32_t *ybuf,
                                            const uint32_t *__restrict__ sched, uint32_t nsteps, uint32_t maxa,
                                            uint32_t maxb, const Modulus<S / TPI> &m, uint32_t r) {
  constexpr int L = S / TPI;
  constexpr int ROW = Layout<S>::kRow;
#pragma unroll 1
  for (int which = 0; which < 2; which++) {  // odd powers of A, then of B
    uint32_t *base = tbl + which * 8 * ROW;
    const uint32_t maxi = which ? maxb : maxa;
    if (maxi == 0) continue;
    load_slice<L>(a, base, r);
    __syncwarp();
    store_slice<L>(ybuf, a, r);
    // k = 0: X^2; k > 0: row k = X^(2k+1)
#pragma unroll 1
    for (uint32_t k = 0; k <= maxi; k++) {
      __syncwarp();
      mont<S, TPI>(a, ybuf, m, r);
      if (k == 0) {
        __syncwarp();
        store_slice<L>(ybuf, a, r);
        load_slice<L>(a, base, r);
      } else {
        store_slice<L>(base + k * ROW, a, r);
      }
    }
    __syncwarp();
  }
  __syncwarp();  // rows 0 and 8, stored by the caller, are read whole below
  const uint32_t s0 = __ldg(sched);
  uint32_t si = 0, nsq = 0, ia = (s0 >> 8) & 0xffu, ib = s0 & 0xffu;  // left of step si
  if (ia != 0xffu) {
    load_slice<L>(a, tbl + ia * ROW, r);
    ia = 0xffu;
  } else {
    load_slice<L>(a, tbl + (8 + ib) * ROW, r);
    ib = 0xffu;
  }
  for (;;) {  // one product in the code, as in exp_window
    const uint32_t *y;
    if (nsq > 0) {
      nsq--;
      __syncwarp();
      store_slice<L>(ybuf, a, r);
      __syncwarp();
      y = ybuf;
    } else if (ia != 0xffu) {
      y = tbl + ia * ROW;
      ia = 0xffu;
    } else if (ib != 0xffu) {
      y = tbl + (8 + ib) * ROW;
      ib = 0xffu;
    } else {
      if (++si >= nsteps) break;
      const uint32_t step = __ldg(sched + si);
      nsq = step >> 16;
      ia = (step >> 8) & 0xffu;
      ib = step & 0xffu;
      continue;
    }
    mont<S, TPI, true>(a, y, m, r);
  }
}

// out[t][i] = c*[t]^(d_i) c_r[t]^(r_i - 1 - d_i) mod r_i for every prime r_i
// of the chunk's key (grid as the CRT mode of k_modexp: blockIdx.y = key *
// parts + i).  With `status`, a c_r divisible by r_i (no inverse mod N)
// sets kStatusNotInvertible.
template <int S, int TPI, int NT>
__global__ void __launch_bounds__(NT, 1) k_blind_crt(const KeyDev *__restrict__ keys, uint32_t K,
                                                  const uint32_t *__restrict__ cstar, const uint32_t *__restrict__ cr,
                                                  uint32_t *__restrict__ out, long long n, int parts,
                                                  uint32_t *__restrict__ status) {
  constexpr int L = S / TPI;
  constexpr int IPB = NT / TPI;
  constexpr int ROW = Layout<S>::kRow;
  constexpr int INST = Layout<S>::kInst;
  const int W = parts * S;
  extern __shared__ __align__(16) uint32_t smem[];
  uint32_t *sR2 = smem, *sOne = smem + ROW, *sR3 = smem + 2 * ROW;
  const uint32_t r = threadIdx.x % TPI, g = threadIdx.x / TPI;
  uint32_t *tbl = smem + Layout<S>::kConstRows * ROW + g * INST;
  uint32_t *ybuf = tbl + kTableMax * ROW;

  const uint32_t key = blockIdx.y / (uint32_t)parts;
  const uint32_t prime = blockIdx.y % (uint32_t)parts;
  const long long first = key + (long long)blockIdx.x * IPB * K;
  if (first >= n) return;  // block-uniform
  const KeyDev &kd = keys[key];
  for (int i = threadIdx.x; i < S; i += NT) {
    sR2[i] = __ldg(kd.R2h[prime] + i);
    sOne[i] = (i == 0);
    sR3[i] = __ldg(kd.R3h[prime] + i);
  }
  __syncthreads();
  // After the barrier the warps are independent: a warp whose instances all
  // lie past the last chunk (the tail block of a key) leaves.
  if (first + (long long)((threadIdx.x / 32) * (32 / TPI)) * K >= n) return;

  const long long t = first + (long long)g * K;
  const bool active = t < n;
  uint32_t a[L];
  Modulus<L> m;
  make_modulus<S, TPI>(m, kd.P[prime], kd.n0h[prime], r);
  crt_input<S, TPI>(a, cstar + t * W, active, parts, sR2, sR3, m, r);  // A = c* R mod r_i
  store_slice<L>(tbl, a, r);
  crt_input<S, TPI>(a, cr + t * W, active, parts, sR2, sR3, m, r);     // B = c_r R mod r_i
  // B = 0 mod r_i: crt_input can leave r_i itself (mont_mul_pairs).  Reducing
  // the pieces first instead took 3,770 and not 3,729 us (2048 bits, 1 MiB),
  // two words instead of two bits in the reduction 3,737 and not 3,726.
  uint32_t any = 0, other = 0;  // not 0, not r_i
#pragma unroll
  for (int j = 0; j < L; j++) {
    any |= a[j];
    other |= a[j] ^ m.n[j];
  }
  uint32_t seen = (any != 0 ? 1u : 0u) | (other != 0 ? 2u : 0u);
  if constexpr (TPI > 1) {
#pragma unroll
    for (int o = 1; o < TPI; o <<= 1) seen |= __shfl_xor_sync(kFull, seen, o, TPI);
  }
  if (status && active && r == 0 && seen != 3u) report(status, kStatusNotInvertible, t);
  store_slice<L>(tbl + 8 * ROW, a, r);
  exp2_window<S, TPI>(a, tbl, ybuf, kd.sched_blind[prime], kd.nsteps_blind[prime], kd.maxa_blind[prime],
                            kd.maxb_blind[prime], m, r);
  mont<S, TPI>(a, sOne, m, r);  // leave the Montgomery domain
  if (active) {
    uint32_t *o = out + t * W + prime * S + r * L;
#pragma unroll
    for (int j = 0; j < L; j++) o[j] = a[j];
  }
}

}  // namespace dev
}  // namespace pmk
