// Head-term kernels for BBP digit extraction (Sze, arXiv:1008.3171, Sec. 3 and 4.3):
// the per-warp tile loop (Montgomery window ladder for s = 2^(e+W) mod m, exact-division
// digits t = floor(2^(e+W)/m) mod 2^W, signed accumulation), the single-range head
// kernel and the persistent queue kernel.  Templates only: each accumulator class is
// instantiated in its own translation unit (bbp_inst.cuh).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "bbp_device.cuh"
#include "bbp_finalize.cuh"
#include "bbp_kernels.cuh"
#include "bbp_tail.cuh"

namespace bbp {

// ---------------------------------------------------------------- head terms
//
// Work split: a warp owns a tile of 32 * S * run consecutive terms; lane l, stream s
// owns the run starting at tile + (l S + s) run.  Along a run, m, the exponent and
// R mod m advance incrementally, and the exponents of a warp stay within
// step * 32 * S * run of each other, so the ladder length (the warp maximum of the
// exponent bit length) is almost always shared.  Each stream evaluates a pair
// (k, k+1) per step, so (-1)^k is static in the code.

// State of one stream at its current term.
struct StreamState {
  uint64_t rel;  // term index relative to k_begin (clamped to the last term)
  uint64_t m;    // modulus a k + b
  uint64_t E;    // exponent of the residue the ladder produces: e + W = d + c - step k + W
  RTrack tr;     // R = q m + r
};

// Modulus paths (the planner picks one per launch range by the moduli's bit length):
//   0: one 32-bit word, lazy residues, bitlen(m) <= 29
//   1: two words, bitlen(m) <= 46 (three-word square, shift after the first REDC step)
//   2: two words, bitlen(m) <= 60 (four-word square)
//   3: one 32-bit word, fully reduced residues, bitlen(m) of 30 or 31
template <int PATH>
struct PathTraits {
  static constexpr bool kWide = PATH == 1 || PATH == 2;
  static constexpr int kRBits = kWide ? 64 : 32;
};

template <int PATH, int NT>
__device__ __forceinline__ void square_all(uint32_t (&x0)[NT], uint32_t (&x1)[NT], const uint32_t (&m0)[NT],
                                           const uint32_t (&m1)[NT], const uint32_t (&mp)[NT],
                                           const uint32_t (&sh)[NT], bool do_shift) {
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    if (PATH == 1) sqr_redc64_p1(x0[t], x1[t], sh[t], Mod64{m0[t], m1[t], mp[t]}, do_shift);
    else if (PATH == 2) sqr_shift_redc64(x0[t], x1[t], sh[t], Mod64{m0[t], m1[t], mp[t]}, do_shift);
    else x0[t] = sqr_shift_redc32<PATH == 3>(x0[t], sh[t], m0[t], m1[t], do_shift);  // m1: m^-1 mod 2^32
  }
}

// The first squaring of a path-1 ladder takes the unreduced first window
// x = (R mod m) << w0 < m 2^w0, beyond the three-word routine's x < 2m: it runs the
// general four-word routine, whose bound is bitlen(m) + 2 w0 + s <= 64.
template <int NT>
__device__ __forceinline__ void square_all_general(uint32_t (&x0)[NT], uint32_t (&x1)[NT], const uint32_t (&m0)[NT],
                                                   const uint32_t (&m1)[NT], const uint32_t (&mp)[NT],
                                                   const uint32_t (&sh)[NT], bool do_shift) {
#pragma unroll
  for (int t = 0; t < NT; ++t) sqr_shift_redc64(x0[t], x1[t], sh[t], Mod64{m0[t], m1[t], mp[t]}, do_shift);
}

template <int NT>
__device__ __forceinline__ void reduce_all(uint32_t (&x0)[NT], uint32_t (&x1)[NT], const uint32_t (&m0)[NT],
                                           const uint32_t (&m1)[NT], const uint32_t (&mp)[NT]) {
#pragma unroll
  for (int t = 0; t < NT; ++t) reduce_once64(x0[t], x1[t], Mod64{m0[t], m1[t], mp[t]});
}

// Quotient digits of every term, least significant first, folded straight into
// the LMAX-limb sum with a signed carry (odd terms subtracted when NEG_ODD).  A
// term of a lane past the range has x = 0, whose digits are all 0.
template <bool WIDE, bool NEG_ODD, int NT, int LMAX>
__device__ __forceinline__ void fold_digits(uint32_t (&acc)[LMAX], uint32_t (&x0)[NT], uint32_t (&x1)[NT],
                                            const uint32_t (&m0)[NT], const uint32_t (&m1)[NT],
                                            const uint32_t (&mp)[NT]) {
  int64_t carry = 0;
#pragma unroll
  for (int i = 0; i < LMAX; ++i) {
    int64_t sum = static_cast<int64_t>(acc[i]) + carry;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      uint32_t q;
      if (WIDE) {
        q = hensel_step64(x0[t], x1[t], Mod64{m0[t], m1[t], mp[t]});
      } else {
        q = x0[t] * mp[t];
        x0[t] = __umulhi(q, m0[t]) + (x0[t] != 0u ? 1u : 0u);
      }
      if (NEG_ODD && (t & 1)) sum -= q;
      else sum += q;
    }
    acc[i] = static_cast<uint32_t>(sum);
    carry = sum >> 32;
  }
}

// `len` squarings of one window group: len - 1 plain, then one with the group's
// value shifted in.  len <= 4.
template <int PATH, int NT>
__device__ __forceinline__ void square_group(int len, uint32_t (&x0)[NT], uint32_t (&x1)[NT],
                                             const uint32_t (&m0)[NT], const uint32_t (&m1)[NT],
                                             const uint32_t (&mp)[NT], const uint32_t (&sh)[NT]) {
  const uint32_t zero[NT] = {};
  switch (len) {
    case 4: square_all<PATH, NT>(x0, x1, m0, m1, mp, zero, false);  // fall through
    case 3: square_all<PATH, NT>(x0, x1, m0, m1, mp, zero, false);  // fall through
    case 2: square_all<PATH, NT>(x0, x1, m0, m1, mp, zero, false);  // fall through
    default: break;
  }
  square_all<PATH, NT>(x0, x1, m0, m1, mp, sh, true);
}

// Ladders of path 1 for parts of its and path 2's moduli (two words, three-word square).
enum Ladder {
  kLadderPlain,
  // Moduli up to kHalfMaxModulus: every second squaring takes one reduction step
  // (sqr_half64_p1).  All factors are powers of two, so a value is followed by its exponent
  // f: a squaring with two steps and a window shift s takes f to 2 f - 64 + s, one with a
  // step to 2 f - 32, the two together to 4 f - 128 + s.  After c plain squarings from
  // R 2^w0 (f = 64 + w0) and k pairs, f = 4^k f1 - 128 (4^k - 1) / 3 + S with
  // f1 = 64 + (w0 and c bits), so f1 and S are the top and the low 2 k bits of
  // U = E + 128 (4^k - 1) / 3.  k is the largest with f1 >= 64.
  // (n = 1e12, 40-bit moduli: 36 squarings with 72 steps -> 35 with 53; a slice of 2e8
  // terms 8.13 -> 7.35 ms.)
  kLadderHalf,
  // Moduli of 47 bits: a squaring without shift leaves x < m + 2^31, one with a shift of 15
  // x < m + 2^46.3 < 2^47.7, and that x's square still fits three words, its first reduction
  // two.  Only the unreduced first window may leave more, so it is reduced fully.
  // (n = 1e14, a slice of 2e8 terms: 10.8 ms on path 2, 9.0 here.)
  kLadder47
};

// One warp tile: terms [ti * tile, (ti + 1) * tile) of the run list of A, added
// into this lane's sum.  Every lane of the warp must call it (warp-wide reductions).
template <int LMAX, int PATH, int S, Ladder LADDER = kLadderPlain>
__device__ __forceinline__ void process_tile(const HeadArgs& A, const uint64_t ti, const uint32_t lane,
                                             uint32_t (&acc)[LMAX]) {
  constexpr int NT = 2 * S;
  constexpr bool WIDE = PathTraits<PATH>::kWide;
  constexpr int RB = PathTraits<PATH>::kRBits;
  const uint64_t run = A.run;
  const uint64_t tile = 32ull * S * run;
  const uint64_t last = A.count - 1;
  const int window = static_cast<int>(A.window);
  // exponent of the residue at k: E(k) = e0 - step k
  const uint64_t e0 = A.d + static_cast<int64_t>(A.c) + A.W;
  uint64_t base[S];
  StreamState st[S];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    base[s] = ti * tile + (static_cast<uint64_t>(lane) * S + s) * run;
    st[s].rel = min(base[s], last);
    const uint64_t k = A.k_begin + st[s].rel;
    st[s].m = static_cast<uint64_t>(A.a) * k + A.b;
    st[s].E = e0 - static_cast<uint64_t>(A.step) * k;
    st[s].tr = r_mod_m_bitserial<RB>(st[s].m);
  }
  for (uint32_t i = 0; i < run; i += 2) {
    uint64_t v[NT];
    uint32_t x0[NT], x1[NT], m0[NT], m1[NT], mp[NT];
    bool valid[NT];
    int nbl = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) {
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const int t = 2 * s + p;
        const uint64_t rel = base[s] + i + p;
        valid[t] = rel < A.count;
        if (valid[t] && rel != st[s].rel) {  // the next k of the run: advance by one
          st[s].rel = rel;
          st[s].m += A.a;
          st[s].E -= A.step;
          r_mod_m_advance<RB>(st[s].tr, st[s].m, A.a);
        }
        x0[t] = lo32(st[s].tr.r);
        x1[t] = hi32(st[s].tr.r);
        m0[t] = lo32(st[s].m);
        m1[t] = hi32(st[s].m);
        mp[t] = neg_inverse32(m0[t]);
        if (!WIDE) m1[t] = 0u - mp[t];  // no high word: the inverse itself
        v[t] = st[s].E - RB;  // E >= W >= RB for head terms
        nbl = max(nbl, bitlen64(v[t]));
      }
    }
    if constexpr (LADDER == kLadderHalf) {
      // the warp's largest and smallest exponents: first lane's first term, last lane's last
      const uint64_t e_max = __shfl_sync(0xffffffffu, v[0], 0) + RB;
      const uint64_t e_min = __shfl_sync(0xffffffffu, v[NT - 1], 31) + RB;
      const int k = (bitlen64((3 * e_min - 128) >> 6) - 1) / 2;  // 64 4^k <= 3 E - 128
      const uint64_t low = (1ull << (2 * k)) - 1ull, off = (0x5555555555555555ull & low) << 7;
      int c = 1;
      while ((((e_max + off) >> (2 * k)) - 64) >> c > A.first_max) ++c;
      uint64_t rem[NT];
      uint32_t sh[NT];
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        const uint64_t u = v[t] + RB + off;
        const uint32_t f1 = static_cast<uint32_t>(u >> (2 * k)) - 64u;
        const uint64_t x = make64(x0[t], x1[t]) << (f1 >> c);
        x0[t] = lo32(x);
        x1[t] = hi32(x);
        rem[t] = (static_cast<uint64_t>(f1 & ((1u << c) - 1u)) << (2 * k)) | (u & low);
      }
      // the c bits of f1, the first on the general routine
      int p = 2 * k + c - 1;
#pragma unroll
      for (int t = 0; t < NT; ++t) sh[t] = static_cast<uint32_t>(rem[t] >> p) & 1u;
      square_all_general<NT>(x0, x1, m0, m1, mp, sh, true);
      while (p > 2 * k) {
        --p;
#pragma unroll
        for (int t = 0; t < NT; ++t) sh[t] = static_cast<uint32_t>(rem[t] >> p) & 1u;
        square_all<PATH, NT>(x0, x1, m0, m1, mp, sh, true);
      }
      reduce_all<NT>(x0, x1, m0, m1, mp);
      while (p > 0) {
        p -= 2;
#pragma unroll
        for (int t = 0; t < NT; ++t) sh[t] = static_cast<uint32_t>(rem[t] >> p) & 3u;
#pragma unroll
        for (int t = 0; t < NT; ++t) sqr_half64_p1(x0[t], x1[t], Mod64{m0[t], m1[t], mp[t]});
        square_all<PATH, NT>(x0, x1, m0, m1, mp, sh, true);
      }
    } else {
    const int nb = static_cast<int>(__reduce_max_sync(0xffffffffu, static_cast<uint32_t>(nbl)));
    int h = nb > 0 ? min(static_cast<int>(A.first), nb - 1) : 0;
    if (A.first_max >= (1u << h) && h + 1 <= nb - 1) {
      // one more first-window bit (one squaring fewer) when the warp's top h + 1
      // exponent bits all stay within the first-window bound of the moduli (the
      // lane with nb bits has top bits >= 2^h, so a smaller bound never admits it)
      uint32_t top = 0;
#pragma unroll
      for (int t = 0; t < NT; ++t) top = max(top, static_cast<uint32_t>(v[t] >> (nb - h - 1)));
      if (__reduce_max_sync(0xffffffffu, top) <= A.first_max) ++h;
    }
    const int low = nb - h;  // bits left after the first window
    uint64_t rem[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      // first window: Montgomery form of 2^w0 is (R mod m) << w0, no squaring
      const uint32_t w0 = h > 0 ? static_cast<uint32_t>(v[t] >> low) : 0u;
      if (WIDE) {
        const uint64_t x = make64(x0[t], x1[t]) << w0;
        x0[t] = lo32(x);
        x1[t] = hi32(x);
      } else {
        x0[t] <<= w0;
      }
      rem[t] = low > 0 ? (v[t] & ((1ull << low) - 1ull)) : 0ull;
    }
    // remaining bits, top down, in groups of at most `window` bits.  Any split of the
    // bits into consecutive groups gives the same power.  Path 1 always has 4-bit
    // windows (its moduli are below 2^47); there the groups are aligned from the
    // bottom, so only the first one is short and the rest run as a fixed
    // four-squaring body.  The other paths align them from the top.
    int p = low;
    const bool w4 = PATH == 1 && window == 4;
    if (PATH == 1 && p > 0) {
      // the first group, with its first squaring on the general routine
      const int len = w4 ? ((p - 1) & 3) + 1 : min(window, p);
      p -= len;
      uint32_t sh[NT];
      const uint32_t zero[NT] = {};
#pragma unroll
      for (int t = 0; t < NT; ++t) sh[t] = static_cast<uint32_t>(rem[t] >> p) & ((1u << len) - 1u);
      if (len == 1) {
        square_all_general<NT>(x0, x1, m0, m1, mp, sh, true);
        if constexpr (LADDER == kLadder47) reduce_all<NT>(x0, x1, m0, m1, mp);
      } else {
        square_all_general<NT>(x0, x1, m0, m1, mp, zero, false);
        if constexpr (LADDER == kLadder47) reduce_all<NT>(x0, x1, m0, m1, mp);
        square_group<PATH, NT>(len - 1, x0, x1, m0, m1, mp, sh);
      }
    }
    if (w4) {
      const uint32_t zero[NT] = {};
      while (p > 0) {
        p -= 4;
        uint32_t sh[NT];
#pragma unroll
        for (int t = 0; t < NT; ++t) sh[t] = static_cast<uint32_t>(rem[t] >> p) & 15u;
        square_all<PATH, NT>(x0, x1, m0, m1, mp, zero, false);
        square_all<PATH, NT>(x0, x1, m0, m1, mp, zero, false);
        square_all<PATH, NT>(x0, x1, m0, m1, mp, zero, false);
        square_all<PATH, NT>(x0, x1, m0, m1, mp, sh, true);
      }
    }
    while (p > 0) {
      const int len = min(window, p);
      p -= len;
      uint32_t sh[NT];
#pragma unroll
      for (int t = 0; t < NT; ++t) sh[t] = static_cast<uint32_t>(rem[t] >> p) & ((1u << len) - 1u);
      square_group<PATH, NT>(len, x0, x1, m0, m1, mp, sh);
    }
    }
    // s = 2^E mod m (0 for a lane past the range), then the W-bit quotient digits
    // folded into the signed sum
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      if (WIDE) {
        reduce_once64(x0[t], x1[t], Mod64{m0[t], m1[t], mp[t]});
      } else if (x0[t] >= m0[t]) {
        x0[t] -= m0[t];
      }
      if (!valid[t]) {
        x0[t] = 0;
        x1[t] = 0;
      }
    }
    if (A.alternating) fold_digits<WIDE, true, NT, LMAX>(acc, x0, x1, m0, m1, mp);
    else fold_digits<WIDE, false, NT, LMAX>(acc, x0, x1, m0, m1, mp);
  }
}

// acc <- -acc mod 2^(32 LMAX)
template <int LMAX>
__device__ __forceinline__ void negate_limbs(uint32_t (&acc)[LMAX]) {
  uint64_t carry = 1;
#pragma unroll
  for (int i = 0; i < LMAX; ++i) {
    const uint64_t s = static_cast<uint64_t>(~acc[i]) + carry;
    acc[i] = static_cast<uint32_t>(s);
    carry = s >> 32;
  }
}

// Sums every thread's LMAX-limb value over the CTA and adds it to the carry-save slots.
template <int LMAX>
__device__ __forceinline__ void flush_cta(uint32_t (&acc)[LMAX], uint32_t L, unsigned long long* slots) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t wid = threadIdx.x >> 5;
  // limbs at or above L hold digits past 2^W: drop them (the sum is mod 2^W)
#pragma unroll
  for (int i = 0; i < LMAX; ++i)
    if (i >= static_cast<int>(L)) acc[i] = 0;
  __shared__ uint32_t red[kHeadThreads / 32][LMAX];
  warp_sum_limbs<LMAX>(acc);
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < LMAX; ++i) red[wid][i] = acc[i];
  }
  __syncthreads();
  if (wid == 0) {
    const uint32_t nw = blockDim.x >> 5;
#pragma unroll
    for (int i = 0; i < LMAX; ++i) acc[i] = lane < nw ? red[lane][i] : 0u;
    warp_sum_limbs<LMAX>(acc);
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < LMAX; ++i)
        if (i < static_cast<int>(L) && acc[i]) atomicAdd(slots + i, static_cast<unsigned long long>(acc[i]));
    }
  }
}

// The half-reduced ladder with two term pairs a thread is held to 80 registers, three CTAs
// an SM (7.35 against 7.58 ms on its slice).  GATED: nothing is done when *A.gate is 0.  The
// test is a template's because its early return costs the ladders up to 2 % by what the
// compiler then makes of them (P = 128, 41-bit moduli, 1e8 terms: 4.71 ms without, 4.79 with),
// or saves as much; launch_head (bbp_inst.cuh) takes the faster one.
template <int LMAX, int PATH, int S, Ladder LADDER = kLadderPlain, bool GATED = false>
__global__ void __launch_bounds__(kHeadThreads, LADDER == kLadderHalf && S == 2 && LMAX <= 16 ? 3 : 0)
head_kernel(const HeadArgs A, const uint64_t ntiles) {
  if (GATED && A.gate && *A.gate == 0u) return;
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t warp = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = (static_cast<uint64_t>(gridDim.x) * blockDim.x) >> 5;

  uint32_t acc[LMAX];
#pragma unroll
  for (int i = 0; i < LMAX; ++i) acc[i] = 0;
  for (uint64_t ti = warp; ti < ntiles; ti += nwarps) process_tile<LMAX, PATH, S, LADDER>(A, ti, lane, acc);

  if (A.negate) negate_limbs<LMAX>(acc);
  flush_cta<LMAX>(acc, A.L, A.slots);
}

// A small query in one launch: the tiles of all head ranges laid end to end, the tail
// terms in CTAs of their own, and the result by the CTA that finishes last.  Launches are
// what such a query is made of: n = 1e6 took nine (zeroing, seven ranges, tails, result)
// and two copies, 82 us; one launch and a result in pinned memory take 40.
template <int LMAX, int S>
__global__ void __launch_bounds__(kHeadThreads) query_kernel(const __grid_constant__ QuerySet Q) {
  if (blockIdx.x < Q.tail_blocks) {
    add_tail_term(Q.tails, static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x);
  } else {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t warp = ((blockIdx.x - Q.tail_blocks) * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = ((gridDim.x - Q.tail_blocks) * blockDim.x) >> 5;
    uint32_t acc[LMAX];
#pragma unroll
    for (int i = 0; i < LMAX; ++i) acc[i] = 0;
    uint32_t r = 0, negated = 0;  // acc holds the sum, negated or not
    for (uint64_t t = warp; t < Q.start[Q.n]; t += nwarps) {
      while (t >= Q.start[r + 1]) ++r;
      if (Q.head[r].negate != negated) {
        negate_limbs<LMAX>(acc);
        negated ^= 1u;
      }
      process_tile<LMAX, 0, S>(Q.head[r], t - Q.start[r], lane, acc);
    }
    if (negated) negate_limbs<LMAX>(acc);
    flush_cta<LMAX>(acc, Q.L, Q.slots);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0 && atomicAdd(Q.finished, 1u) + 1u == gridDim.x) {
    __threadfence();
    finalize_into(Q.slots, static_cast<int>(Q.L), Q.P, Q.bound, Q.out, Q.valid, Q.limbs);
  }
}

// ---------------------------------------------------------------- persistent queue

// The job of tile t (tiles of the group's jobs laid end to end): the last j in [lo, hi)
// with job_start[j] <= t, 33 ways at a time.  All lanes get it.
__device__ __forceinline__ uint32_t job_of_tile(const uint64_t* job_start, uint32_t lo, uint32_t hi, uint64_t t,
                                                uint32_t lane) {
  while (hi - lo > 1) {
    const uint32_t step = (hi - lo + 32) / 33;
    const uint32_t at = lo + min(hi - lo, (lane + 1) * step);
    const uint32_t below = __popc(__ballot_sync(0xffffffffu, at < hi && job_start[at] <= t));
    const uint32_t next = lo + (below + 1) * step;
    lo += below * step;
    hi = min(hi, next);
  }
  return lo;
}

template <int LMAX, int PATH, int S>
__global__ void __launch_bounds__(kHeadThreads) queue_kernel(const BatchDev B, const uint32_t job_begin,
                                                             const uint32_t job_end, unsigned long long* cursor) {
  const uint32_t lane = threadIdx.x & 31u;
  // the warp's current job lives in shared memory (like kernel arguments, it is
  // read-only and uniform, so it need not occupy registers)
  __shared__ HeadArgs job_sm[kHeadThreads / 32];
  HeadArgs& A = job_sm[threadIdx.x >> 5];
  // One counter hands out the tiles of all jobs: a warp whose tiles end a job goes on in the
  // next.  (A counter per job, with a cursor moved past exhausted ones, cost about 2.5 us a job
  // in contention: 3.0 ms for the 1200 jobs of 55 small queries, whatever their work.)  Every
  // hand-out ends, nothing waits on other threads.
  const uint64_t base = B.job_start[job_begin], total = B.job_start[job_end] - base;
  uint64_t t = 0, end = 0;  // the warp's tiles, [t, end)
  uint32_t j = job_begin;
  for (;;) {
    if (t == end) {
      unsigned long long at = 0;
      if (lane == 0) at = atomicAdd(cursor, static_cast<unsigned long long>(B.grab));
      t = __shfl_sync(0xffffffffu, at, 0);
      if (t >= total) break;
      end = min(t + B.grab, total);
      j = job_of_tile(B.job_start, j, job_end, base + t, lane);  // tiles come in ascending order
    } else {
      ++j;
    }
    static_assert(sizeof(HeadArgs) % 4 == 0, "HeadArgs is copied as 32-bit words");
    {
      const uint32_t* src = reinterpret_cast<const uint32_t*>(B.jobs + j);
      uint32_t* dst = reinterpret_cast<uint32_t*>(&A);
      for (uint32_t w = lane; w < sizeof(HeadArgs) / 4; w += 32) dst[w] = src[w];
      __syncwarp();
    }
    const uint64_t first = B.job_start[j] - base, ntiles = B.job_start[j + 1] - base - first;
    const uint64_t t0 = t - first, t1 = min(end - first, ntiles);
    t = first + t1;
    uint32_t acc[LMAX];
#pragma unroll
    for (int i = 0; i < LMAX; ++i) acc[i] = 0;
    for (uint64_t ti = t0; ti < t1; ++ti) process_tile<LMAX, PATH, S>(A, ti, lane, acc);
#pragma unroll
    for (int i = 0; i < LMAX; ++i)
      if (i >= static_cast<int>(A.L)) acc[i] = 0;
    warp_sum_limbs<LMAX>(acc);
    if (lane == 0) {
      if (A.negate) negate_limbs<LMAX>(acc);
#pragma unroll
      for (int i = 0; i < LMAX; ++i)
        if (i < static_cast<int>(A.L) && acc[i]) atomicAdd(A.slots + i, static_cast<unsigned long long>(acc[i]));
      __threadfence();
      const uint64_t done = atomicAdd(B.job_done + j, static_cast<unsigned long long>(t1 - t0)) + (t1 - t0);
      if (done == ntiles) retire_job(B, B.job_query[j]);
    }
    __syncwarp();
  }
}

}  // namespace bbp
