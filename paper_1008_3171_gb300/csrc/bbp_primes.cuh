// Kernels of the prime form of a query's head sum (bbp_primes.h says what is summed),
// templates over the accumulator class.  Three kernels cover the prime powers:
//
//   prime_kernel       primes above A / 23: H is one of a few rational constants, so a
//                      prime costs one modular power of 2, a product and W bits of quotient
//   prime_sum_kernel   primes below, down to sqrt(A): H summed mod p, 1, 8 or 32 threads each
//   prime_power_kernel primes up to sqrt(A) and prime powers: one warp each
//
// Every part is a residue x = 2^W r mod q of a fraction r / q; its W bits are the
// exact-division digits of -x / q, as for a term (bbp_device.cuh).  Each is rounded
// down, so the sum errs by less than one unit per part -- fewer parts than terms.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "bbp_device.cuh"
#include "bbp_kernels.cuh"
#include "bbp_primes.h"
#include "bbp_tile.cuh"

namespace bbp {

// ---------------------------------------------------------------- primes above A / 23

// One prime's residue from the ladder.  Every factor in it is a power of two, so a value
// is followed by its exponent f alone: start at x = 2^f with f = t in [0, l) (below 2 p, no
// reduction), and each squaring with a reduction by 2^r and a window shift s takes f to
// 2 f - r + s.  After j squarings f = t 2^j + S - OFF, S collecting the shifts (j bits) and
// OFF the reductions, and this has to be e mod p - 1.  So t and S are the top and the low
// j bits of u = e + OFF mod (p - 1), taken in the window [l 2^j - (p - 1), l 2^j): j = l - 5
// (two words) or l - 4 (one word) makes l 2^j >= p - 1.  l is the warp's largest bit
// length; no 2^64 mod p is needed, and the first five bits cost no squaring.
//
// `off` is OFF - l 2^j, `p1` is p - 1.
__device__ __forceinline__ uint64_t reduced_exponent(uint64_t e, int64_t off, uint64_t p1, uint64_t top) {
  const uint64_t a = e + static_cast<uint64_t>(off);
  // floor(a / (p - 1)), at most about 60: the single-precision quotient is off by at most one
  uint32_t q = static_cast<uint32_t>(__fdividef(static_cast<float>(a), static_cast<float>(p1)));
  int64_t rem = static_cast<int64_t>(a) - static_cast<int64_t>(q * p1);
  if (rem < 0) rem += static_cast<int64_t>(p1);
  if (rem >= static_cast<int64_t>(p1)) rem -= static_cast<int64_t>(p1);
  return static_cast<uint64_t>(rem) + top - p1;
}

__device__ __forceinline__ uint32_t redc_den(uint64_t t, const PrimeClass& C) {  // < den for t < den 2^32
  const uint32_t u = lo32(t) * C.neg_inv;
  const uint32_t r = hi32(t) + __umulhi(u, C.den) + (lo32(t) != 0u ? 1u : 0u);
  return min(r, r - C.den);
}

__device__ __forceinline__ uint32_t mul_den(uint32_t a, uint32_t b, const PrimeClass& C) {
  return redc_den(static_cast<uint64_t>(a) * b, C);
}

// v 2^32 mod den, v < 2^60
__device__ __forceinline__ uint32_t into_den(uint64_t v, const PrimeClass& C) {
  const uint32_t a = mul_den(lo32(v), C.r2, C) + mul_den(hi32(v), C.r3, C);
  return min(a, a - C.den);
}

// y / den mod p for y < p: (y + p t) / den with t = -y p^-1 mod den.  p^-1 is p^(lambda - 1):
// den has few prime factors, so lambda is at most 720.
__device__ __forceinline__ uint64_t divide_by_den(uint64_t y, uint64_t p, const PrimeClass& C) {
  const uint32_t pm = into_den(p, C);
  uint32_t inv = pm;
  for (int b = 30 - __clz(static_cast<int>(C.lambda)); b >= 0; --b) {
    inv = mul_den(inv, inv, C);
    if ((C.lambda >> b) & 1u) inv = mul_den(inv, pm, C);
  }
  uint32_t t = redc_den(mul_den(into_den(y, C), inv, C), C);  // y p^-1 mod den
  t = t != 0u ? C.den - t : 0u;
  return (y + p * t) * C.den_inv;  // exact, so the low 64 bits are enough
}

// HALF (two words, p below kPrimeHalfMax): the ladder alternates a squaring with one
// reduction step (r = 32) and one with two (r = 64) and a two-bit window.  With s <= 3 the
// second leaves x < p + 2^35, the first then x^2 / 2^32 + p < 2^48, whose square still
// fits three words.  A quarter of the reduction steps fall away: 25 multiply-pipe units for
// two squarings in the place of 30 (2.0e7 primes near 1e10: 775 -> 717 us).
template <int PATH, bool HALF, int NT>
__device__ __forceinline__ void prime_residues(const uint64_t e, const uint64_t (&p)[NT], const bool (&valid)[NT],
                                               const PrimeClass* classes, uint32_t (&x0)[NT], uint32_t (&x1)[NT],
                                               uint32_t (&m0)[NT], uint32_t (&m1)[NT], uint32_t (&mp)[NT]) {
  constexpr bool WIDE = PathTraits<PATH>::kWide;
  constexpr int RB = PathTraits<PATH>::kRBits;
  int l = 0;
#pragma unroll
  for (int t = 0; t < NT; ++t) l = max(l, bitlen64(p[t]));
  l = static_cast<int>(__reduce_max_sync(0xffffffffu, static_cast<uint32_t>(l)));
  const int j = WIDE ? l - 5 : l - 4;
  // OFF: RB (2^j - 1) with every reduction by RB; HALF: f -> 4 f - 128 + s for two squarings,
  // after one of f -> 2 f - 64 + s if j is odd
  const uint64_t two_j = 1ull << j;
  const uint64_t off = HALF ? (j & 1 ? 32 * two_j : 0) + 128 * (((two_j >> (j & 1)) - 1) / 3) : RB * (two_j - 1);
  const int64_t diff = static_cast<int64_t>(off) - static_cast<int64_t>(l * two_j);
  uint64_t rem[NT];
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    m0[t] = lo32(p[t]);
    m1[t] = hi32(p[t]);
    mp[t] = neg_inverse32(m0[t]);
    const uint64_t u = reduced_exponent(e, diff, p[t] - 1, l * two_j);
    const uint64_t x = 1ull << static_cast<uint32_t>(u >> j);
    x0[t] = lo32(x);
    x1[t] = hi32(x);
    rem[t] = u & (two_j - 1);
  }
  int b = j;
  if (HALF) {
    uint32_t sh[NT];
    if (b & 1) {
      --b;
#pragma unroll
      for (int t = 0; t < NT; ++t) sh[t] = static_cast<uint32_t>(rem[t] >> b);
      square_all<PATH, NT>(x0, x1, m0, m1, mp, sh, true);
    }
    while (b > 0) {
      b -= 2;
#pragma unroll
      for (int t = 0; t < NT; ++t) sh[t] = static_cast<uint32_t>(rem[t] >> b) & 3u;
#pragma unroll
      for (int t = 0; t < NT; ++t) sqr_half64_p1(x0[t], x1[t], Mod64{m0[t], m1[t], mp[t]});
      square_all<PATH, NT>(x0, x1, m0, m1, mp, sh, true);
    }
  } else if (WIDE) {
    // groups of four bits from the bottom; the first one is short
    const int len = ((b - 1) & 3) + 1;
    b -= len;
    uint32_t sh[NT];
    const uint32_t zero[NT] = {};
#pragma unroll
    for (int t = 0; t < NT; ++t) sh[t] = static_cast<uint32_t>(rem[t] >> b);
    square_group<PATH, NT>(len, x0, x1, m0, m1, mp, sh);
    while (b > 0) {
      b -= 4;
#pragma unroll
      for (int t = 0; t < NT; ++t) sh[t] = static_cast<uint32_t>(rem[t] >> b) & 15u;
      square_all<PATH, NT>(x0, x1, m0, m1, mp, zero, false);
      square_all<PATH, NT>(x0, x1, m0, m1, mp, zero, false);
      square_all<PATH, NT>(x0, x1, m0, m1, mp, zero, false);
      square_all<PATH, NT>(x0, x1, m0, m1, mp, sh, true);
    }
  } else {
    // One bit at a time, the bit taken as a doubled operand of the square: x (2 x) stays below
    // m 2^32 for a lazy x < 2 m of up to 29 bits (path 0) and a reduced x < m of up to 31 (path
    // 3).  The reduction subtracts (Arith1): one three-operand add after the high product.
    uint32_t bits[NT], inv[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      bits[t] = lo32(rem[t]);  // j <= 27
      inv[t] = 0u - mp[t];
    }
    while (b > 0) {
      --b;
      const uint32_t mask = 1u << b;
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        const uint64_t T = static_cast<uint64_t>(x0[t]) * ((bits[t] & mask) ? x0[t] + x0[t] : x0[t]);
        const uint32_t h = __umulhi(lo32(T) * inv[t], m0[t]);
        if (PATH == 3) {
          const uint32_t r = hi32(T) - h;  // in (-m, m)
          x0[t] = min(r, r + m0[t]);
        } else {
          x0[t] = hi32(T) + m0[t] - h;
        }
      }
    }
  }
  // times H, with p's sign
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    int c = 0;
    while (p[t] <= classes[c].above) ++c;
    const PrimeClass& C = classes[c];
    const uint32_t mod4 = (m0[t] >> 1) & 1u;  // 0: p = 1 mod 4, 1: p = 3
    const uint32_t n0 = lo32(C.num[mod4]), n1 = hi32(C.num[mod4]);
    uint64_t y;
    if (WIDE) {
      // x num / 2^64 mod p: x < 2 p < 2^47, num < 2^54, so the result is below 2 p (x = 2^(e + 64))
      const uint64_t a = static_cast<uint64_t>(x0[t]) * n0;
      const uint64_t b1 = static_cast<uint64_t>(x0[t]) * n1 + hi32(a);
      const uint64_t b2 = static_cast<uint64_t>(x1[t]) * n0 + lo32(b1);
      const uint64_t top = static_cast<uint64_t>(x1[t]) * n1 + hi32(b1) + hi32(b2);
      const uint64_t low = make64(lo32(a), lo32(b2));
      // low + u p = 0 mod 2^64, one word at a time
      uint32_t u = lo32(low) * mp[t];
      const uint64_t s1 = hi32(low) + static_cast<uint64_t>(__umulhi(u, m0[t])) + (lo32(low) != 0u ? 1u : 0u) +
                          static_cast<uint64_t>(u) * m1[t];
      u = lo32(s1) * mp[t];
      y = top + hi32(s1) + static_cast<uint64_t>(__umulhi(u, m0[t])) + (lo32(s1) != 0u ? 1u : 0u) +
          static_cast<uint64_t>(u) * m1[t];
    } else {
      const uint64_t a = static_cast<uint64_t>(x0[t]) * n0;
      const uint64_t b1 = static_cast<uint64_t>(x0[t]) * n1 + hi32(a);
      uint32_t u = lo32(a) * mp[t];
      const uint64_t s1 = b1 + __umulhi(u, m0[t]) + (lo32(a) != 0u ? 1u : 0u);
      u = lo32(s1) * mp[t];
      y = static_cast<uint64_t>(hi32(s1)) + __umulhi(u, m0[t]) + (lo32(s1) != 0u ? 1u : 0u);
    }
    if (y >= p[t]) y -= p[t];
    if (C.den > 1u) y = divide_by_den(y, p[t], C);
    if (((C.negative >> mod4) & 1u) && y != 0) y = p[t] - y;
    if (!valid[t]) y = 0;
    x0[t] = lo32(y);
    x1[t] = hi32(y);
  }
}

// Hands the next `n` primes of the list to the warp.
__device__ __forceinline__ uint32_t take_primes(uint32_t* taken, uint32_t n, uint32_t lane) {
  uint32_t at = 0;
  if (lane == 0) at = atomicAdd(taken, n);
  return __shfl_sync(0xffffffffu, at, 0);
}

// Primes per thread: independent chains that keep the multiply pipe fed at two CTAs an SM
// (n = 4e10, two words: 83.5 ms with four, 82.4 with five, 84.8 with six; one word: 1.745 ms
// at n = 1e9 with four, 1.751 with five).  With 16 or 24 accumulator limbs the fifth takes the
// registers that the sieve runs in (n = 1e10, P = 400 and 600: 21.2 and 22.7 ms with four, 21.4
// and 24.1 with five); with 40 there are none for it either way (P = 1000: 27.4, 26.7 ms).
template <int LMAX, int PATH>
constexpr int kPrimeNT = PathTraits<PATH>::kWide && (LMAX <= 10 || LMAX == 40) ? 5 : 4;

template <int LMAX, int PATH, bool HALF>
__global__ void __launch_bounds__(kHeadThreads) prime_kernel(const __grid_constant__ PrimeArgs A) {
  __shared__ PrimeClass classes[kMaxPrimeClasses];
  for (uint32_t i = threadIdx.x; i < A.nclasses * (sizeof(PrimeClass) / 4); i += blockDim.x)
    reinterpret_cast<uint32_t*>(classes)[i] = reinterpret_cast<const uint32_t*>(A.classes)[i];
  __syncthreads();
  constexpr int NT = kPrimeNT<LMAX, PATH>;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t count = min(*A.count, A.cap);
  uint32_t acc[LMAX];
#pragma unroll
  for (int i = 0; i < LMAX; ++i) acc[i] = 0;
  // warps take their primes as they come: other kernels share the SMs and delay some CTAs
  for (uint32_t at; (at = take_primes(A.taken, 32 * NT, lane)) < count;) {
    uint64_t p[NT];
    bool valid[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const uint32_t i = at + 32 * t + lane;
      valid[t] = i < count;
      p[t] = A.base + A.list[min(i, count - 1)];
    }
    uint32_t x0[NT], x1[NT], m0[NT], m1[NT], mp[NT];
    prime_residues<PATH, HALF, NT>(A.e, p, valid, classes, x0, x1, m0, m1, mp);
    fold_digits<PathTraits<PATH>::kWide, false, NT, LMAX>(acc, x0, x1, m0, m1, mp);
  }
  flush_cta<LMAX>(acc, A.L, A.slots);
}

// ---------------------------------------------------------------- sums mod p

// Residues mod m < 2^31 in one word.  Between operations a residue is below m; `lazy`
// ones are below 2 m.  t 2^-32 mod m is hi(t) - hi(u m) with u = lo(t) m^-1: the low
// words of t and u m are equal, so nothing carries and m - hi(u m) + hi(t) is one
// three-operand add.
struct Arith1 {
  using T = uint32_t;
  uint32_t m, mp, minv;  // mp = -m^-1, minv = m^-1 mod 2^32
  uint32_t r1;           // 2^32 mod m: 1 in Montgomery form
  __device__ explicit Arith1(uint64_t q)
      : m(lo32(q)), mp(neg_inverse32(lo32(q))), minv(0u - mp), r1(static_cast<uint32_t>(r_mod_m_bitserial<32>(q).r)) {}
  __device__ __forceinline__ T lazy_redc(uint64_t t) const {  // t 2^-32, t < m 2^32 (or below 2 m for hi(t) < m)
    return hi32(t) + m - __umulhi(lo32(t) * minv, m);
  }
  __device__ __forceinline__ T lazy_redc_neg(uint64_t t) const {  // -t 2^-32
    return __umulhi(lo32(t) * minv, m) + m - hi32(t);
  }
  __device__ __forceinline__ T fix(uint32_t r) const { return min(r, r - m); }  // r < 2 m
  __device__ __forceinline__ T redc(uint64_t t) const { return fix(lazy_redc(t)); }
  __device__ __forceinline__ T mul(T a, T b) const { return redc(static_cast<uint64_t>(a) * b); }
  __device__ __forceinline__ T add(T a, T b) const { return fix(a + b); }
  __device__ __forceinline__ T neg(T a) const { return a != 0u ? m - a : 0u; }
  __device__ __forceinline__ T one() const { return r1; }
  __device__ __forceinline__ T plain(T a) const { return redc(a); }  // out of Montgomery form
  __device__ __forceinline__ uint32_t digit(T& x) const {            // next exact-division digit
    const uint32_t q = x * mp;
    x = __umulhi(q, m) + (x != 0u ? 1u : 0u);
    return q;
  }
};

// Residues mod m < 2^46 in one 64-bit word, fully reduced.
struct Arith2 {
  using T = uint64_t;
  static constexpr int kBits = 64;
  uint64_t m, mp;
  uint64_t r1;  // 2^64 mod m
  __device__ explicit Arith2(uint64_t q) : m(q), r1(r_mod_m_bitserial<64>(q).r) {
    const uint64_t x = 0u - neg_inverse32(lo32(q));
    mp = 0ull - x * (2ull - q * x);
  }
  __device__ __forceinline__ T fix(uint64_t r) const { return r >= m ? r - m : r; }
  __device__ __forceinline__ T mul(T a, T b) const {
    const uint64_t lo = a * b;
    return fix(__umul64hi(a, b) + __umul64hi(lo * mp, m) + (lo != 0 ? 1u : 0u));
  }
  __device__ __forceinline__ T mul_word(T a, uint32_t c, T b) const {
    const uint64_t p0 = static_cast<uint64_t>(lo32(a)) * c;
    const uint64_t p1 = static_cast<uint64_t>(hi32(a)) * c;  // a < 2^46: below 2^46
    const uint64_t s0 = p0 + b;                              // 64 bits with a carry
    const uint64_t top = p1 + hi32(s0) + (s0 < p0 ? (1ull << 32) : 0ull);
    const uint32_t u = lo32(s0) * lo32(mp);
    return fix(top + __umulhi(u, lo32(m)) + (lo32(s0) != 0u ? 1u : 0u) + static_cast<uint64_t>(u) * hi32(m));
  }
  __device__ __forceinline__ T add(T a, T b) const { return fix(a + b); }
  __device__ __forceinline__ T neg(T a) const { return a != 0 ? m - a : 0; }
  __device__ __forceinline__ T one() const { return r1; }
  __device__ __forceinline__ T plain(T a) const { return mul(a, 1); }
  __device__ __forceinline__ uint32_t digit(T& x) const {
    uint32_t x0 = lo32(x), x1 = hi32(x);
    const uint32_t q = hensel_step64(x0, x1, Mod64{lo32(m), hi32(m), lo32(mp)});
    x = make64(x0, x1);
    return q;
  }
};

// a / p for the limits of the sums and primes from sqrt(A) on
template <int FORMULA>
__device__ __forceinline__ uint32_t small_quotient(uint64_t a, uint64_t p) {
  const float q = __fdividef(static_cast<float>(a), static_cast<float>(p));
  return corrected_quotient<FORMULA>(static_cast<uint32_t>(q), a, p);
}

// den^-1 2^e (Montgomery form) for a unit `den` mod m whose group of units has
// exponent phi: den^(phi - 1) and 2^e in one ladder.  0 <= e < phi.  In one word two bits
// at a time: the bits of e double an operand of the squares, those of phi - 1 choose
// among 1, den, den^2, den^3.  Every lane of the warp must call it.
template <class A>
__device__ typename A::T inverse_times_power(const A& M, typename A::T den, uint64_t phi, uint64_t e) {
  using T = typename A::T;
  const T one = M.one();
  T z = one;
  if constexpr (sizeof(T) == 4) {
    const uint32_t f = lo32(phi) - 1u, g = lo32(e);
    const T den2 = M.mul(den, den), den3 = M.mul(den2, den);
    const int bits = 32 - __clz(static_cast<int>(__reduce_max_sync(0xffffffffu, lo32(phi))));
    for (int b = (bits - 1) & ~1; b >= 0; b -= 2) {
      z = M.mul(z, (g >> (b + 1)) & 1u ? z + z : z);
      z = M.mul(z, (g >> b) & 1u ? z + z : z);
      const T lo = (f >> b) & 1u ? den : one, hi = (f >> b) & 1u ? den3 : den2;
      z = M.mul(z, (f >> (b + 1)) & 1u ? hi : lo);
    }
  } else {
    const uint64_t f = phi - 1;
    for (int b = bitlen64(phi) - 1; b >= 0; --b) {
      z = M.mul(z, z);
      if ((f >> b) & 1u) z = M.mul(z, den);
      if ((e >> b) & 1u) z = M.add(z, z);
    }
  }
  return z;
}

// 2^e in Montgomery form
template <class A>
__device__ typename A::T power_of_two(const A& M, uint64_t e) {
  typename A::T z = M.one();
  for (int b = bitlen64(e) - 1; b >= 0; --b) {
    z = M.mul(z, z);
    if ((e >> b) & 1u) z = M.add(z, z);
  }
  return z;
}

// e mod phi of a signed exponent
__device__ __forceinline__ uint64_t exponent_mod(int64_t e, uint64_t phi) {
  const int64_t r = e % static_cast<int64_t>(phi);
  return static_cast<uint64_t>(r < 0 ? r + static_cast<int64_t>(phi) : r);
}

// The sums mod p, three of each formula: the term at i is s(i) w^-i / c, c = stride i + c0, with
// w a power of two for a prime p.
//
//   kind       w     c        s(i)
//   0 A      2^2    2 i + 1   (-1)^i
//   1 B      2^10   2 i + 1   (-1)^i
//   2 C      2^5    2 i + 1   + + - -
//   3 D      2^2    4 i + c0  (-1)^i   c0 = p mod 4
//   4 E      2^4    4 i + c0  +        c0 = 4 - p mod 4
//   5 F      2^4    2 i + 1   +
template <int KIND>
struct SumKind {
  static constexpr uint32_t kW = KIND == 1 ? 10u : KIND == 2 ? 5u : KIND >= 4 ? 4u : 2u;  // log2 w
  static constexpr uint32_t kStride = KIND == 3 || KIND == 4 ? 4u : 2u;
  static constexpr bool kAlternates = KIND == 0 || KIND == 1 || KIND == 3;
  static constexpr bool kInTwos = KIND == 2;  // the signs + + - -
  // two terms at once while w^2 c (c - stride) <= 2^31, which keeps every product below m 2^32
  static constexpr uint32_t kPairTop = KIND == 0 || KIND == 3 ? 11583u : KIND == 2 ? 1447u : KIND >= 4 ? 2896u : 0u;

  // Whether den changes sign after term i (s(i - 1) is not s(i)).
  __device__ static __forceinline__ bool flips(uint32_t i) { return kAlternates || (kInTwos && (i & 1u) == 0u); }
  // s(i) of the last term, times the sign that den has collected over [lo, hi): num's sign.
  __device__ static __forceinline__ bool negative(uint32_t lo, uint32_t hi) {
    if (kAlternates) return ((hi - lo) ^ (hi - 1u)) & 1u;
    if (kInTwos) return (((hi + 1u) / 2u - (lo + 1u) / 2u) ^ ((hi - 1u) >> 1)) & 1u;
    return false;
  }
};

// One term, from the last down: num <- c num + den, den <- w c den, with s carried in den's
// sign (den <- -w c den where s changes), so a step is two products by a word, two
// reductions and no selection; each reduction leaves the same factor 2^-32 in both.
template <int KIND>
__device__ __forceinline__ void sum_step(const Arith1& M, uint32_t i, uint32_t c, uint32_t& N, uint32_t& D) {
  using K = SumKind<KIND>;
  N = M.lazy_redc(static_cast<uint64_t>(N) * c + D);
  const uint64_t t = static_cast<uint64_t>(D) * (c << K::kW);
  if (K::kInTwos) {
    const uint32_t r = M.lazy_redc(t);
    D = (i & 1u) ? r : 2u * M.m - r;
  } else {
    D = K::kAlternates ? M.lazy_redc_neg(t) : M.lazy_redc(t);
  }
}

// Two terms, i odd at c and i - 1 at c' = c - stride: three products serve both.
//   signs alternate:  num <- c c' num - (w c - c') den, den <- w^2 c c' den   (d = -den)
//   + +, then - -:    num <- c c' num + (w c + c') den, den <- -w^2 c c' den
//   no change:        num <- c c' num + (w c + c') den, den <- w^2 c c' den
template <int KIND>
__device__ __forceinline__ void sum_pair(const Arith1& M, uint32_t c, uint32_t& N, uint32_t& d) {
  using K = SumKind<KIND>;
  const uint32_t c2 = c - K::kStride, alpha = c * c2;
  const uint32_t beta = K::kAlternates ? (c << K::kW) - c2 : (c << K::kW) + c2;
  N = M.lazy_redc(static_cast<uint64_t>(N) * alpha + static_cast<uint64_t>(d) * beta);
  const uint64_t t = static_cast<uint64_t>(d) * (alpha << (2u * K::kW));
  d = K::kInTwos ? M.lazy_redc_neg(t) : M.lazy_redc(t);
}

// Where a lane starts among the pairs: nothing done yet, or its last term done if that
// is the first of a pair.
template <int KIND>
__device__ __forceinline__ void pair_start(const Arith1& M, uint32_t hi, uint32_t c0, uint32_t& N, uint32_t& D) {
  using K = SumKind<KIND>;
  N = 0;
  D = 1;
  if (hi & 1u) {
    const uint64_t wc = static_cast<uint64_t>(K::kStride * (hi - 1u) + c0) << K::kW;
    N = M.lazy_redc(1u);
    D = K::kAlternates || K::kInTwos ? M.lazy_redc_neg(wc) : M.lazy_redc(wc);
  }
}

template <int KIND>
__device__ __forceinline__ uint32_t pair_sign(const Arith1& M, uint32_t d) {  // den <-> the pairs' d
  return SumKind<KIND>::kAlternates ? 2u * M.m - d : d;
}

// Fractions of primes p < 2^31, one a lane: the sum over 0 <= i < n of s(i) w^-i / c as
// w num / den.  Every lane of the warp must call it.
//
// The lanes of a warp walk i together from the largest n, so no lane waits for another's
// loop (and c is uniform where c0 is 1); until its own n a lane keeps num = den = 0 mod p.
// In multiply-pipe units (low half 1, high half or full product 2) a term costs 10 singly
// and 6.3 in pairs.  (One term at a time, every lane with its own loop: the primes up to
// A / 23 of n = 4e10 took 16.9 ms, now 10.)
template <int KIND>
__device__ __forceinline__ void prime_sum(const Arith1& M, uint32_t n, uint32_t c0, uint32_t& num, uint32_t& den) {
  using K = SumKind<KIND>;
  const uint32_t top = __reduce_max_sync(0xffffffffu, n);
  const uint32_t first = K::kStride == 2u ? 1u : c0;
  uint32_t N = 0, D = 0;
  uint32_t i = top;
  while (i > 0 && (K::kPairTop == 0 || K::kStride * i > K::kPairTop || (i & 1u))) {
    if (i == n) {
      N = 0;
      D = 1;
    }
    --i;
    sum_step<KIND>(M, i, K::kStride * i + first, N, D);
  }
  if (K::kPairTop != 0 && i > 0) {
    if (n < i) {
      N = 0;
      D = 0;
    }
    uint32_t n0, d0;
    pair_start<KIND>(M, n, first, n0, d0);
    const uint32_t start = n >> 1, d_start = pair_sign<KIND>(M, d0);
    uint32_t d = pair_sign<KIND>(M, D);
    const bool late = n <= i;  // starts within the pairs
    // down to where every lane has started, then without looking
    const uint32_t all = min(i / 2u, __reduce_min_sync(0xffffffffu, start));
    uint32_t h = i / 2;
    for (; h > all; --h) {
      if (late && h == start) {
        N = n0;
        d = d_start;
      }
      sum_pair<KIND>(M, K::kStride * (2u * h - 1u) + first, N, d);
    }
    if (late && h == start) {
      N = n0;
      d = d_start;
    }
    uint32_t c = K::kStride * (2u * h - 1u) + first;
    for (; h > 0; --h) {
      sum_pair<KIND>(M, c, N, d);
      c -= 2u * K::kStride;
    }
    D = pair_sign<KIND>(M, d);
    if (late && start == 0u) {  // n = 1 (or none): no pair
      N = n0;
      D = d0;
    }
  } else if (n == 0) {
    N = 0;
    D = 1;
  }
  num = M.fix(N);
  den = M.fix(D);
  if (n != 0 && K::negative(0, n)) num = M.neg(num);
}

// The same over lo <= i < hi, relative to the term at lo (w num / den with w^-(i - lo)), lo
// even, each lane with its own range; the lanes walk them in step, and none looks for its
// start once all have started.
template <int KIND>
__device__ __forceinline__ void range_sum(const Arith1& M, uint32_t lo, uint32_t hi, uint32_t c0, uint32_t& num,
                                          uint32_t& den) {
  using K = SumKind<KIND>;
  const uint32_t steps = __reduce_max_sync(0xffffffffu, hi - lo);
  const bool pairs = K::kPairTop != 0u && __reduce_max_sync(0xffffffffu, K::kStride * hi) <= K::kPairTop;
  const uint32_t first = K::kStride == 2u ? 1u : c0;
  uint32_t N = 0, D = 1;
  if (pairs) {
    uint32_t n0, d0;
    pair_start<KIND>(M, hi, first, n0, d0);
    const uint32_t d_start = pair_sign<KIND>(M, d0);
    uint32_t k = (steps + 1u) / 2u;
    uint32_t c = K::kStride * (2u * (lo / 2u + k) - 1u) + first, d = 1;
    const uint32_t mine = (hi - lo) / 2u, all = __reduce_min_sync(0xffffffffu, hi > lo ? mine : k);
    auto begin = [&] {
      if (k == mine) {
        N = n0;
        d = d_start;
      }
    };
    for (; k > all; --k) {
      begin();
      sum_pair<KIND>(M, c, N, d);
      c -= 2u * K::kStride;
    }
    begin();
    for (; k > 0u; --k) {
      sum_pair<KIND>(M, c, N, d);
      c -= 2u * K::kStride;
    }
    D = pair_sign<KIND>(M, d);
    if (mine == 0u) {  // one term, or none
      N = n0;
      D = d0;
    }
  } else {
    uint32_t k = steps, c = K::kStride * (lo + steps) + first;
    const uint32_t mine = hi - lo, all = __reduce_min_sync(0xffffffffu, hi > lo ? mine : k);
    auto begin = [&] {
      if (k == mine) {
        N = 0;
        D = 1;
      }
    };
    for (; k > all; --k) {
      begin();
      c -= K::kStride;
      sum_step<KIND>(M, lo + k - 1u, c, N, D);
    }
    begin();
    for (; k > 0u; --k) {
      c -= K::kStride;
      sum_step<KIND>(M, lo + k - 1u, c, N, D);
    }
  }
  if (hi <= lo) {
    N = 0;
    D = 1;
  }
  num = M.fix(N);
  den = M.fix(D);
  if (hi > lo && K::negative(lo, hi)) num = M.neg(num);
}

// The sum over 0 <= i < n shared by GROUP neighbouring lanes with the same prime: each takes
// about as many terms, an even number but for the last, and the fractions are put together
// two by two, w^s with the s terms of the lower one:
//   w num / den = w (num den' w^s + num' den) / (den den' w^s).
// The group's first lane has the result.
template <int KIND, int GROUP>
__device__ __forceinline__ void group_sum(const Arith1& M, uint32_t n, uint32_t c0, uint32_t& num, uint32_t& den) {
  const uint32_t g = threadIdx.x & (GROUP - 1), share = n / GROUP & ~1u;
  const uint32_t extra = (n & ~1u) - share * GROUP;  // even: two more for the first lanes
  const uint32_t lo = share * g + min(2u * g, extra);
  const uint32_t hi = g == GROUP - 1 ? n : lo + share + (2u * g < extra ? 2u : 0u);
  range_sum<KIND>(M, lo, hi, c0, num, den);
  uint32_t z = M.one(), e = SumKind<KIND>::kW * (hi - lo);  // w^s
  const int bits = 32 - __clz(static_cast<int>(__reduce_max_sync(0xffffffffu, e)));
  for (int b = bits - 1; b >= 0; --b) z = M.mul(z, (e >> b) & 1u ? z + z : z);
#pragma unroll
  for (int d = 1; d < GROUP; d <<= 1) {
    const uint32_t num2 = __shfl_down_sync(0xffffffffu, num, d, GROUP);
    const uint32_t den2 = __shfl_down_sync(0xffffffffu, den, d, GROUP);
    const uint32_t z2 = __shfl_down_sync(0xffffffffu, z, d, GROUP);
    num = M.add(M.mul(M.mul(num, z), den2), M.mul(den, num2));
    den = M.mul(M.mul(den, z), den2);
    z = M.mul(z, z2);
  }
}

// The largest c = s p at most `last` with c = c0 mod stride, 0 if there is none (p odd)
template <int KIND>
__device__ __forceinline__ uint64_t last_multiple(uint64_t last, uint64_t p, uint32_t c0) {
  constexpr uint32_t mask = SumKind<KIND>::kStride - 1u;
  const uint64_t s = last / p, s0 = (c0 * p) & mask;  // p^-1 = p mod 4
  return s < s0 ? 0 : (s - ((s - s0) & mask)) * p;
}

// The same over lo <= i < hi, relative to the term at lo (w num / den with w^-(i - lo)), the
// terms with c a multiple of p left out; the lanes walk their ranges in step.  WORD: modulo
// p, with w a word; else modulo a power of p, with h (a residue in Montgomery form) for w.
template <int KIND, bool WORD>
__device__ __forceinline__ void prime_share(const Arith1& M, uint32_t lo, uint32_t hi, uint32_t c0, uint32_t p,
                                            uint32_t h, uint32_t& num, uint32_t& den) {
  using K = SumKind<KIND>;
  const uint32_t steps = __reduce_max_sync(0xffffffffu, hi > lo ? hi - lo : 0u);
  const uint32_t first = K::kStride == 2u ? 1u : c0;
  uint32_t k = steps, N = 0, D = 1;
  uint32_t last = K::kStride * (lo + steps) + first;  // one stride above c
  uint32_t skip = hi > lo ? static_cast<uint32_t>(last_multiple<KIND>(K::kStride * (hi - 1u) + first, p, first)) : 0u;
  const uint32_t mine = hi > lo ? hi - lo : 0u, all = __reduce_min_sync(0xffffffffu, mine ? mine : k);
  auto begin = [&] {
    if (k == mine) {
      N = 0;
      D = 1;
    }
  };
  auto step = [&] {
    last -= K::kStride;
    uint32_t c = last, add = D;
    if (c == skip) {
      c = 1u;
      add = 0u;
      skip = skip > K::kStride * p ? skip - K::kStride * p : 0u;
    }
    N = M.lazy_redc(static_cast<uint64_t>(N) * c + add);
    const uint64_t t = WORD ? static_cast<uint64_t>(D) * (c << K::kW)
                            : static_cast<uint64_t>(M.lazy_redc(static_cast<uint64_t>(D) * c)) * h;
    if (K::kInTwos) {
      const uint32_t r = M.lazy_redc(t);
      D = ((lo + k - 1u) & 1u) ? r : 2u * M.m - r;
    } else {
      D = K::kAlternates ? M.lazy_redc_neg(t) : M.lazy_redc(t);
    }
  };
  for (; k > all; --k) {
    begin();
    step();
  }
  begin();
  for (; k > 0u; --k) step();
  if (hi <= lo) {
    N = 0;
    D = 1;
  }
  num = M.fix(N);
  den = M.fix(D);
  if (hi > lo && K::negative(lo, hi)) num = M.neg(num);
}

// The same modulo q < 2^46, one term at a time: WORD: q = p and h = w; else q = p^a and
// h = 2^(kW q) mod q in Montgomery form.
template <int KIND, bool WORD, bool SKIP>
__device__ __forceinline__ void power_sum(const Arith2& M, uint64_t i0, uint64_t i1, uint32_t c0, uint64_t p,
                                          uint64_t h, uint64_t& num, uint64_t& den) {
  using K = SumKind<KIND>;
  num = 0;
  den = 1;
  if (i0 >= i1) return;
  const uint32_t first = K::kStride == 2u ? 1u : c0;
  uint64_t skip = SKIP ? last_multiple<KIND>(K::kStride * (i1 - 1) + first, p, first) : 0;
  uint32_t i = static_cast<uint32_t>(i1);
  do {
    --i;
    const uint32_t c = K::kStride * i + first;
    uint32_t k = c;
    if (SKIP && c == static_cast<uint32_t>(skip)) {
      skip = skip > K::kStride * p ? skip - K::kStride * p : 0;
      k = 1u;
      num = M.mul_word(num, 1u, 0);
    } else {
      const bool minus = K::kAlternates ? (i & 1u) : K::kInTwos ? (i & 2u) : false;
      num = M.mul_word(num, c, minus ? M.neg(den) : den);
    }
    den = WORD ? M.mul_word(den, k * static_cast<uint32_t>(h), 0) : M.mul(M.mul_word(den, k, 0), h);
  } while (i > i0);
}

template <class A, int LMAX>
__device__ __forceinline__ void fold_one(const A& M, typename A::T x, uint32_t (&acc)[LMAX]) {
  uint32_t carry = 0;
#pragma unroll
  for (int i = 0; i < LMAX; ++i) {
    const uint64_t s = static_cast<uint64_t>(acc[i]) + M.digit(x) + carry;
    acc[i] = lo32(s);
    carry = hi32(s);
  }
}

// Terms with c = stride i + c0 up to `top`
template <int KIND, typename T>
__device__ __forceinline__ T summands(T top, uint32_t c0) {
  if (SumKind<KIND>::kStride == 2u) return (top + 1u) / 2u;
  return top >= c0 ? (top - c0) / 4u + 1u : 0u;
}

// GROUP lanes per prime: num / den of the formula's three sums, one ladder for the inverse
// of their denominators and the power of 2.
//   Eq. 2: H = 16 (num_A / den_A - 4 num_B / den_B - num_C / den_C), times chi(p)
//   Eq. 1: H = 8 (2 num_D / den_D - num_E / den_E - num_F / den_F) for p = 1 mod 4,
//          H = -8 (num_D / den_D + 4 num_E / den_E + num_F / den_F) for p = 3 mod 4
// One lane per prime would walk up to sqrt(A) / 2 terms in a row where the sums are long
// (n = 1e9: 600 us with the SM full, for 180 us of work): 32 lanes share a prime below
// A / 8000, eight one below A / 1000.
template <class A, int FORMULA, int GROUP, int LMAX>
__global__ void __launch_bounds__(kHeadThreads) prime_sum_kernel(const __grid_constant__ PrimeArgs G) {
  constexpr int K0 = FORMULA == 0 ? 0 : 3;
  const uint32_t count = min(*G.count, G.cap);
  uint32_t acc[LMAX];
#pragma unroll
  for (int i = 0; i < LMAX; ++i) acc[i] = 0;
  using T = typename A::T;
  const uint32_t lane = threadIdx.x & 31u;
  for (uint32_t at; (at = take_primes(G.taken, 32 / GROUP, lane)) < count;) {
    const uint32_t i = at + lane / GROUP;  // a lane past the end repeats the last prime and adds nothing
    const uint64_t p = G.base + G.list[min(i, count - 1)];
    const A M(p);
    const uint32_t r = lo32(p) & 3u;
    const uint32_t i0 = summands<K0>(small_quotient<FORMULA>(G.A, p), r), i1 = summands<K0 + 1>(small_quotient<FORMULA>(G.B, p), 4u - r),
                   i2 = summands<K0 + 2>(small_quotient<FORMULA>(G.C, p), 1u);
    T n0, d0, n1, d1, n2, d2;
    if constexpr (GROUP > 1) {
      group_sum<K0, GROUP>(M, i0, r, n0, d0);
      group_sum<K0 + 1, GROUP>(M, i1, 4u - r, n1, d1);
      group_sum<K0 + 2, GROUP>(M, i2, 1u, n2, d2);
    } else if constexpr (sizeof(T) == 4) {
      prime_sum<K0>(M, i0, r, n0, d0);
      prime_sum<K0 + 1>(M, i1, 4u - r, n1, d1);
      prime_sum<K0 + 2>(M, i2, 1u, n2, d2);
    } else {
      power_sum<K0, true, false>(M, 0, i0, r, p, 1u << SumKind<K0>::kW, n0, d0);
      power_sum<K0 + 1, true, false>(M, 0, i1, 4u - r, p, 1u << SumKind<K0 + 1>::kW, n1, d1);
      power_sum<K0 + 2, true, false>(M, 0, i2, 1u, p, 1u << SumKind<K0 + 2>::kW, n2, d2);
    }
    const T d12 = M.mul(d1, d2);
    T t0 = M.mul(n0, d12), t1 = M.mul(M.mul(n1, d0), d2);
    const T t2 = M.mul(M.mul(n2, d0), d1);
    if (FORMULA == 0 || r == 3u) {  // 4 times the second
      t1 = M.add(t1, t1);
      t1 = M.add(t1, t1);
    } else {
      t0 = M.add(t0, t0);
    }
    const T rest = M.add(t1, t2);
    // Eq. 2: chi(p) (t0 - rest); Eq. 1: t0 - rest or -(t0 + rest)
    T num = FORMULA == 0 || r == 1u ? M.add(t0, M.neg(rest)) : M.add(t0, rest);
    if (r == 3u) num = M.neg(num);
    const uint64_t e0 = G.e + (FORMULA == 0 ? 4 : 3);
    const uint64_t e = e0 - small_quotient<FORMULA>(e0, p - 1) * (p - 1);
    const T inv = inverse_times_power<A>(M, M.mul(d0, d12), p - 1, e);
    T x = M.plain(M.mul(num, inv));
    if (i >= count || (lane & (GROUP - 1)) != 0u) x = 0;
    fold_one<A, LMAX>(M, x, acc);
  }
  flush_cta<LMAX>(acc, G.L, G.slots);
}

// The sum over v < n of r^v, r in Montgomery form
template <class A>
__device__ typename A::T geometric(const A& M, typename A::T r, uint64_t n) {
  const typename A::T one = M.one();
  typename A::T s = 0, w = one;  // sum of the first k powers, r^k
  for (int b = bitlen64(n) - 1; b >= 0; --b) {
    s = M.add(s, M.mul(s, w));
    w = M.mul(w, w);
    if ((n >> b) & 1u) {
      s = M.add(M.mul(s, r), one);
      w = M.mul(w, r);
    }
  }
  return s;
}

// What one lane adds of sum KIND to the part of q = p^a: its share of the summands
// [lo, hi), times `factor`, as a fraction added to num / den (all in Montgomery form).
// Summand i carries s(i) 2^(start - ratio q i) / c; e is taken mod phi.
template <class A, int KIND, bool PRIME>
__device__ __forceinline__ void add_share(const A& M, uint64_t p, uint64_t q, uint64_t phi, int64_t e, uint64_t lo,
                                          uint64_t hi, typename A::T factor, uint32_t lane, typename A::T& num,
                                          typename A::T& den) {
  using T = typename A::T;
  using K = SumKind<KIND>;
  const uint64_t share = (hi - lo + 31) / 32;
  const uint64_t i0 = lo + min(hi - lo, lane * share), i1 = min(hi, i0 + share);
  if (hi <= lo) return;  // the same for every lane
  constexpr int64_t kRatio = K::kW;
  const int64_t sq = static_cast<int64_t>(PRIME ? 1 : q);  // 2^p = 2 mod p
  const uint32_t r4 = lo32(q) & 3u, c0 = KIND == 3 ? r4 : KIND == 4 ? 4u - r4 : 1u;
  T n_s, d_s;
  const T h = PRIME ? 0 : power_of_two<A>(M, exponent_mod(kRatio * sq, phi));
  if constexpr (sizeof(T) == 4)
    prime_share<KIND, PRIME>(M, static_cast<uint32_t>(i0), static_cast<uint32_t>(i1), c0, lo32(p), h, n_s, d_s);
  else
    power_sum<KIND, false, true>(M, i0, i1, c0, p, h, n_s, d_s);
  int64_t start = 0;
  bool minus = true;
  if (KIND == 0) start = e + 3 - sq, minus = (q & 2u) != 0;
  if (KIND == 1) start = e + 1 - 5 * sq, minus = (q & 2u) == 0;
  if (KIND == 2) start = e - 1 - 5 * (static_cast<int64_t>(q) - 1) / 2, minus = (q & 4u) == 0;
  if (KIND == 3) start = e + 2 - (static_cast<int64_t>(q) * c0 - 1) / 2, minus = ((q * c0) & 7u) != 1u;
  if (KIND == 4) start = e + 2 - sq * c0;
  if (KIND == 5) start = e + 1 - 2 * sq;
  // with the h that multiplies the fraction
  T k = power_of_two<A>(M, exponent_mod(start + kRatio * sq * (1 - static_cast<int64_t>(i0)), phi));
  k = M.mul(M.mul(k, factor), n_s);
  num = M.add(M.mul(num, d_s), M.mul(minus ? M.neg(k) : k, den));
  den = M.mul(den, d_s);
}

// Prime power of work item `unit`, 0 if there is none: for PRIME the primes in turn; else
// p^2 of every prime, then p^3 and p^4 of the first 3200 (p up to 29,000 > A^(1/3)), then
// p^5 ... p^28 of the first 128 (3^28 > A).
template <bool PRIME>
__device__ __forceinline__ uint64_t prime_power_of(const PrimeArgs& G, uint32_t unit, uint32_t count, uint64_t* p) {
  uint32_t i = unit, a = 2;
  if (!PRIME && unit >= count) {
    const uint32_t first = min(count, 3200u), second = min(count, 128u);
    i -= count;
    if (i < 2 * first) {
      a = 3 + i / first;
      i %= first;
    } else {
      i -= 2 * first;
      a = 5 + i / second;
      i %= second;
    }
  }
  *p = G.list[i];
  if (PRIME) return *p <= G.A ? *p : 0;
  uint64_t q = *p;
  for (uint32_t k = 1; k < a; ++k) {
    if (q > G.A / *p) return 0;
    q *= *p;
  }
  return q;
}

// One warp per prime power q = p^a: PRIME: a = 1; else a >= 2 and q below (Arith1) or from
// (Arith2) 2^31 on.  The summands of each sum repeat with a constant
// ratio after `period` of them (c^-1 mod q after q, the signs after 1 or 4 times that), so at most `period` of them are added up, times a geometric sum: the lanes
// share them evenly, each lane's part being its own fraction over q.
template <class A, int FORMULA, bool PRIME, int LMAX>
__global__ void __launch_bounds__(kHeadThreads) prime_power_kernel(const __grid_constant__ PrimeArgs G) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t count = min(*G.count, G.cap);
  constexpr int K0 = FORMULA == 0 ? 0 : 3;
  const uint32_t units = PRIME ? count : count + 2 * min(count, 3200u) + 24 * min(count, 128u);
  using T = typename A::T;
  uint32_t acc[LMAX];
#pragma unroll
  for (int i = 0; i < LMAX; ++i) acc[i] = 0;
  for (uint32_t unit = warp; unit < units; unit += nwarps) {
    uint64_t p;
    const uint64_t q = prime_power_of<PRIME>(G, unit, count, &p);
    if (q == 0 || (!PRIME && (q < (1ull << 31)) != (sizeof(T) == 4))) continue;
    const A M(q);
    const uint64_t phi = PRIME ? p - 1 : q / p * (p - 1);
    const int64_t e = static_cast<int64_t>(G.e % phi);
    // lane s < 3 works out sum s's repetitions: n summands, `whole` periods of them and `rest`
    const uint32_t s = min(lane, 2u), r4 = lo32(q) & 3u;
    const uint64_t top = (s == 0 ? G.A : s == 1 ? G.B : G.C) / q;
    const uint64_t n = FORMULA == 0 || s == 2 ? summands<0>(top, 1u) : s == 0 ? summands<3>(top, r4) : summands<4>(top, 4u - r4);
    const uint64_t period_s = FORMULA == 0 && s == 2 ? 4 * q : q;
    const uint64_t whole_s = n / period_s, rest_s = n - whole_s * period_s;
    T once = M.one(), more = 0;  // the first `rest` summands count whole + 1 times, the others whole times
    const bool repeats = __any_sync(0xffffffffu, whole_s != 0);
    if (repeats) {
      const uint32_t ratio = s == 0 ? SumKind<K0>::kW : s == 1 ? SumKind<K0 + 1>::kW : SumKind<K0 + 2>::kW;
      const bool alternates = s == 0 ? SumKind<K0>::kAlternates : s == 1 && SumKind<K0 + 1>::kAlternates;
      // (where nothing repeats, q^2 may pass 64 bits: then `whole` is 0 and r is not used)
      const uint64_t turn = (PRIME ? 1 : q % phi) * (period_s % phi) % phi * ratio;
      T r = power_of_two<A>(M, exponent_mod(-static_cast<int64_t>(turn), phi));
      if (alternates) r = M.neg(r);  // the period is odd
      more = geometric<A>(M, r, whole_s);
      once = M.add(M.mul(more, r), M.one());
    }
    auto of = [&](auto v, int k) { return __shfl_sync(0xffffffffu, v, k); };
    for (int pass = 0; pass < (repeats ? 2 : 1); ++pass) {
      T num = 0, den = M.one();
      const bool f = pass == 0;
      const T factor = f ? once : more;
      const uint64_t lo = f ? 0 : rest_s, hi = f ? rest_s : whole_s ? period_s : rest_s;
      add_share<A, K0, PRIME>(M, p, q, phi, e, of(lo, 0), of(hi, 0), of(factor, 0), lane, num, den);
      add_share<A, K0 + 1, PRIME>(M, p, q, phi, e, of(lo, 1), of(hi, 1), of(factor, 1), lane, num, den);
      add_share<A, K0 + 2, PRIME>(M, p, q, phi, e, of(lo, 2), of(hi, 2), of(factor, 2), lane, num, den);
      const T x = M.plain(M.mul(num, inverse_times_power<A>(M, den, phi, 0)));  // every lane: warp-wide
      fold_one<A, LMAX>(M, x, acc);
    }
  }
  flush_cta<LMAX>(acc, G.L, G.slots);
}

}  // namespace bbp
