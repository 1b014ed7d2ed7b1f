// Kernels of the prime form of a query's head sum (bbp_primes.h says what is summed),
// templates over the accumulator class.  Three kernels cover the prime powers:
//
//   prime_kernel       primes above A / 23: H is one of a few rational constants, so a
//                      prime costs one modular power of 2, a product and W bits of quotient
//   prime_sum_kernel   primes below: H summed mod p, one prime per thread
//   prime_power_kernel primes and prime powers with long sums: one warp each
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

// One prime's residue from the ladder: the exponent is reduced into
//   V = e mod (p - 1) - (p - 1) - K,   K = (RB - l) 2^j,
// so that its top, t = (V >> j) + RB, lies in [0, l): 2^t is below 2 p, needs no
// reduction, and stands for 2^(t - RB) in Montgomery form.  The ladder then takes the
// remaining j = l - 5 (two words) or l - 4 (one word) bits: no R mod p is needed and
// the first five bits cost no squaring.  l is the warp's largest bit length;
// p - 1 <= l 2^j = K' keeps every V of the warp in the window.
template <int PATH>
__device__ __forceinline__ uint64_t reduced_exponent(uint64_t e, uint64_t p1, int l, int j) {
  constexpr int RB = PathTraits<PATH>::kRBits;
  const uint64_t a = e + (static_cast<uint64_t>(RB - l) << j);
  // floor(a / (p - 1)), at most about 60: the single-precision quotient is off by at most one
  uint32_t q = static_cast<uint32_t>(__fdividef(static_cast<float>(a), static_cast<float>(p1)));
  int64_t rem = static_cast<int64_t>(a) - static_cast<int64_t>(q * p1);
  if (rem < 0) rem += static_cast<int64_t>(p1);
  if (rem >= static_cast<int64_t>(p1)) rem -= static_cast<int64_t>(p1);
  return static_cast<uint64_t>(rem) + (static_cast<uint64_t>(l) << j) - p1;  // V + RB 2^j
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

template <int PATH, int NT>
__device__ __forceinline__ void prime_residues(const uint64_t e, const uint64_t (&p)[NT], const bool (&valid)[NT],
                                               const PrimeClass* classes, uint32_t (&x0)[NT], uint32_t (&x1)[NT],
                                               uint32_t (&m0)[NT], uint32_t (&m1)[NT], uint32_t (&mp)[NT]) {
  constexpr bool WIDE = PathTraits<PATH>::kWide;
  int l = 0;
#pragma unroll
  for (int t = 0; t < NT; ++t) l = max(l, bitlen64(p[t]));
  l = static_cast<int>(__reduce_max_sync(0xffffffffu, static_cast<uint32_t>(l)));
  const int j = WIDE ? l - 5 : l - 4;
  uint64_t rem[NT];
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    m0[t] = lo32(p[t]);
    m1[t] = hi32(p[t]);
    mp[t] = neg_inverse32(m0[t]);
    const uint64_t u = reduced_exponent<PATH>(e, p[t] - 1, l, j);
    const uint64_t x = 1ull << static_cast<uint32_t>(u >> j);
    x0[t] = lo32(x);
    x1[t] = hi32(x);
    rem[t] = u & ((1ull << j) - 1ull);
  }
  int b = j;
  if (WIDE) {
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
    // one bit at a time: moduli of up to 29 (lazy) and 31 bits (reduced) allow a shift of one
    while (b > 0) {
      --b;
      uint32_t sh[NT];
#pragma unroll
      for (int t = 0; t < NT; ++t) sh[t] = static_cast<uint32_t>(rem[t] >> b) & 1u;
      square_all<PATH, NT>(x0, x1, m0, m1, mp, sh, true);
    }
  }
  // times H, with p's sign
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    int c = 0;
    while (p[t] <= classes[c].above) ++c;
    const PrimeClass& C = classes[c];
    const uint32_t n0 = lo32(C.num), n1 = hi32(C.num);
    uint64_t y;
    if (WIDE) {
      // x num / 2^64 mod p: x < 2 p < 2^47, num < 2^54, so the result is below 2 p
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
    if ((m0[t] & 2u) && y != 0) y = p[t] - y;  // chi(p) = -1 for p = 3 mod 4
    if (!valid[t]) y = 0;
    x0[t] = lo32(y);
    x1[t] = hi32(y);
  }
}

// Sums every thread's LMAX-limb value over the CTA and adds it to the carry-save slots.
template <int LMAX>
__device__ __forceinline__ void flush_cta(uint32_t (&acc)[LMAX], uint32_t L, unsigned long long* slots) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t wid = threadIdx.x >> 5;
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

constexpr int kPrimeNT = 4;  // primes per thread

template <int LMAX, int PATH>
__global__ void __launch_bounds__(kHeadThreads) prime_kernel(const __grid_constant__ PrimeArgs A) {
  __shared__ PrimeClass classes[kMaxPrimeClasses];
  for (uint32_t i = threadIdx.x; i < A.nclasses * (sizeof(PrimeClass) / 4); i += blockDim.x)
    reinterpret_cast<uint32_t*>(classes)[i] = reinterpret_cast<const uint32_t*>(A.classes)[i];
  __syncthreads();
  constexpr int NT = kPrimeNT;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t count = min(*A.count, A.cap);
  uint32_t acc[LMAX];
#pragma unroll
  for (int i = 0; i < LMAX; ++i) acc[i] = 0;
  for (uint32_t at = warp * (32 * NT); at < count; at += nwarps * (32 * NT)) {
    uint64_t p[NT];
    bool valid[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const uint32_t i = at + 32 * t + lane;
      valid[t] = i < count;
      p[t] = A.base + A.list[min(i, count - 1)];
    }
    uint32_t x0[NT], x1[NT], m0[NT], m1[NT], mp[NT];
    prime_residues<PATH, NT>(A.e, p, valid, classes, x0, x1, m0, m1, mp);
    fold_digits<PathTraits<PATH>::kWide, false, NT, LMAX>(acc, x0, x1, m0, m1, mp);
  }
  flush_cta<LMAX>(acc, A.L, A.slots);
}

// ---------------------------------------------------------------- sums mod p

// Residues mod m < 2^31 in one word, fully reduced.
struct Arith1 {
  using T = uint32_t;
  static constexpr int kBits = 32;
  uint32_t m, mp;
  __device__ explicit Arith1(uint64_t q) : m(lo32(q)), mp(neg_inverse32(lo32(q))) {}
  __device__ __forceinline__ T redc(uint64_t t) const {  // t 2^-32 mod m, t < m 2^32
    const uint32_t u = lo32(t) * mp;
    const uint32_t r = hi32(t) + __umulhi(u, m) + (lo32(t) != 0u ? 1u : 0u);
    return min(r, r - m);
  }
  __device__ __forceinline__ T mul(T a, T b) const { return redc(static_cast<uint64_t>(a) * b); }
  // (a c + b) 2^-32 mod m for a word c < 2^32
  __device__ __forceinline__ T mul_word(T a, uint32_t c, T b) const { return redc(static_cast<uint64_t>(a) * c + b); }
  __device__ __forceinline__ T add(T a, T b) const {
    const uint32_t r = a + b;
    return min(r, r - m);
  }
  __device__ __forceinline__ T neg(T a) const { return a != 0u ? m - a : 0u; }
  __device__ __forceinline__ T one() const { return static_cast<T>(r_mod_m_bitserial<32>(m).r); }
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
  __device__ explicit Arith2(uint64_t q) : m(q) {
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
  __device__ __forceinline__ T one() const { return r_mod_m_bitserial<64>(m).r; }
  __device__ __forceinline__ T plain(T a) const { return mul(a, 1); }
  __device__ __forceinline__ uint32_t digit(T& x) const {
    uint32_t x0 = lo32(x), x1 = hi32(x);
    const uint32_t q = hensel_step64(x0, x1, Mod64{lo32(m), hi32(m), lo32(mp)});
    x = make64(x0, x1);
    return q;
  }
};

// den^-1 2^e (Montgomery form) for a unit `den` mod m whose group of units has
// exponent phi: den^(phi - 1) and 2^e in one ladder.  0 <= e < phi.
template <class A>
__device__ typename A::T inverse_times_power(const A& M, typename A::T den, uint64_t phi, uint64_t e) {
  const typename A::T one = M.one();
  typename A::T z = one;
  const uint64_t f = phi - 1;
  for (int b = bitlen64(phi) - 1; b >= 0; --b) {
    z = M.mul(z, z);
    if ((f >> b) & 1u) z = M.mul(z, den);
    if ((e >> b) & 1u) z = M.add(z, z);
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

// The sum over i0 <= i < i1 of s(i) h^-(i - i0) / c, c = 2 i + 1, as the fraction
// h num / den, terms whose c is a multiple of p left out.  s(i) changes sign with bit
// `flip` of i.  From the last term down: num <- c num + s den, den <- h c den, each
// reduction leaving the same factor 2^-32 in both.  WORD: h is a word (a power of two
// below 2^11 with h c < 2^32); else h is a residue in Montgomery form.
template <class A, bool WORD, bool SKIP>
__device__ __forceinline__ void sum_fraction(const A& M, uint64_t i0, uint64_t i1, uint32_t flip, uint64_t p,
                                             typename A::T h, typename A::T& num, typename A::T& den) {
  num = 0;
  den = 1;
  if (i0 >= i1) return;
  uint64_t skip = 0;  // the largest odd multiple of p not above the last c
  if (SKIP) {
    skip = (2 * i1 - 1) / p;
    skip = skip == 0 ? 0 : ((skip - 1) | 1u) * p;
  }
  uint32_t c = static_cast<uint32_t>(2 * i1 - 1);
  const uint32_t c0 = static_cast<uint32_t>(2 * i0 + 1);
  const uint32_t bit = 2 * flip;  // of c: bit `flip` of i is bit 2 flip of c
  for (;;) {
    if (SKIP && c == static_cast<uint32_t>(skip)) {
      skip = skip > p ? skip - 2 * p : 0;
      num = M.mul_word(num, 1u, 0);
      den = WORD ? M.mul_word(den, static_cast<uint32_t>(h), 0) : M.mul(M.mul_word(den, 1u, 0), h);
    } else {
      num = M.mul_word(num, c, (c & bit) ? M.neg(den) : den);
      den = WORD ? M.mul_word(den, c * static_cast<uint32_t>(h), 0) : M.mul(M.mul_word(den, c, 0), h);
    }
    if (c == c0) break;
    c -= 2;
  }
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

// One prime per thread: num / den of the three sums with i0 = 0, one ladder for the
// inverse of their denominators and the power of 2.
//   H = 16 (num_A / den_A - 4 num_B / den_B - num_C / den_C)
template <class A, int LMAX>
__global__ void __launch_bounds__(kHeadThreads) prime_sum_kernel(const __grid_constant__ PrimeArgs G) {
  const uint32_t count = min(*G.count, G.cap);
  uint32_t acc[LMAX];
#pragma unroll
  for (int i = 0; i < LMAX; ++i) acc[i] = 0;
  using T = typename A::T;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    const uint64_t p = G.base + G.list[i];
    const A M(p);
    T nA, dA, nB, dB, nC, dC;
    sum_fraction<A, true, false>(M, 0, (G.A / p + 1) / 2, 1, p, 4, nA, dA);
    sum_fraction<A, true, false>(M, 0, (G.B / p + 1) / 2, 1, p, 1024, nB, dB);
    sum_fraction<A, true, false>(M, 0, (G.C / p + 1) / 2, 2, p, 32, nC, dC);
    const T bc = M.mul(dB, dC);
    const T b4 = M.add(nB, nB);
    T num = M.mul(nA, bc);
    num = M.add(num, M.neg(M.mul(M.mul(M.add(b4, b4), dA), dC)));
    num = M.add(num, M.neg(M.mul(M.mul(nC, dA), dB)));
    const T inv = inverse_times_power<A>(M, M.mul(dA, bc), p - 1, (G.e + 4) % (p - 1));
    T x = M.plain(M.mul(num, inv));
    if (p & 2u) x = M.neg(x);
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

// One warp per prime power q = p^a.  The summands of each sum repeat with a constant
// ratio after `period` odd c (c^-1 mod q after q, the signs after 1 or 4 of those), so
// at most `period` of them are added up, times a geometric sum: the lanes share them
// evenly, each lane's part being its own fraction over q.  PRIME: a = 1 (p in the
// list), else every a >= 2 with p^a <= A.
template <class A, bool PRIME, int LMAX>
__global__ void __launch_bounds__(kHeadThreads) prime_power_kernel(const __grid_constant__ PrimeArgs G) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t count = min(*G.count, G.cap);
  using T = typename A::T;
  uint32_t acc[LMAX];
#pragma unroll
  for (int i = 0; i < LMAX; ++i) acc[i] = 0;
  for (uint32_t at = warp; at < count; at += nwarps) {
    const uint64_t p = G.base + G.list[at];
    const uint64_t last = G.A / p;  // q p is another power up to A while q <= A / p
    for (uint64_t q = PRIME ? p : p * p; q <= G.A; q *= p) {
      const A M(q);
      const uint64_t phi = q / p * (p - 1);
      const int64_t sq = static_cast<int64_t>(q), e = static_cast<int64_t>(G.e);
      const bool chi_neg = (q & 2u) != 0, psi_neg = (q & 4u) != 0;
      const uint64_t limit[3] = {G.A, G.B, G.C};
      uint64_t whole[3], rest[3], period[3];
      bool repeats = false;
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        const uint64_t n = (limit[s] / q + 1) / 2;  // odd c up to limit / q
        period[s] = s == 2 ? 4 * q : q;
        whole[s] = n / period[s];
        rest[s] = n % period[s];
        repeats |= whole[s] > 0;
      }
      for (int pass = 0; pass < (repeats ? 2 : 1); ++pass) {
        // pass 0: the first `rest` summands, whole + 1 times; pass 1: the others, whole times
        T num = 0, den = M.one();
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          const uint64_t lo = pass == 0 ? 0 : rest[s], hi = pass == 0 ? rest[s] : period[s];
          const uint64_t times = whole[s] + (pass == 0 ? 1 : 0);
          const uint64_t share = (hi - lo + 31) / 32;
          const uint64_t i0 = lo + min(hi - lo, lane * share), i1 = min(hi, i0 + share);
          if (times == 0 || i0 >= i1) continue;
          constexpr uint32_t kRatio[3] = {2, 10, 5};  // summand i carries 2^(-ratio q i)
          const int64_t ratio = kRatio[s];
          const T h = PRIME ? static_cast<T>(1u << kRatio[s])
                            : power_of_two<A>(M, exponent_mod(ratio * sq, phi));
          T n_s, d_s;
          sum_fraction<A, PRIME, true>(M, i0, i1, s == 2 ? 2 : 1, p, h, n_s, d_s);
          // times 2^(e + const - (power at i0)), h of the fraction included
          const int64_t start = s == 0 ? e + 3 - sq : s == 1 ? e + 1 - 5 * sq : e - 1 - 5 * (sq - 1) / 2;
          T k = power_of_two<A>(M, exponent_mod(start + ratio * sq - ratio * sq * static_cast<int64_t>(i0), phi));
          if (times > 1) {
            const int64_t per = static_cast<int64_t>(period[s]);
            T r = power_of_two<A>(M, exponent_mod(-ratio * sq * per, phi));
            if (s != 2) r = M.neg(r);
            k = M.mul(k, geometric<A>(M, r, times));
          }
          const bool minus = s == 0 ? chi_neg : s == 1 ? !chi_neg : !psi_neg;
          k = M.mul(k, n_s);
          // num / den + k / d_s
          num = M.add(M.mul(num, d_s), M.mul(minus ? M.neg(k) : k, den));
          den = M.mul(den, d_s);
        }
        const T x = M.plain(M.mul(num, inverse_times_power<A>(M, den, phi, 0)));
        fold_one<A, LMAX>(M, x, acc);
      }
      if (PRIME || q > last) break;
    }
  }
  flush_cta<LMAX>(acc, G.L, G.slots);
}

}  // namespace bbp
