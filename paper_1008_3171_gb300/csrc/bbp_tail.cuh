// Tail terms (exponent e < 0), shared by the tail kernels and the one-launch query kernel.
#pragma once

#include <cstdint>

#include "bbp_device.cuh"
#include "bbp_kernels.cuh"

namespace bbp {

// A tail term is B_k = 2^e / m with e < 0 (Eq. 5); its W-bit value is
// floor(2^(W+e)/m) = floor(floor(2^W/m) / 2^-e): the fraction of 1/m, shifted
// (Sec. 4.3: shift by b bits, then divide to W - b bits).  There are only about
// W/step of them per series, so one thread per term with plain loops.
// t (W/32 limbs, signed by (-1)^k and the series sign, mod 2^W) of tail term k.
__device__ inline void tail_term(const TailArgs& A, const uint64_t k, uint32_t* t) {
  const int64_t e = static_cast<int64_t>(A.d) + A.c - static_cast<int64_t>(A.step) * static_cast<int64_t>(k);
  const uint32_t L = A.L;
  const int64_t bshift = -e;  // 1 <= bshift <= W
  const uint64_t m = static_cast<uint64_t>(A.a) * k + A.b;
  uint32_t q[kMaxLimbs];
  for (uint32_t i = 0; i < L; ++i) { q[i] = 0; t[i] = 0; }
  if (e >= 0 || bshift > static_cast<int64_t>(A.W)) return;
  const uint32_t b = static_cast<uint32_t>(bshift);
  if (m == 1) {
    const uint32_t bit = A.W - b;  // floor(2^(W-b) / 1), below 2^W since b >= 1
    t[bit >> 5] = 1u << (bit & 31u);
  } else {
    uint64_t x = 1;  // 2^W mod m by doubling; m < 2^62
    for (uint32_t i = 0; i < A.W; ++i) {
      x <<= 1;
      if (x >= m) x -= m;
    }
    Mod64 M{lo32(m), hi32(m), neg_inverse32(lo32(m))};
    uint32_t x0 = lo32(x), x1 = hi32(x);
    for (uint32_t i = 0; i < L; ++i) q[i] = hensel_step64(x0, x1, M);
    // t = q >> b
    const uint32_t bl = b >> 5, bb = b & 31u;
    for (uint32_t i = 0; i < L; ++i) {
      const uint32_t src = i + bl;
      uint32_t lo = src < L ? q[src] : 0u;
      uint32_t hi = src + 1 < L ? q[src + 1] : 0u;
      t[i] = bb ? ((lo >> bb) | (hi << (32u - bb))) : lo;
    }
  }
  const bool neg = ((A.alternating && (k & 1ull)) ? 1u : 0u) ^ A.negate;
  if (neg) {
    uint64_t carry = 1;
    for (uint32_t i = 0; i < L; ++i) {
      const uint64_t s = static_cast<uint64_t>(~t[i]) + carry;
      t[i] = static_cast<uint32_t>(s);
      carry = s >> 32;
    }
  }
}

// The i-th term of the ranges of S laid end to end, added to its accumulators.
__device__ inline void add_tail_term(const TailSet& S, uint64_t i) {
  uint32_t r = 0;
  while (r < S.n && i >= S.a[r].count) i -= S.a[r++].count;
  if (r >= S.n) return;
  const TailArgs& A = S.a[r];
  uint32_t t[kMaxLimbs];
  tail_term(A, A.k_begin + i, t);
  for (uint32_t l = 0; l < A.L; ++l)
    if (t[l]) atomicAdd(A.slots + l, static_cast<unsigned long long>(t[l]));
}

}  // namespace bbp
