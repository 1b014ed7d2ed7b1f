// The prime form of a whole query's head sum, host side: limits, classes and launch
// arguments.  Pure C++, no CUDA calls.
//
// Every head term is 2^e / m mod 1 with m odd.  Splitting 1/m into partial fractions
// over the prime powers q = p^a that divide m exactly,
//
//   1/m = sum_q ((m/q)^-1 mod q) / q   (mod 1),
//
// and collecting by q turns the sum over all terms into a sum over the prime powers up to
// the largest modulus: one modular exponentiation 2^d mod p per prime serves every term
// whose modulus p divides.
//
// Bellard's formula (Eq. 2), in terms of odd m:
//
//   series 10k+1, 10k+3, 10k+5, 10k+7, 10k+9 together
//       =  8 sum_m chi(m) 2^(d-m) / m  -  2 sum_m chi(m) 2^(d-5m) / m      (A and B)
//   series 4k+1, 4k+3 together
//       = -  sum_m psi(m) 2^(d-1-5(m-1)/2) / m                             (C)
//
// with chi(m) = (-1)^((m-1)/2) and psi(m) = +1 for m = 1, 3 mod 8, -1 for 5, 7 mod 8 (the
// second sum of A, B corrects the multiples of 5, whose sign and exponent differ).
// For a prime p, m = c p with p not dividing c: 2^(cp) = 2^c mod p, and
// psi(p) 2^((p-1)/2) = chi(p) mod p, so p's part is
//
//   chi(p) 2^d H / p,   H = 4 sum_(c <= A/p) chi(c) 4^-i / c - 1/16 sum_(c <= B/p) chi(c) 1024^-i / c
//                           - 1/2 sum_(c <= C/p) psi(c) 32^-i / c    (mod p),  c = 2i + 1 odd,
//
// where A, B, C are the largest m of the three sums.  The BBP formula (Eq. 1):
//
//   series 8k+1, 8k+5:  sum over m = 1 mod 4 of (2/m) 2^(d+2-(m-1)/2) / m   (up to A)
//   series 4k+3:      - sum over m = 3 mod 4 of 2^(d+2-m) / m               (up to B)
//   series 2k+1:      - sum over odd m of 2^(d+1-2m) / m                    (up to C)
//
// and with (2/p) 2^((p-1)/2) = 1 mod p, p's part is 2^d H / p with
//
//   H = 4 sum_(c = p mod 4) (2/c) 2^-((c-1)/2) / c - 4 sum_(c = -p mod 4) 2^-c / c - 2 sum_c 4^-c / c.
//
// H is one rational number for all primes with the same three limits (and, for Eq. 1, the
// same residue mod 4).
#pragma once

#include <cstdint>
#include <vector>

#ifdef __CUDACC__
#define BBP_HOST_DEVICE __host__ __device__
#else
#define BBP_HOST_DEVICE
#endif

namespace bbp {

// floor(a / p) from q, the single-precision quotient cut to a whole number.  That is off by two
// ulps and the rounding of a and p (2^-24 each, nothing for p < 2^24).  Quotients of the sums are
// at most sqrt(A): up to 2^21.7 for Eq. 2, whose ulps are 1/4, so that one correction is enough;
// up to 2^22.2 for Eq. 1, where an ulp is 1/2, and past 2^22 (n > 8.8e12) it may take two.
// (Two for both: 0.7 % of a whole query at n = 1e9 and 4e10.)
template <int FORMULA>
BBP_HOST_DEVICE inline uint32_t corrected_quotient(uint32_t q, uint64_t a, uint64_t p) {
  const int64_t m = static_cast<int64_t>(p);
  int64_t rem = static_cast<int64_t>(a) - static_cast<int64_t>(q * p);
  if (FORMULA == 1 && q >= 1u << 21) {
    if (rem < 0) --q, rem += m;
    if (rem >= m) ++q, rem -= m;
  }
  if (rem < 0) --q;
  if (rem >= m) ++q;
  return q;
}

// Largest moduli of the three sums: every term of a modulus up to these is a head
// term.  Eq. 2's (at most one) head term above `A` and all tail terms are left to the
// term-by-term kernels.
struct PrimeLimits {
  int formula = 0;
  uint64_t A = 0, B = 0, C = 0;
};
PrimeLimits prime_limits(int formula, uint64_t d);
// First k of series j that the prime form does not cover.
uint64_t prime_first_k(const PrimeLimits& lim, uint32_t j, uint64_t d);

// Primes up to here take the half-reduced ladder: with x <= p + 2^35, x^2 / 2^32 + p stays
// below 2^48.
constexpr uint64_t kPrimeHalfMax = 1'020'000'000'000;  // as kHalfMaxModulus

// Primes with the same +-H = num / (den 2^kPrimeShift), by p mod 4: those above `above`, up to the
// previous class's `above`.
constexpr int kPrimeShift = 24;   // every denominator of H up to kPrimeMaxC divides den 2^24
constexpr uint32_t kPrimeMaxC = 21;  // classes reach down to A / (kPrimeMaxC + 2)
constexpr int kMaxPrimeClasses = 24;
struct PrimeClass {
  uint64_t above;
  uint64_t num[2];   // |H| den 2^24 < 2^54 for p = 1 and 3 mod 4
  uint64_t den_inv;  // den^-1 mod 2^64
  uint32_t den;      // lcm of the odd numbers up to A / p: 1, 3, 15, ... < 2^24
  uint32_t neg_inv;  // -den^-1 mod 2^32
  uint32_t r2, r3;   // 2^64 mod den, 2^96 mod den
  uint32_t lambda;   // exponent of the group of units mod den, minus 1
  uint32_t negative; // bit 0, 1: the part of p = 1, 3 mod 4 is negative
};
// Classes in descending order of `above`; the last one's `above` is A / (kPrimeMaxC + 2).
std::vector<PrimeClass> prime_classes(const PrimeLimits& lim);

// Whether the prime form serves this query: position in range, and the error bound
// small enough against the guard bits that its result is almost always certain to
// equal the term-by-term one (see launch_prime_check in bbp_sieve.cuh).
bool prime_form_serves(int formula, uint64_t n, uint32_t P, uint32_t W, uint64_t bound);

// 32-bit product halves the prime form multiplies for a query of `limbs` limbs (a model,
// counted as in head_term_imad, with the primes' number taken as the integral of
// 1 / ln x): per prime above A / 23 the squarings of its ladder, the product with H and
// the quotient digits; per prime below, a ladder with a product at each bit, and 12 per
// summand of its sums.
double prime_form_imad(const PrimeLimits& lim, int limbs);

// P = 128, term by term and by primes: n = 2e7 334 and 217 us, 3e7 474 and 241, 1e8 1560 and 354.
// About 200 us of the latter are launches and chains.
constexpr uint64_t kPrimeMinN = 16'000'000;
// The largest product of w = 2^10 and a c in the sums mod p (Eq. 2's second sum, c <= sqrt(0.4 n))
// stays below 2^31; Eq. 1's (w = 2^4, c <= sqrt(4 n)) are smaller.  Its A = 2 n is below 2^44.4, where
// small_quotient and the 46-bit arithmetic reach.
constexpr uint64_t kPrimeMaxN = 10'900'000'000'000;

}  // namespace bbp
