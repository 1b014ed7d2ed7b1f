// Host side of the prime form of a query's head sum (bbp_primes.h).
#include "bbp_primes.h"

#include <algorithm>
#include <cmath>
#include <numeric>

#include "bbp_planner.h"

namespace bbp {

namespace {

uint64_t odd_down(uint64_t v) { return v == 0 ? 0 : (v & 1 ? v : v - 1); }

uint32_t pow_mod(uint32_t e, uint32_t m) {  // 2^e mod m
  uint64_t r = 1 % m;
  for (uint32_t i = 0; i < e; ++i) r = r * 2 % m;
  return static_cast<uint32_t>(r);
}

}  // namespace

PrimeLimits prime_limits(int formula, uint64_t d) {
  PrimeLimits l;
  l.formula = formula;
  if (formula == 0) {
    // A: exponents d + 3 - m (and d + 1 - m for multiples of 5) are not negative up to
    // m = d + 1.  C: d - 1 - 5 (m - 1) / 2 is not negative up to 1 + 2 (d - 1) / 5.
    l.A = odd_down(d + 1);
    l.B = odd_down(l.A / 5);
    l.C = d >= 1 ? odd_down(1 + 2 * (d - 1) / 5) : 0;
  } else {
    // d + 2 - (m - 1) / 2, d + 2 - m and d + 1 - 2 m are not negative
    l.A = 2 * d + 5;
    l.B = odd_down(d + 2);
    l.C = odd_down((d + 1) / 2);
  }
  return l;
}

uint64_t prime_first_k(const PrimeLimits& lim, uint32_t j, uint64_t d) {
  if (lim.formula != 0) return head_end(formula_def(lim.formula), j, d);
  const SeriesDef& s = formula_def(0).s[j];
  const uint64_t top = s.a == 10 ? lim.A : lim.C;
  return top < s.b ? 0 : (top - s.b) / s.a + 1;
}

namespace {

// H den 2^kPrimeShift of the primes p = r mod 4 with the quotients ca, cb, cc
int64_t numerator(int formula, uint32_t r, int64_t den, uint64_t ca, uint64_t cb, uint64_t cc) {
  auto scaled = [&](int64_t v, int64_t bits) { return v * (int64_t{1} << (kPrimeShift + bits)); };
  int64_t num = 0;
  for (uint64_t c = 1; c <= ca; c += 2) {
    const int64_t f = den / static_cast<int64_t>(c), i = static_cast<int64_t>(c / 2);
    if (formula == 0) {
      num += scaled(i & 1 ? -f : f, 2 - 2 * i);
      if (c <= cb) num -= scaled(i & 1 ? -f : f, -4 - 10 * i);
      if (c <= cc) num -= scaled(i & 2 ? -f : f, -1 - 5 * i);
    } else {
      const bool minus = c % 8 == 3 || c % 8 == 5;  // (2/c)
      if (c % 4 == r) num += scaled(minus ? -f : f, 2 - i);
      if (c % 4 != r && c <= cb) num -= scaled(f, 2 - static_cast<int64_t>(c));
      if (c <= cc) num -= scaled(f, 1 - 2 * static_cast<int64_t>(c));
    }
  }
  return formula == 0 && r == 3 ? -num : num;  // chi(p)
}

}  // namespace

std::vector<PrimeClass> prime_classes(const PrimeLimits& lim) {
  std::vector<uint64_t> cuts;  // H changes below each of these
  for (uint32_t c = 1; c <= kPrimeMaxC + 2; c += 2) cuts.push_back(lim.A / c);
  const uint64_t bottom = lim.A / (kPrimeMaxC + 2);
  for (uint32_t c = 1; lim.C / c > bottom; c += 2) cuts.push_back(lim.C / c);
  for (uint32_t c = 1; lim.B / c > bottom; c += 2) cuts.push_back(lim.B / c);
  std::sort(cuts.begin(), cuts.end(), std::greater<uint64_t>());
  cuts.erase(std::unique(cuts.begin(), cuts.end()), cuts.end());
  std::vector<PrimeClass> out;
  for (size_t i = 1; i < cuts.size(); ++i) {
    const uint64_t p = cuts[i] + 1;  // the class: cuts[i] < p <= cuts[i - 1]
    const uint64_t ca = lim.A / p, cb = lim.B / p, cc = lim.C / p;
    PrimeClass k{};
    k.above = cuts[i];
    uint64_t den = 1;
    for (uint64_t c = 3; c <= ca; c += 2) den = std::lcm(den, c);
    for (uint32_t r = 1; r <= 3; r += 2) {
      const int64_t num = numerator(lim.formula, r, static_cast<int64_t>(den), ca, cb, cc);
      k.num[r / 2] = static_cast<uint64_t>(num < 0 ? -num : num);
      if (num < 0) k.negative |= 1u << (r / 2);
    }
    k.den = static_cast<uint32_t>(den);
    uint64_t inv = den;  // Newton-Hensel lifting of den^-1 mod 2^64 (x = den: correct to 3 bits)
    for (int it = 0; it < 5; ++it) inv *= 2 - den * inv;
    k.den_inv = inv;
    k.neg_inv = 0u - static_cast<uint32_t>(inv);
    k.r2 = pow_mod(64, k.den);
    k.r3 = pow_mod(96, k.den);
    uint32_t lambda = 1;
    uint32_t rest = k.den;
    for (uint32_t f = 3; f <= kPrimeMaxC; f += 2) {
      uint32_t q = 1;
      while (rest % f == 0) {
        rest /= f;
        q *= f;
      }
      if (q > 1) lambda = std::lcm(lambda, q / f * (f - 1));
    }
    k.lambda = lambda - 1;
    out.push_back(k);
  }
  return out;
}

double prime_form_imad(const PrimeLimits& lim, int limbs) {
  const double top = static_cast<double>(lim.A), bottom = top / (kPrimeMaxC + 2), root = std::sqrt(top);
  double total = 0;
  for (double x = root; x < top;) {  // in steps of 1 % of x
    const double hi = std::min(top, x * 1.01), mid = 0.5 * (x + hi);
    const int l = bitlen(static_cast<uint64_t>(mid));
    const bool wide = l > 31;
    const double ladder = wide ? 13.0 * (l - 5) : 4.0 * (l - 4), digits = (wide ? 4.0 : 2.0) * limbs + 6.0;
    // Eq. 2: odd c up to A / p, and up to 0.2 and 0.4 of that; Eq. 1: a quarter, an eighth, an eighth
    const double summands = (lim.formula == 0 ? 0.8 : 0.5) * top / mid;
    const double per = mid > bottom ? ladder + digits + (wide ? 16.0 : 10.0) : 2.0 * ladder + digits + 12.0 * summands;
    total += per * (hi - x) / std::log(mid);
    x = hi;
  }
  return total;
}

bool prime_form_serves(int formula, uint64_t n, uint32_t P, uint32_t W, uint64_t bound) {
  if (n < kPrimeMinN || n > kPrimeMaxN) return false;
  if (formula != 0 && formula != 1) return false;
  // the result is uncertain for 6 bound in 2^(W - P) positions: ask for less than one in 64
  return bitlen(bound) + 9 <= static_cast<int>(W - P);
}

}  // namespace bbp
