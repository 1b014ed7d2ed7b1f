// Segmented sieve of Eratosthenes on the device, and the check that decides whether the
// prime form's result stands (bbp_sieve.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace bbp {

constexpr int kSieveThreads = 512;
constexpr int kSieveMaxWords = 1 << 14;  // 64 KB of odd numbers, 2^20 numbers a segment

// Primes p with `above` < p <= `upto` in the `segments` segments of 64 * words numbers
// from `base` (a multiple of 64 * words), as offsets from `base`, ascending within a
// segment, appended to list[0, cap) through *count.  *count counts all of them: a
// count past `cap` says that some are missing.  The base primes are the `nprimes` odd
// primes from 67 on, ascending, with inv[i] = floor((2^64 - 1) / primes[i]); they must
// reach the square root of `upto`.
struct SieveArgs {
  uint64_t base, above, upto;
  uint32_t segments, words;
  const uint32_t* primes;
  const uint64_t* inv;
  const uint32_t* nprimes;
  uint32_t* list;
  uint32_t* count;
  uint32_t cap;
};
cudaError_t launch_sieve(const SieveArgs& a, int blocks, cudaStream_t s);
int sieve_occupancy(int words);

// primes[0, *count) <- the odd primes up to `upto` (< 2^23) ascending, *count their number,
// inv their reciprocals; the first kSieveTinyPrimes of them are below 67.
constexpr int kSieveTinyPrimes = 17;
cudaError_t launch_base_primes(uint32_t upto, uint32_t* primes, uint64_t* inv, uint32_t* count, uint32_t* nsieve,
                               cudaStream_t s);

// The prime form's sum S' and the term-by-term sum S both err by less than `bound`
// units from the exact value, so they differ by less than 2 bound: if S' mod 2^(W - P)
// keeps 3 bound from both ends, S has the same top P bits and certifies all of them
// (S mod 2^(W - P) keeps `bound` from both ends).  Then out and *valid are written and
// *redo = 0; else, or if one of the `nlists` lists holds more than `cap` primes, *redo = 1
// and nothing is written.
cudaError_t launch_prime_check(const unsigned long long* slots, int L, uint32_t P, uint64_t bound,
                               const uint32_t* counts, uint32_t nlists, uint32_t cap, uint8_t* out, uint32_t* valid,
                               uint32_t* redo, cudaStream_t s);

}  // namespace bbp
