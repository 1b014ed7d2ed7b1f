// Segmented sieve of Eratosthenes on the device, and the check that decides whether the
// prime form's result stands (bbp_sieve.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace bbp {

constexpr int kSieveThreads = 512;
constexpr uint32_t kSieveMaxEntries = 192u << 10;  // bytes of shared memory

// A base prime p as the sieve reads it.
struct SievePrime {
  uint32_t p;
  uint32_t inv;    // floor((2^32 - 1) / p)
  uint32_t inv30;  // 30^-1 mod p
  uint32_t at;     // -base / 30 mod p for the list being sieved
};

// Primes p with `above` < p <= `upto` among the numbers prime to 30 of `segments`
// segments of 30 * entries numbers (entries a multiple of 32; segments * entries < 2^28)
// from `base` (a multiple of 30), as offsets from `base` in no particular order, appended
// to list[0, cap) through *count.  *count counts all of them: a count past `cap` says that
// some are missing.  The base primes are the *nprimes primes from 17 on (none above
// `above`), ascending, up to at least the square root of `upto`; their `at` is set here.
struct SieveArgs {
  uint64_t base, above, upto;
  uint32_t segments, entries;
  uint32_t one_mod_4;  // 1: only the primes 1 mod 4
  SievePrime* primes;
  const uint32_t* nprimes;
  uint32_t* list;
  uint32_t* count;
  uint32_t cap;
};
cudaError_t launch_sieve(const SieveArgs& a, int sms, cudaStream_t s);

// primes[0, *count) <- the odd primes up to `upto` (below 2^23) ascending, *count their
// number, *nsieve the number of those from 17 on, which are at sieve[kSieveTinyPrimes]
// and after.
constexpr int kSieveTinyPrimes = 5;
cudaError_t launch_base_primes(uint32_t upto, uint32_t* primes, SievePrime* sieve, uint32_t* count, uint32_t* nsieve,
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
