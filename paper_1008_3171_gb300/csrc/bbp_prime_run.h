// Running the prime form of a query's head sum (bbp_primes.h): workspaces, and a query's
// lists of primes, all at once or some at a time.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "bbp.h"
#include "bbp_kernels.cuh"
#include "bbp_primes.h"

struct PrimeState;  // device memory, streams and events of one query at a time

namespace bbp {

// The workspace for position n, made or enlarged to lists of up to `max_list` primes;
// false if it is not there and cannot be made now (a stream capture is going on on `st`,
// or memory is short): the caller then sums the terms.
constexpr uint32_t kPrimeListMax = 24u << 20;      // single queries: two lists of 96 MB
constexpr uint32_t kPrimeLaneListMax = 6u << 20;   // each of several workspaces: two of 24 MB
bool prime_workspace(PrimeState** state, uint64_t n, uint32_t max_list, cudaStream_t st);
void release_prime_state(PrimeState** state);
// Waits for what runs on the workspace's own streams, beside the caller's (NULL: nothing).
void wait_prime_state(PrimeState* state);

// One query on one workspace and one stream: begin, every list in order, finish.  Runs on a
// workspace follow one another, on whatever streams; captured ones are ordered by who replays
// them.
class PrimeRun {
 public:
  // The query at position n, W working bits, into `slots` (to which the terms that the
  // prime form does not cover are added by the caller).  Host work alone; not BBP_OK: the caller
  // sums the terms.
  bbp_status plan(PrimeState* state, int sm_count, int formula, uint64_t n, uint32_t W, unsigned long long* slots);
  size_t lists() const { return lists_.size(); }
  double share(size_t i) const;  // list i's part of the numbers up to n
  // Base primes and prime powers.
  bbp_status begin(cudaStream_t st);
  // Lists [first, last).
  bbp_status run(size_t first, size_t last, cudaStream_t st);
  // The check of the finished sum: d_out and d_valid (may be NULL) are written and
  // *d_redo = 0, or *d_redo = 1.
  bbp_status finish(uint32_t P, uint64_t bound, uint8_t* d_out, uint32_t* d_valid, uint32_t* d_redo, cudaStream_t st);
  uint64_t launches() const { return launches_; }  // kernels so far

 private:
  struct List {
    uint64_t base, lo, hi;
    uint32_t segments;
    PrimeKernel kernel;
    uint32_t one_mod_4;  // only primes 1 mod 4 matter
  };
  PrimeState* state_ = nullptr;
  int sms_ = 0, lmax_ = 0, formula_ = 0;
  bool captured_ = false;
  uint32_t base_to_ = 0;
  uint64_t e_ = 0, launches_ = 0;
  PrimeArgs args_{};
  std::vector<List> lists_;
};

}  // namespace bbp
