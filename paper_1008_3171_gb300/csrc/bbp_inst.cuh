// Launchers of the head and queue kernels for one accumulator class.  A
// translation unit defines BBP_LMAX (limbs per thread) and includes this file,
// so the seven classes compile in parallel; bbp_kernels.cu dispatches to them.
#pragma once

#ifndef BBP_LMAX
#error "define BBP_LMAX (accumulator limbs) before including bbp_inst.cuh"
#endif

#include <algorithm>

#include "bbp_primes.cuh"
#include "bbp_tile.cuh"

#define BBP_CAT2(a, b) a##b
#define BBP_CAT(a, b) BBP_CAT2(a, b)

namespace bbp {
namespace {

// The half-reduced ladder of 4 and 16 limbs is faster as the gated kernel, gate or not (1e8 terms,
// 40-bit moduli: P = 64 3.76 against 3.79 ms, P = 448 4.42 against 4.53).
template <int S, Ladder LADDER>
constexpr bool kGatedFaster = LADDER == kLadderHalf && S == 2 && (BBP_LMAX == 4 || BBP_LMAX == 16);

template <int PATH, int S, Ladder LADDER = kLadderPlain, bool GATED = kGatedFaster<S, LADDER>>
cudaError_t launch_head_t(const HeadArgs& a, int blocks, int threads, cudaStream_t s) {
  const uint64_t tile = 32ull * S * a.run;
  const uint64_t ntiles = (a.count + tile - 1) / tile;
  head_kernel<BBP_LMAX, PATH, S, LADDER, GATED><<<blocks, threads, 0, s>>>(a, ntiles);
  return cudaGetLastError();
}

template <int PATH, int S, Ladder LADDER = kLadderPlain, bool GATED = kGatedFaster<S, LADDER>>
int head_occupancy_t(int threads) {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, head_kernel<BBP_LMAX, PATH, S, LADDER, GATED>, threads, 0) != cudaSuccess)
    return 1;
  return n > 0 ? n : 1;
}

template <int PATH, int S>
cudaError_t launch_queue_t(const BatchDev& b, uint32_t jb, uint32_t je, unsigned long long* cursor, int blocks,
                           cudaStream_t s) {
  queue_kernel<BBP_LMAX, PATH, S><<<blocks, kHeadThreads, 0, s>>>(b, jb, je, cursor);
  return cudaGetLastError();
}

template <int PATH, int S>
int queue_occupancy_t() {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, queue_kernel<BBP_LMAX, PATH, S>, kHeadThreads, 0) !=
      cudaSuccess)
    return 1;
  return n > 0 ? n : 1;
}

template <int S>
cudaError_t launch_query_t(const QuerySet& q, int blocks, int threads, cudaStream_t s) {
  query_kernel<BBP_LMAX, S><<<q.tail_blocks + blocks, threads, 0, s>>>(q);
  return cudaGetLastError();
}

template <typename K>
cudaError_t launch_prime_t(K kernel, const PrimeArgs& a, int sms, cudaStream_t s, int most = 32) {
  // the sieve's CTAs need the SM's shared memory while these run
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                       cudaSharedmemCarveoutMaxShared);
  int n = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, kHeadThreads, 0);
  if (e != cudaSuccess) return e;
  kernel<<<std::max(1, std::min(n, most)) * sms, kHeadThreads, 0, s>>>(a);
  return cudaGetLastError();
}

// prime_kernel's CTAs per SM: two of the four that fit, so that the next list's sieve has
// registers all along.  With four the sieve, of higher priority, takes most of the SM until it
// is done, and the rest runs alone: n = 4e10 86.4 ms, with three 84.9, two 83.5 (although the
// lists alone, nothing beside them, take 57.9 ms with two and 55.0 with four; all with four
// primes a thread, kPrimeNT).
constexpr int kPrimeCtas = 2;

}  // namespace

cudaError_t BBP_CAT(launch_prime_l, BBP_LMAX)(const PrimeArgs& a, PrimeKernel k, int formula, int sms,
                                              cudaStream_t s) {
  const bool f = formula != 0;
  switch (k) {
    case kPrimes0: return launch_prime_t(prime_kernel<BBP_LMAX, 0, false>, a, sms, s, kPrimeCtas);
    case kPrimes1: return launch_prime_t(prime_kernel<BBP_LMAX, 1, false>, a, sms, s, kPrimeCtas);
    case kPrimesHalf: return launch_prime_t(prime_kernel<BBP_LMAX, 1, true>, a, sms, s, kPrimeCtas);
    case kPrimes3: return launch_prime_t(prime_kernel<BBP_LMAX, 3, false>, a, sms, s, kPrimeCtas);
    case kSums32: return launch_prime_t(f ? prime_sum_kernel<Arith1, 1, 32, BBP_LMAX> : prime_sum_kernel<Arith1, 0, 32, BBP_LMAX>, a, sms, s);
    case kSums8: return launch_prime_t(f ? prime_sum_kernel<Arith1, 1, 8, BBP_LMAX> : prime_sum_kernel<Arith1, 0, 8, BBP_LMAX>, a, sms, s);
    case kSums1: return launch_prime_t(f ? prime_sum_kernel<Arith1, 1, 1, BBP_LMAX> : prime_sum_kernel<Arith1, 0, 1, BBP_LMAX>, a, sms, s);
    case kSums2: return launch_prime_t(f ? prime_sum_kernel<Arith2, 1, 1, BBP_LMAX> : prime_sum_kernel<Arith2, 0, 1, BBP_LMAX>, a, sms, s);
    case kPrimeWarps: return launch_prime_t(f ? prime_power_kernel<Arith1, 1, true, BBP_LMAX> : prime_power_kernel<Arith1, 0, true, BBP_LMAX>, a, sms, s);
    case kPowers1: return launch_prime_t(f ? prime_power_kernel<Arith1, 1, false, BBP_LMAX> : prime_power_kernel<Arith1, 0, false, BBP_LMAX>, a, sms, s);
    case kPowers2: return launch_prime_t(f ? prime_power_kernel<Arith2, 1, false, BBP_LMAX> : prime_power_kernel<Arith2, 0, false, BBP_LMAX>, a, sms, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t BBP_CAT(launch_query_l, BBP_LMAX)(const QuerySet& q, int streams, int blocks, int threads, cudaStream_t s) {
  return streams == 2 ? launch_query_t<2>(q, blocks, threads, s) : launch_query_t<1>(q, blocks, threads, s);
}

int BBP_CAT(query_occupancy_l, BBP_LMAX)(int streams, int threads) {
  int n = 0;
  const cudaError_t e =
      streams == 2 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, query_kernel<BBP_LMAX, 2>, threads, 0)
                   : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, query_kernel<BBP_LMAX, 1>, threads, 0);
  return e == cudaSuccess && n > 0 ? n : 1;
}

// path 0..3 (kNumPaths) and the launch_head ones, streams 1 or 2 (anything else runs 1; gated
// launches, kPathRoomy and kPathRoomy47 run the paths' own number)
cudaError_t BBP_CAT(launch_head_l, BBP_LMAX)(const HeadArgs& a, int path, int streams, int blocks, int threads,
                                             cudaStream_t s) {
  const bool two = streams == 2;
  if (a.gate) {
    switch (path) {
      case 0: return launch_head_t<0, 1, kLadderPlain, true>(a, blocks, threads, s);
      case 1: case kPathRoomy: return launch_head_t<1, 2, kLadderPlain, true>(a, blocks, threads, s);
      case 2: return launch_head_t<2, 1, kLadderPlain, true>(a, blocks, threads, s);
      case 3: return launch_head_t<3, 1, kLadderPlain, true>(a, blocks, threads, s);
      case kPathHalf: return launch_head_t<1, 2, kLadderHalf, true>(a, blocks, threads, s);
      case kPath47: case kPathRoomy47: return launch_head_t<1, 2, kLadder47, true>(a, blocks, threads, s);
      default: return cudaErrorInvalidValue;
    }
  }
  switch (path) {
    case kPathRoomy: return launch_head_t<1, 2, kLadderPlain, true>(a, blocks, threads, s);
    case kPathRoomy47: return launch_head_t<1, 2, kLadder47, true>(a, blocks, threads, s);
    case 0: return two ? launch_head_t<0, 2>(a, blocks, threads, s) : launch_head_t<0, 1>(a, blocks, threads, s);
    case 1: return two ? launch_head_t<1, 2>(a, blocks, threads, s) : launch_head_t<1, 1>(a, blocks, threads, s);
    case 2: return two ? launch_head_t<2, 2>(a, blocks, threads, s) : launch_head_t<2, 1>(a, blocks, threads, s);
    case 3: return two ? launch_head_t<3, 2>(a, blocks, threads, s) : launch_head_t<3, 1>(a, blocks, threads, s);
    case kPathHalf: return two ? launch_head_t<1, 2, kLadderHalf>(a, blocks, threads, s) : launch_head_t<1, 1, kLadderHalf>(a, blocks, threads, s);
    case kPath47: return two ? launch_head_t<1, 2, kLadder47>(a, blocks, threads, s) : launch_head_t<1, 1, kLadder47>(a, blocks, threads, s);
    default: return cudaErrorInvalidValue;
  }
}

int BBP_CAT(head_occupancy_l, BBP_LMAX)(int path, int streams, int threads) {
  const bool two = streams == 2;
  switch (path) {
    case kPathRoomy: return head_occupancy_t<1, 2, kLadderPlain, true>(threads);
    case kPathRoomy47: return head_occupancy_t<1, 2, kLadder47, true>(threads);
    case 0: return two ? head_occupancy_t<0, 2>(threads) : head_occupancy_t<0, 1>(threads);
    case 1: return two ? head_occupancy_t<1, 2>(threads) : head_occupancy_t<1, 1>(threads);
    case 2: return two ? head_occupancy_t<2, 2>(threads) : head_occupancy_t<2, 1>(threads);
    case 3: return two ? head_occupancy_t<3, 2>(threads) : head_occupancy_t<3, 1>(threads);
    case kPathHalf: return two ? head_occupancy_t<1, 2, kLadderHalf>(threads) : head_occupancy_t<1, 1, kLadderHalf>(threads);
    case kPath47: return two ? head_occupancy_t<1, 2, kLadder47>(threads) : head_occupancy_t<1, 1, kLadder47>(threads);
    default: return 1;
  }
}

cudaError_t BBP_CAT(launch_queue_l, BBP_LMAX)(const BatchDev& b, uint32_t jb, uint32_t je, unsigned long long* cursor,
                                              int path, int streams, int blocks, cudaStream_t s) {
  const bool two = streams == 2;
  switch (path) {
    case 0: return two ? launch_queue_t<0, 2>(b, jb, je, cursor, blocks, s) : launch_queue_t<0, 1>(b, jb, je, cursor, blocks, s);
    case 1: return two ? launch_queue_t<1, 2>(b, jb, je, cursor, blocks, s) : launch_queue_t<1, 1>(b, jb, je, cursor, blocks, s);
    case 2: return two ? launch_queue_t<2, 2>(b, jb, je, cursor, blocks, s) : launch_queue_t<2, 1>(b, jb, je, cursor, blocks, s);
    case 3: return two ? launch_queue_t<3, 2>(b, jb, je, cursor, blocks, s) : launch_queue_t<3, 1>(b, jb, je, cursor, blocks, s);
    default: return cudaErrorInvalidValue;
  }
}

int BBP_CAT(queue_occupancy_l, BBP_LMAX)(int path, int streams) {
  const bool two = streams == 2;
  switch (path) {
    case 0: return two ? queue_occupancy_t<0, 2>() : queue_occupancy_t<0, 1>();
    case 1: return two ? queue_occupancy_t<1, 2>() : queue_occupancy_t<1, 1>();
    case 2: return two ? queue_occupancy_t<2, 2>() : queue_occupancy_t<2, 1>();
    case 3: return two ? queue_occupancy_t<3, 2>() : queue_occupancy_t<3, 1>();
    default: return 1;
  }
}

}  // namespace bbp
