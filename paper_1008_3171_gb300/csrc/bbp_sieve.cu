// Segmented sieve for the prime form of a query (bbp_primes.h): which primes there are,
// as compact lists the prime kernels read.
#include <cuda_runtime.h>

#include <algorithm>

#include "bbp_device.cuh"
#include "bbp_finalize.cuh"
#include "bbp_sieve.cuh"

namespace bbp {

namespace {

// Odd primes below 67: their multiples are laid down as word patterns (no atomics).
__constant__ uint32_t kTiny[kSieveTinyPrimes] = {3, 5, 7, 11, 13, 17, 19, 23, 29, 31, 37, 41, 43, 47, 53, 59, 61};

// Bits o, o + p, o + 2p, ... of a word
__device__ __forceinline__ uint32_t comb(uint32_t p, uint32_t o) {
  uint32_t m = 0;
  for (; o < 32u; o += p) m |= 1u << o;
  return m;
}

__device__ __forceinline__ uint32_t mod_reciprocal(uint64_t v, uint32_t p, uint64_t inv) {
  const uint32_t r = lo32(v) - lo32(__umul64hi(v, inv)) * p;  // floor or one less: r < 2 p
  return r >= p ? r - p : r;
}

// Index (bit) of the first odd multiple of p at or after `base` (even): 2 i + 1 = -base mod p
__device__ __forceinline__ uint32_t first_multiple(uint64_t base, uint32_t p, uint64_t inv) {
  const uint32_t r = mod_reciprocal(base + 1, p, inv);
  if (r == 0u) return 0u;
  const uint32_t t = p - r;  // base + 1 + t is a multiple
  return (t & 1u ? t + p : t) >> 1;
}

// Bit i of the segment's words is the number base + 2 i + 1; a set bit is composite.
//
// What bounds it: shared-memory atomics (about 1.1 marks per odd number) and the first
// multiples, one reciprocal product per base prime and segment.  Primes below 67 would be
// two thirds of the marks; they go in as patterns, a word at a time.  Primes up to 32
// marks a segment take a warp each, larger ones a thread each.
__device__ void sieve_segment(uint64_t base, uint32_t words, uint64_t upto, const uint32_t* primes,
                              const uint64_t* inv, uint32_t nprimes, uint32_t* seg) {
  const uint32_t tid = threadIdx.x, lane = tid & 31u, wid = tid >> 5, nthreads = blockDim.x;
  for (uint32_t w = tid; w < words; w += nthreads) seg[w] = 0;
  for (int t = 0; t < kSieveTinyPrimes; ++t) {
    const uint32_t p = kTiny[t];
    // offset of the first multiple in word tid, then in steps of nthreads words
    const uint32_t step = (32u * nthreads) % p;
    const uint32_t r = static_cast<uint32_t>((base + 1 + 64ull * tid) % p);
    uint32_t o = r == 0u ? 0u : ((p - r) & 1u ? 2u * p - r : p - r) >> 1;
    const uint32_t pattern = comb(p, 0u);
    for (uint32_t w = tid; w < words; w += nthreads) {
      if (o < 32u) seg[w] |= pattern << o;
      o = o >= step ? o - step : o + p - step;
    }
  }
  __syncthreads();
  const uint32_t bits = 32u * words;
  const uint64_t end = min(base + 2 * static_cast<uint64_t>(bits), upto + 1);
  // warp-wide primes: at least 32 marks each
  uint32_t i = wid;
  for (; i < nprimes; i += nthreads >> 5) {
    const uint32_t p = primes[i];
    if (p > words || static_cast<uint64_t>(p) * p >= end) break;
    uint32_t at = first_multiple(base, p, inv[i]);
    const uint64_t sq = static_cast<uint64_t>(p) * p;
    if (sq > base) at = max(at, static_cast<uint32_t>((sq - base - 1) >> 1));  // smaller multiples have smaller factors
    for (uint32_t k = at + lane * p; k < bits; k += 32u * p) atomicOr(seg + (k >> 5), 1u << (k & 31u));
  }
  // the first prime above `words` (the list is ascending)
  uint32_t lo = 0, hi = nprimes;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (primes[mid] > words) hi = mid;
    else lo = mid + 1;
  }
  for (i = lo + tid; i < nprimes; i += nthreads) {
    const uint32_t p = primes[i];
    const uint64_t sq = static_cast<uint64_t>(p) * p;
    if (sq >= end) break;
    uint32_t at = first_multiple(base, p, inv[i]);
    if (sq > base) at = max(at, static_cast<uint32_t>((sq - base - 1) >> 1));
    for (uint32_t k = at; k < bits; k += p) atomicOr(seg + (k >> 5), 1u << (k & 31u));
  }
  __syncthreads();
}

// Set bits of ~seg whose number lies in (above, upto]: word w
__device__ __forceinline__ uint32_t prime_bits(uint64_t base, uint32_t w, uint64_t above, uint64_t upto,
                                               const uint32_t* seg) {
  uint32_t v = ~seg[w];
  const uint64_t first = base + 64ull * w + 1;  // number of bit 0
  if (first + 62 <= above || first > upto) return 0u;
  if (first <= above) {
    const uint32_t k = static_cast<uint32_t>((above - first) / 2 + 1);  // bits 0 .. k-1 are not above
    v &= k < 32u ? ~0u << k : 0u;
  }
  if (first + 62 > upto) {
    const uint32_t k = static_cast<uint32_t>((upto - first) / 2 + 1);
    if (k < 32u) v &= (1u << k) - 1u;
  }
  return v;
}

// Appends the segment's primes to the list in ascending order; one atomic per segment.
__device__ void emit_segment(uint64_t base, uint32_t words, uint64_t above, uint64_t upto, const uint32_t* seg,
                             uint64_t list_base, uint32_t* list, uint32_t* count, uint32_t cap) {
  __shared__ uint32_t start[kSieveThreads / 32 + 1];
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const uint32_t share = (words + nwarps - 1) / nwarps;
  const uint32_t w0 = wid * share, w1 = min(words, w0 + share);
  uint32_t mine = 0;
  for (uint32_t w = w0 + lane; w < w1; w += 32) mine += __popc(prime_bits(base, w, above, upto, seg));
  mine = __reduce_add_sync(0xffffffffu, mine);
  if (lane == 0) start[wid] = mine;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t total = 0;
    for (uint32_t k = 0; k < nwarps; ++k) {
      const uint32_t c = start[k];
      start[k] = total;
      total += c;
    }
    const uint32_t at = total ? atomicAdd(count, total) : 0u;
    for (uint32_t k = 0; k < nwarps; ++k) start[k] += at;
  }
  __syncthreads();
  uint32_t at = start[wid];
  for (uint32_t wb = w0; wb < w1; wb += 32) {
    const uint32_t w = wb + lane;
    uint32_t v = w < w1 ? prime_bits(base, w, above, upto, seg) : 0u;
    const uint32_t c = __popc(v);
    uint32_t sum = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(0xffffffffu, sum, d);
      if (lane >= static_cast<uint32_t>(d)) sum += o;
    }
    uint32_t k = at + sum - c;
    const uint32_t off = static_cast<uint32_t>(base - list_base) + 64u * w + 1u;
    while (v) {
      const uint32_t b = __ffs(static_cast<int>(v)) - 1;
      v &= v - 1;
      if (k < cap) list[k] = off + 2u * b;
      ++k;
    }
    at += __shfl_sync(0xffffffffu, sum, 31);
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kSieveThreads) sieve_kernel(const SieveArgs a) {
  extern __shared__ uint32_t seg[];
  const uint32_t n = *a.nprimes;
  for (uint32_t s = blockIdx.x; s < a.segments; s += gridDim.x) {
    const uint64_t base = a.base + 64ull * a.words * s;
    if (base > a.upto) break;
    sieve_segment(base, a.words, a.upto, a.primes, a.inv, n, seg);
    emit_segment(base, a.words, a.above, a.upto, seg, a.base, a.list, a.count, a.cap);
  }
}

// The base primes, by one CTA: primes below 67 are known, those up to 4096 come from a
// sieve by them, the rest from a sieve by those.
__global__ void __launch_bounds__(kSieveThreads) base_primes_kernel(uint32_t upto, uint32_t* primes, uint64_t* inv,
                                                                    uint32_t* count, uint32_t* nsieve) {
  extern __shared__ uint32_t seg[];
  const uint32_t tid = threadIdx.x;
  if (tid < kSieveTinyPrimes) {
    primes[tid] = kTiny[tid];
    inv[tid] = ~0ull / kTiny[tid];
  }
  if (tid == 0) *count = kSieveTinyPrimes;
  __syncthreads();
  uint32_t above = 66;
  uint64_t base = 0;
  while (above < upto) {
    // sieving by the primes found so far reaches up to the square of the next one
    const uint32_t known = above;
    const uint32_t reach = above < 4095u ? min(upto, 4095u) : upto;
    const uint32_t words = static_cast<uint32_t>(min(static_cast<uint64_t>(kSieveMaxWords), (reach - base) / 64 + 1));
    const uint64_t last = min(static_cast<uint64_t>(reach), base + 64 * static_cast<uint64_t>(words) - 1);
    const uint32_t n = *reinterpret_cast<volatile uint32_t*>(count);
    sieve_segment(base, words, last, primes + kSieveTinyPrimes, inv + kSieveTinyPrimes, n - kSieveTinyPrimes, seg);
    emit_segment(base, words, known, last, seg, 0, primes, count, ~0u);
    const uint32_t m = *reinterpret_cast<volatile uint32_t*>(count);
    __threadfence_block();
    for (uint32_t i = n + tid; i < m; i += blockDim.x) inv[i] = ~0ull / primes[i];
    __syncthreads();
    above = static_cast<uint32_t>(last);
    base = (last + 1) / 64 * 64;
  }
  if (tid == 0) *nsieve = *reinterpret_cast<volatile uint32_t*>(count) - kSieveTinyPrimes;
}

__global__ void prime_check_kernel(const unsigned long long* slots, int L, uint32_t P, uint64_t bound,
                                   const uint32_t* counts, uint32_t nlists, uint32_t cap, uint8_t* out,
                                   uint32_t* valid, uint32_t* redo) {
  const uint32_t lane = threadIdx.x;
  bool over = false;
  for (uint32_t i = lane; i < nlists; i += 32) over |= counts[i] > cap;
  over = __any_sync(0xffffffffu, over);
  if (lane != 0) return;
  uint32_t S[kMaxLimbs], neg[kMaxLimbs];
  uint64_t carry = 0, ncarry = 1;
  for (int i = 0; i < L; ++i) {
    const uint64_t v = __ldcg(slots + i) + carry;
    S[i] = lo32(v);
    carry = v >> 32;
    const uint64_t w = static_cast<uint64_t>(~S[i]) + ncarry;
    neg[i] = lo32(w);
    ncarry = w >> 32;
  }
  const int low = 32 * L - static_cast<int>(P);
  const bool stands = !over && low_bits_at_least(S, low, 3 * bound) && low_bits_at_least(neg, low, 3 * bound);
  *redo = stands ? 0u : 1u;
  if (stands) finalize_into(slots, L, P, 0, out, valid, nullptr);
}

}  // namespace

int sieve_occupancy(int words) {
  const size_t smem = sizeof(uint32_t) * static_cast<size_t>(words);
  if (cudaFuncSetAttribute(sieve_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(sizeof(uint32_t) * kSieveMaxWords)) != cudaSuccess)
    return 1;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, sieve_kernel, kSieveThreads, smem) != cudaSuccess) return 1;
  return std::max(1, n);
}

cudaError_t launch_sieve(const SieveArgs& a, int blocks, cudaStream_t s) {
  sieve_kernel<<<blocks, kSieveThreads, sizeof(uint32_t) * a.words, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_base_primes(uint32_t upto, uint32_t* primes, uint64_t* inv, uint32_t* count, uint32_t* nsieve,
                               cudaStream_t s) {
  const int smem = static_cast<int>(sizeof(uint32_t) * kSieveMaxWords);
  const cudaError_t e = cudaFuncSetAttribute(base_primes_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  base_primes_kernel<<<1, kSieveThreads, smem, s>>>(upto, primes, inv, count, nsieve);
  return cudaGetLastError();
}

cudaError_t launch_prime_check(const unsigned long long* slots, int L, uint32_t P, uint64_t bound,
                               const uint32_t* counts, uint32_t nlists, uint32_t cap, uint8_t* out, uint32_t* valid,
                               uint32_t* redo, cudaStream_t s) {
  prime_check_kernel<<<1, 32, 0, s>>>(slots, L, P, bound, counts, nlists, cap, out, valid, redo);
  return cudaGetLastError();
}

}  // namespace bbp
