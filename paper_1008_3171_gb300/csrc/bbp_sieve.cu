// Segmented sieve for the prime form of a query (bbp_primes.h): which primes there are,
// as compact lists the prime kernels read.
#include <cuda_runtime.h>

#include <algorithm>

#include "bbp_device.cuh"
#include "bbp_finalize.cuh"
#include "bbp_sieve.cuh"

namespace bbp {

namespace {

// Odd primes below 17: their multiples are laid down as bit patterns.
constexpr uint32_t kTiny[kSieveTinyPrimes] = {3, 5, 7, 11, 13};
__constant__ uint32_t kTinyDev[kSieveTinyPrimes] = {3, 5, 7, 11, 13};
__constant__ uint32_t kWheel[8] = {1, 7, 11, 13, 17, 19, 23, 29};

// Bits 0, p, 2p, ... of a word
__host__ __device__ constexpr uint32_t comb(uint32_t p) {
  uint32_t m = 0;
  for (uint32_t o = 0; o < 32u; o += p) m |= 1u << o;
  return m;
}

// A segment is the progression first, first + STEP, ... : entry i, a byte of shared
// memory, is first + STEP i.  Either the odd numbers (STEP 2) or one of the eight classes
// prime to 30 (STEP 30), which has 8 / 15 of the entries and so of the marks of a sieve
// of the odd numbers, and needs no multiples of 3 and 5.

// v mod p
__device__ __forceinline__ uint32_t mod_prime(uint32_t v, const SievePrime& s) {
  const uint32_t r = v - __umulhi(v, s.inv) * s.p;  // the quotient is right or one less: r < 2 p
  return min(r, r - s.p);
}

// First entry of class r, `skipped` entries after the list's base, that is a multiple of p:
// i = -(base + 30 skipped + r) / 30 mod p.  skipped < 2^28, r inv30 < 2^28.
__device__ __forceinline__ uint32_t first_multiple(const SievePrime& s, uint32_t skipped, uint32_t r) {
  const uint32_t x = s.at - mod_prime(skipped + r * s.inv30, s);
  return min(x, x + s.p);
}

// First odd number from `first` (odd, below 2^24) on that is a multiple of p, from p^2 on
__device__ __forceinline__ uint32_t first_odd_multiple(const SievePrime& s, uint32_t first) {
  const uint64_t sq = static_cast<uint64_t>(s.p) * s.p;
  if (sq >= first) return static_cast<uint32_t>(sq - first) / 2;
  const uint32_t r = mod_prime(first, s);
  const uint32_t t = r ? s.p - r : 0u;
  return (t & 1u ? t + s.p : t) >> 1;
}

// Multiples of tiny prime number K and up among the entries 32 w ... 32 w + 31, as bits.
// tiny[k]: the first entry that is a multiple of the k-th tiny prime.
template <int K>
__device__ __forceinline__ uint32_t tiny_word(const uint32_t* tiny, uint32_t w) {
  if constexpr (K < kSieveTinyPrimes) {
    constexpr uint32_t p = kTiny[K], shift = 32u % p;
    const uint32_t o = (tiny[K] + (p - shift) * w) % p;  // first multiple from 32 w on
    return (o < 32u ? comb(p) << o : 0u) | tiny_word<K + 1>(tiny, w);
  } else {
    return 0u;
  }
}

// Marks the entries with a base prime factor (possibly the prime itself, but from its
// square on for STEP 2), and works out where the tiny primes' multiples start.  `skipped`
// and `cls`: see first_multiple (STEP 30).
//
// What bounds it: instruction issue -- about 1.7 marks an entry, and the first multiples.
// An entry is a byte so that a mark is a plain store (a bit an entry takes a shared-memory
// atomic, about one lane a clock and SM).  A first multiple is one 32-bit reduction: the
// part that depends on the list is worked out once per list.  First multiples are taken
// one prime a lane, the marks of a prime up to 149 by the whole CTA, of one with at least
// 32 marks by a warp, of a larger one by its thread.
template <int STEP>
__device__ void sieve_segment(uint64_t first, uint32_t skipped, uint32_t cls, uint32_t entries, uint64_t upto,
                              const SievePrime* primes, uint32_t nprimes, uint8_t* seg, uint32_t* tiny) {
  constexpr uint32_t kShared = 32;  // primes from 17 to 157
  __shared__ uint2 shared_at[kShared];
  __shared__ uint32_t used, warped;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, wid = tid >> 5, nthreads = blockDim.x, nwarps = nthreads >> 5;
  const uint64_t end = min(first + STEP * static_cast<uint64_t>(entries), upto + 1);
  auto start = [&](const SievePrime& s) {
    return STEP == 30 ? first_multiple(s, skipped, cls) : first_odd_multiple(s, static_cast<uint32_t>(first));
  };
  auto load = [&](uint32_t i) {
    const uint4 v = *reinterpret_cast<const uint4*>(primes + i);
    return SievePrime{v.x, v.y, v.z, v.w};
  };
  if (tid < kSieveTinyPrimes) {
    const uint32_t p = kTinyDev[tid];
    uint32_t x = static_cast<uint32_t>(first % p), i = 0;
    for (; i < p && x != 0u; ++i) x = (x + STEP) % p;  // i = p: no multiples (3 and 5 in the classes prime to 30)
    tiny[tid] = i;
  }
  if (tid == 32 || tid == 64) {  // primes whose square is below `end`; primes with 32 marks
    uint32_t lo = 0, hi = nprimes;
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1, p = primes[mid].p;
      if (tid == 32 ? static_cast<uint64_t>(p) * p >= end : p > entries / 32) hi = mid;
      else lo = mid + 1;
    }
    (tid == 32 ? used : warped) = lo;
  }
  for (uint32_t w = tid; w < entries / 16; w += nthreads) reinterpret_cast<uint4*>(seg)[w] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  const uint32_t n = used;
  const uint32_t n0 = min(n, kShared), n1 = max(n0, min(n, warped));
  if (tid < n0) {
    const SievePrime s = load(tid);
    shared_at[tid] = make_uint2(s.p, start(s));
  }
  __syncthreads();
  for (uint32_t i = 0; i < n0; ++i) {
    const uint2 s = shared_at[i];
    for (uint32_t k = s.y + tid * s.x; k < entries; k += nthreads * s.x) seg[k] = 1;
  }
  // warp w takes primes w, w + nwarps, ...: 32 of them at a time, one lane each for the start
  for (uint32_t b = n0 + wid; b < n1; b += 32 * nwarps) {
    const uint32_t mine = b + lane * nwarps;
    const SievePrime s = load(min(mine, n1 - 1));
    const uint32_t p_l = mine < n1 ? s.p : 0u, at_l = start(s);
    for (uint32_t j = 0; j < 32; ++j) {
      const uint32_t p = __shfl_sync(0xffffffffu, p_l, j);
      if (p == 0u) break;
      for (uint32_t k = __shfl_sync(0xffffffffu, at_l, j) + lane * p; k < entries; k += 32u * p) seg[k] = 1;
    }
  }
#pragma unroll 2
  for (uint32_t i = n1 + tid; i < n; i += nthreads) {
    const SievePrime s = load(i);
    for (uint32_t k = start(s); k < entries; k += s.p) seg[k] = 1;
  }
  __syncthreads();
}

// 32 entries as bits: a set bit is a marked one
__device__ __forceinline__ uint32_t pack_entries(const uint8_t* seg, uint32_t w) {
  const uint4 a = reinterpret_cast<const uint4*>(seg)[2 * w], b = reinterpret_cast<const uint4*>(seg)[2 * w + 1];
  // bytes 0 or 1: the product gathers the four low bits in the top byte's low nibble
  auto four = [](uint32_t v) { return (v * 0x10204080u) >> 28; };
  const uint32_t lo = four(a.x) | four(a.y) << 4 | four(a.z) << 8 | four(a.w) << 12;
  const uint32_t hi = four(b.x) | four(b.y) << 4 | four(b.z) << 8 | four(b.w) << 12;
  return lo | hi << 16;
}

// Primes among the entries 32 w ... 32 w + 31 that lie in (above, upto]
template <int STEP>
__device__ __forceinline__ uint32_t prime_bits(uint64_t first, uint32_t w, uint64_t above, uint64_t upto,
                                               const uint8_t* seg, const uint32_t* tiny) {
  uint32_t v = ~(pack_entries(seg, w) | tiny_word<STEP == 30 ? 2 : 0>(tiny, w));
  const uint64_t lo = first + 32ull * STEP * w;  // number of bit 0
  if (lo + 31 * STEP <= above || lo > upto) return 0u;
  if (lo <= above) v &= ~0u << (static_cast<uint32_t>(above - lo) / STEP + 1);  // at most 31
  if (lo + 31 * STEP > upto) v &= (2u << (static_cast<uint32_t>(upto - lo) / STEP)) - 1u;  // at most 30
  return v;
}

// Appends the segment's primes, less `origin`, to the list in ascending order; one atomic
// per segment: those in the bits `keep` of every 32 entries.  The bits of a word replace its
// entries for the second pass.
template <int STEP>
__device__ void emit_segment(uint64_t first, uint32_t entries, uint64_t above, uint64_t upto, uint8_t* seg,
                             const uint32_t* tiny, uint32_t keep, uint64_t origin, uint32_t* list, uint32_t* count,
                             uint32_t cap) {
  __shared__ uint32_t start[kSieveThreads / 32 + 1];
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, nwarps = blockDim.x >> 5, words = entries / 32;
  const uint32_t share = (words + nwarps - 1) / nwarps;
  const uint32_t w0 = wid * share, w1 = min(words, w0 + share);
  uint32_t mine = 0;
  for (uint32_t w = w0 + lane; w < w1; w += 32) {
    const uint32_t v = prime_bits<STEP>(first, w, above, upto, seg, tiny) & keep;
    reinterpret_cast<uint32_t*>(seg)[8 * w] = v;
    mine += __popc(v);
  }
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
    uint32_t v = w < w1 ? reinterpret_cast<const uint32_t*>(seg)[8 * w] : 0u;
    const uint32_t c = __popc(v);
    uint32_t sum = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(0xffffffffu, sum, d);
      if (lane >= static_cast<uint32_t>(d)) sum += o;
    }
    const uint32_t k = at + sum - c;
    const uint32_t off = static_cast<uint32_t>(first - origin) + 32u * STEP * w;
    if (k > cap || c > cap - k) v = 0;  // does not fit: the count says so
    for (uint32_t* to = list + k; v; ++to) {
      *to = off + STEP * (31u - static_cast<uint32_t>(__clz(static_cast<int>(v & (0u - v)))));
      v &= v - 1;
    }
    at += __shfl_sync(0xffffffffu, sum, 31);
  }
  __syncthreads();
}

// `at` of every base prime for the list from `base`
__global__ void sieve_offsets_kernel(SievePrime* primes, const uint32_t* nprimes, uint64_t base) {
  const uint32_t n = *nprimes;
  const uint64_t b = base / 30;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t p = primes[i].p;
    const uint32_t r = static_cast<uint32_t>(b % p);
    primes[i].at = r ? p - r : 0u;
  }
}

// One CTA per class and segment
__global__ void __launch_bounds__(kSieveThreads, 4) sieve_kernel(const SieveArgs a) {
  extern __shared__ __align__(16) uint8_t seg[];
  __shared__ uint32_t tiny[kSieveTinyPrimes];
  const uint32_t skipped = a.entries * (blockIdx.x >> 3), cls = kWheel[blockIdx.x & 7u];
  const uint64_t first = a.base + 30ull * skipped + cls;
  if (first > a.upto) return;
  sieve_segment<30>(first, skipped, cls, a.entries, a.upto, a.primes, *a.nprimes, seg, tiny);
  // 30 i + first mod 4 alternates
  const uint32_t keep = a.one_mod_4 == 0u ? ~0u : (first & 3u) == 1u ? 0x55555555u : 0xaaaaaaaau;
  emit_segment<30>(first, a.entries, a.above, a.upto, seg, tiny, keep, a.base, a.list, a.count, a.cap);
}

// The base primes, by one CTA: primes below 17 are known, those up to 256 come from a
// sieve by them, those up to 65536 from a sieve by those, the rest from a sieve by all.
__global__ void __launch_bounds__(kSieveThreads) base_primes_kernel(uint32_t upto, uint32_t* primes, SievePrime* sieve,
                                                                    uint32_t* count, uint32_t* nsieve) {
  extern __shared__ __align__(16) uint8_t seg[];
  __shared__ uint32_t tiny[kSieveTinyPrimes];
  const uint32_t tid = threadIdx.x;
  if (tid < kSieveTinyPrimes) primes[tid] = kTinyDev[tid];
  if (tid == 0) *count = kSieveTinyPrimes;
  __syncthreads();
  uint32_t above = 16;
  uint64_t base = 0;
  while (above < upto) {
    // sieving by the primes up to `above` reaches its square
    const uint32_t known = above;
    const uint32_t reach = above < 65536u ? min(upto, above * above) : upto;
    const uint32_t entries = static_cast<uint32_t>(min(static_cast<uint64_t>(kSieveMaxEntries),
                                                       (reach - base) / 64 * 32 + 32));
    const uint64_t last = min(static_cast<uint64_t>(reach), base + 2 * static_cast<uint64_t>(entries) - 1);
    const uint32_t n = *reinterpret_cast<volatile uint32_t*>(count);
    sieve_segment<2>(base + 1, 0, 0, entries, last, sieve + kSieveTinyPrimes, n - kSieveTinyPrimes, seg, tiny);
    emit_segment<2>(base + 1, entries, known, last, seg, tiny, ~0u, 0, primes, count, ~0u);
    const uint32_t m = *reinterpret_cast<volatile uint32_t*>(count);
    for (uint32_t i = n + tid; i < m; i += blockDim.x) {
      const uint32_t p = primes[i];
      uint32_t t = 0;  // 30^-1 = (1 + t p) / 30
      while (t < 30u && (1u + t * (p % 30u)) % 30u != 0u) ++t;
      sieve[i] = SievePrime{p, ~0u / p, static_cast<uint32_t>((1 + static_cast<uint64_t>(t) * p) / 30), 0u};
    }
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

cudaError_t launch_sieve(const SieveArgs& a, int sms, cudaStream_t s) {
  const int smem = static_cast<int>(kSieveMaxEntries);
  const cudaError_t e = cudaFuncSetAttribute(sieve_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  sieve_offsets_kernel<<<sms, 256, 0, s>>>(a.primes, a.nprimes, a.base);
  sieve_kernel<<<8 * a.segments, kSieveThreads, a.entries, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_base_primes(uint32_t upto, uint32_t* primes, SievePrime* sieve, uint32_t* count, uint32_t* nsieve,
                               cudaStream_t s) {
  const int smem = static_cast<int>(kSieveMaxEntries);
  const cudaError_t e = cudaFuncSetAttribute(base_primes_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  base_primes_kernel<<<1, kSieveThreads, smem, s>>>(upto, primes, sieve, count, nsieve);
  return cudaGetLastError();
}

cudaError_t launch_prime_check(const unsigned long long* slots, int L, uint32_t P, uint64_t bound,
                               const uint32_t* counts, uint32_t nlists, uint32_t cap, uint8_t* out, uint32_t* valid,
                               uint32_t* redo, cudaStream_t s) {
  prime_check_kernel<<<1, 32, 0, s>>>(slots, L, P, bound, counts, nlists, cap, out, valid, redo);
  return cudaGetLastError();
}

}  // namespace bbp
