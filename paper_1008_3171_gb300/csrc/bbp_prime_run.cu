// Runs the prime form of a query's head sum (bbp_primes.h) on a plan: base primes, the
// prime powers with long sums, then the primes up to n in lists of bounded length, each
// sieved and summed.  Two list buffers and three streams: the caller's stream sums a list
// while the next is sieved on a second one, and the prime powers run on a third.
//
// Measured on a GB300, whole bbp_bits calls, term by term -> by primes: n = 1e9, P = 128:
// 15.6 -> 1.75 ms; n = 1e9, P = 64 by Eq. 1: 20.5 -> 2.54 ms; n = 3e8, P = 1000:
// 7.88 -> 0.91 ms; n = 4e10, P = 256: 1005 -> 82.3 ms.  At 4e10 the kernels one after
// another: 56.1 ms primes above A / 23, 14.3 those below, 4.0 prime powers, 13.9 sieve.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "bbp_planner.h"
#include "bbp_prime_run.h"
#include "bbp_sieve.cuh"

namespace bbp {

namespace {

constexpr uint32_t kBaseCap = 565000;               // odd primes below 2^23: 564,162
// At the largest position lists of 6 M primes number 7.3e4 for Eq. 2 and 1.46e5 for Eq. 1, whose
// moduli reach 2 n (152 SMs; 1.9e5 at most from 120 to 160).
constexpr uint32_t kMaxLists = 1u << 18;
constexpr uint32_t kSieveEntries = 64u << 10;       // of a sieve segment: three CTAs an SM
constexpr uint64_t kLongSum = 8000, kGroupSum = 1000;  // primes below A / these take 32, 8 lanes

uint64_t isqrt(uint64_t v) {
  uint64_t r = static_cast<uint64_t>(std::sqrt(static_cast<double>(v)));
  while (r * r > v) --r;
  while ((r + 1) * (r + 1) <= v) ++r;
  return r;
}

}  // namespace

}  // namespace bbp

// Device memory, streams and events of one query at a time.
struct PrimeState {
  uint32_t* list[2] = {};
  uint32_t list_cap = 0;
  // A capture has recorded the lists: a graph may be replayed while the plan lives, so lists
  // that are replaced by longer ones are kept until it goes.  Those are at least twice as long
  // then, from 1.1e6 to 2.5e7 primes: no more than kKeptLists are ever kept, together less than
  // twice the longest.
  static constexpr int kKeptLists = 12;
  bool captured = false;
  int nkept = 0;
  uint32_t* kept[kKeptLists] = {};
  uint32_t* primes = nullptr;  // base primes
  bbp::SievePrime* sieve_primes = nullptr;
  // [0] base primes, [1] those from 17 on; then the length of each list, then the primes of
  // each handed out so far
  uint32_t* counts = nullptr;
  cudaStream_t sieve = nullptr, sums = nullptr;  // beside the caller's stream
  cudaEvent_t ready[2] = {}, used[2] = {}, base = nullptr, done = nullptr;
  cudaEvent_t idle = nullptr;   // the last run that was not captured, on
  cudaStream_t last = nullptr;  // this stream
  bool ran = false;
};

namespace bbp {

namespace {
constexpr size_t kCountHead = 4;

bool make_state(PrimeState* s) {
  int low = 0, high = 0;
  bool ok = cudaDeviceGetStreamPriorityRange(&low, &high) == cudaSuccess &&
            cudaStreamCreateWithPriority(&s->sieve, cudaStreamNonBlocking, high) == cudaSuccess &&
            cudaStreamCreateWithPriority(&s->sums, cudaStreamNonBlocking, high) == cudaSuccess &&
            cudaMalloc(&s->primes, sizeof(uint32_t) * kBaseCap) == cudaSuccess &&
            cudaMalloc(&s->sieve_primes, sizeof(SievePrime) * kBaseCap) == cudaSuccess &&
            cudaMalloc(&s->counts, sizeof(uint32_t) * (kCountHead + 2 * kMaxLists)) == cudaSuccess;
  auto event = [&](cudaEvent_t* e) {
    ok = ok && cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess;
  };
  for (cudaEvent_t& e : s->ready) event(&e);
  for (cudaEvent_t& e : s->used) event(&e);
  event(&s->base);
  event(&s->done);
  event(&s->idle);
  return ok;
}
}  // namespace

void wait_prime_state(PrimeState* s) {
  if (!s) return;
  if (s->sieve) cudaStreamSynchronize(s->sieve);
  if (s->sums) cudaStreamSynchronize(s->sums);
}

void release_prime_state(PrimeState** state) {
  PrimeState* s = *state;
  if (!s) return;
  wait_prime_state(s);
  for (cudaEvent_t e : s->ready)
    if (e) cudaEventDestroy(e);
  for (cudaEvent_t e : s->used)
    if (e) cudaEventDestroy(e);
  if (s->base) cudaEventDestroy(s->base);
  if (s->done) cudaEventDestroy(s->done);
  if (s->idle) cudaEventDestroy(s->idle);
  if (s->sieve) cudaStreamDestroy(s->sieve);
  if (s->sums) cudaStreamDestroy(s->sums);
  for (uint32_t* l : s->list) cudaFree(l);
  for (uint32_t* l : s->kept) cudaFree(l);
  cudaFree(s->primes);
  cudaFree(s->sieve_primes);
  cudaFree(s->counts);
  delete s;
  *state = nullptr;
}

// Lets this thread allocate while some other stream is being captured, which a capture in the
// default mode forbids and would not survive: queries that allocate nothing but at a plan's
// first use are called beside captures.
class AllocateBesideCaptures {
 public:
  AllocateBesideCaptures() { cudaThreadExchangeStreamCaptureMode(&mode_); }
  ~AllocateBesideCaptures() { cudaThreadExchangeStreamCaptureMode(&mode_); }
  AllocateBesideCaptures(const AllocateBesideCaptures&) = delete;

 private:
  cudaStreamCaptureMode mode_ = cudaStreamCaptureModeRelaxed;
};

bool prime_workspace(PrimeState** state, uint64_t n, uint32_t max_list, cudaStream_t st) {
  // primes of one list: all of them up to the limit
  const double x = static_cast<double>(n);
  uint32_t want = static_cast<uint32_t>(std::min<double>(max_list, 1.2 * x / std::log(x) + 4096.0));
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const bool capturing = cap != cudaStreamCaptureStatusNone;
  if (*state && (*state)->list_cap >= want) {
    (*state)->captured |= capturing;
    return true;
  }
  if (capturing) return false;
  const AllocateBesideCaptures guard;
  if (!*state) {
    *state = new (std::nothrow) PrimeState();
    if (!*state) return false;
    if (!make_state(*state)) {
      cudaGetLastError();
      release_prime_state(state);
      return false;
    }
  }
  PrimeState* s = *state;
  if (s->captured) {
    if (s->nkept + 2 > PrimeState::kKeptLists) return false;
    want = std::max(want, std::min(max_list, 2 * s->list_cap));
    for (uint32_t*& l : s->list) {
      s->kept[s->nkept++] = l;
      l = nullptr;
    }
    s->captured = false;
  }
  s->list_cap = 0;
  for (uint32_t*& l : s->list) {
    cudaFree(l);  // waits for the work that reads it
    l = nullptr;
    if (cudaMalloc(&l, sizeof(uint32_t) * want) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
  }
  s->list_cap = want;
  return true;
}

bbp_status PrimeRun::plan(PrimeState* state, int sm_count, int formula, uint64_t n, uint32_t W,
                          unsigned long long* slots) {
  state_ = state;
  sms_ = sm_count;
  formula_ = formula;
  launches_ = 0;
  lists_.clear();
  lmax_ = head_lmax_for(static_cast<int>(W / 32));
  if (lmax_ == 0) return BBP_EINVAL;
  const PrimeLimits lim = prime_limits(formula, n - 1);
  const std::vector<PrimeClass> classes = prime_classes(lim);
  if (classes.empty() || classes.size() > static_cast<size_t>(kMaxPrimeClasses)) return BBP_EINVAL;
  PrimeArgs& a = args_;
  a = PrimeArgs{};
  a.L = W / 32;
  a.A = lim.A;
  a.B = lim.B;
  a.C = lim.C;
  a.slots = slots;
  a.nclasses = static_cast<uint32_t>(classes.size());
  std::copy(classes.begin(), classes.end(), a.classes);
  e_ = n - 1 + W;
  const uint64_t root = isqrt(lim.A);
  base_to_ = static_cast<uint32_t>(root);  // below 2^23
  const uint64_t bottom = classes.back().above;
  // lists: primes in (base_to, A], cut where their kernel changes
  struct Span { uint64_t lo, hi; PrimeKernel k; };
  std::vector<Span> spans;
  {
    const uint64_t one_word = (1ull << 31) - 1;
    // a list of its own pays from about n = 6e8 on
    const uint64_t shared32 = lim.A / kLongSum > 3 * root ? std::min(lim.A / kLongSum, one_word) : 0;
    const uint64_t shared8 = std::min(lim.A / kGroupSum, one_word);
    const uint64_t cuts[] = {shared32, shared8, bottom, (1ull << 29) - 1, (1ull << 31) - 1, kPrimeHalfMax,
                             formula == 1 ? lim.B : lim.A, lim.A};
    std::vector<uint64_t> c(std::begin(cuts), std::end(cuts));
    std::sort(c.begin(), c.end());
    uint64_t lo = base_to_;
    for (uint64_t hi : c) {
      hi = std::min(hi, lim.A);
      if (hi <= lo) continue;
      PrimeKernel k;
      if (hi <= bottom) k = hi <= shared32 ? kSums32 : hi <= shared8 ? kSums8 : hi <= one_word ? kSums1 : kSums2;
      else k = hi < (1ull << 29) ? kPrimes0 : hi < (1ull << 31) ? kPrimes3 : hi <= kPrimeHalfMax ? kPrimesHalf : kPrimes1;
      spans.push_back(Span{lo, hi, k});
      lo = hi;
    }
  }
  constexpr uint64_t seg = 30ull * kSieveEntries;
  for (const Span& s : spans) {
    uint64_t lo = s.lo;
    while (lo < s.hi) {
      const uint64_t base = (lo + 1) / seg * seg;
      // about 1 / ln x of the numbers are primes; a list that came out longer than the buffer
      // would be seen by the check
      const double room = 0.85 * state_->list_cap * (std::log(static_cast<double>(std::max<uint64_t>(lo, 1000))) - 1.1);
      uint64_t nseg = std::max<uint64_t>(1, static_cast<uint64_t>(room) / seg);
      // whole waves of the sieve's CTAs, eight a segment, one an SM beside the primes' kernels
      const uint64_t wave = std::max<uint64_t>(1, static_cast<uint64_t>(sms_) / 8);
      if (nseg > wave) nseg -= nseg % wave;
      const uint64_t hi = std::min(s.hi, base + nseg * seg - 1);
      // Eq. 1 above B: c = 1 alone, which only p = 1 mod 4 has
      lists_.push_back(List{base, lo, hi, static_cast<uint32_t>((hi - base) / seg + 1), s.k,
                            formula == 1 && lo >= lim.B ? 1u : 0u});
      lo = hi;
    }
  }
  return lists_.size() > kMaxLists ? BBP_ERANGE : BBP_OK;
}

double PrimeRun::share(size_t i) const {
  return static_cast<double>(lists_[i].hi - lists_[i].lo) / static_cast<double>(args_.A);
}

// The caller's stream runs the lists' kernels, the sieve runs one list ahead on its own
// stream, the prime powers (few, with long chains) run beside them on a third.
bbp_status PrimeRun::begin(cudaStream_t st) {
  PrimeState* const S = state_;
  cudaError_t err = cudaSuccess;
  auto chk = [&](cudaError_t r) { if (err == cudaSuccess) err = r; };
  // a run on another stream may still read the lists that this one writes
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  chk(cudaStreamIsCapturing(st, &cap));
  captured_ = cap != cudaStreamCaptureStatusNone;
  if (S->ran && S->last != st && !captured_) chk(cudaStreamWaitEvent(st, S->idle, 0));
  chk(cudaMemsetAsync(S->counts, 0, sizeof(uint32_t) * (kCountHead + 2 * lists_.size()), st));
  chk(launch_base_primes(base_to_, S->primes, S->sieve_primes, S->counts, S->counts + 1, st));
  chk(cudaEventRecord(S->base, st));
  chk(cudaStreamWaitEvent(S->sieve, S->base, 0));
  chk(cudaStreamWaitEvent(S->sums, S->base, 0));
  PrimeArgs a = args_;
  a.list = S->primes;
  a.count = S->counts;
  a.cap = kBaseCap;
  a.e = e_;
  const bool above_word = a.A >= (1ull << 31);
  chk(launch_prime(a, kPowers1, formula_, lmax_, sms_, S->sums));
  if (above_word) chk(launch_prime(a, kPowers2, formula_, lmax_, sms_, S->sums));
  chk(launch_prime(a, kPrimeWarps, formula_, lmax_, sms_, S->sums));
  chk(cudaEventRecord(S->done, S->sums));
  launches_ += above_word ? 4 : 3;
  return err == cudaSuccess ? BBP_OK : BBP_ECUDA;
}

bbp_status PrimeRun::run(size_t first, size_t last, cudaStream_t st) {
  PrimeState* const S = state_;
  cudaError_t err = cudaSuccess;
  auto chk = [&](cudaError_t r) { if (err == cudaSuccess) err = r; };
  uint32_t* const lengths = S->counts + kCountHead;
  SieveArgs v{};
  v.entries = kSieveEntries;
  v.primes = S->sieve_primes + kSieveTinyPrimes;
  v.nprimes = S->counts + 1;
  v.cap = S->list_cap;
  PrimeArgs a = args_;
  a.cap = S->list_cap;
  for (size_t i = first; i < last; ++i) {
    const List& l = lists_[i];
    const size_t slot = i & 1;
    if (i >= 2) chk(cudaStreamWaitEvent(S->sieve, S->used[slot], 0));  // the buffer's last list is done
    v.list = S->list[slot];
    v.base = l.base;
    v.above = l.lo;
    v.upto = l.hi;
    v.segments = l.segments;
    v.one_mod_4 = l.one_mod_4;
    v.count = lengths + i;
    chk(launch_sieve(v, sms_, S->sieve));
    chk(cudaEventRecord(S->ready[slot], S->sieve));
    chk(cudaStreamWaitEvent(st, S->ready[slot], 0));
    a.list = S->list[slot];
    a.base = l.base;
    a.count = lengths + i;
    a.taken = lengths + lists_.size() + i;
    const bool sums = l.kernel == kSums1 || l.kernel == kSums2 || l.kernel == kSums8 || l.kernel == kSums32;
    a.e = sums ? e_ : e_ - kPrimeShift + 64;  // the product with H leaves a factor 2^-64
    chk(launch_prime(a, l.kernel, formula_, lmax_, sms_, st));
    chk(cudaEventRecord(S->used[slot], st));
    launches_ += 3;
  }
  return err == cudaSuccess ? BBP_OK : BBP_ECUDA;
}

bbp_status PrimeRun::finish(uint32_t P, uint64_t bound, uint8_t* d_out, uint32_t* d_valid, uint32_t* d_redo,
                            cudaStream_t st) {
  cudaError_t err = cudaStreamWaitEvent(st, state_->done, 0);
  if (err == cudaSuccess)
    err = launch_prime_check(args_.slots, static_cast<int>(args_.L), P, bound, state_->counts + kCountHead,
                             static_cast<uint32_t>(lists_.size()), state_->list_cap, d_out, d_valid, d_redo, st);
  ++launches_;
  if (!captured_) {
    if (err == cudaSuccess) err = cudaEventRecord(state_->idle, st);
    state_->last = st;
    state_->ran = err == cudaSuccess;
  }
  return err == cudaSuccess ? BBP_OK : BBP_ECUDA;
}

}  // namespace bbp
