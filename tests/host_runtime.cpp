// The library's host runtime (plans, queries by primes, batches, serving) on a CUDA runtime
// that only keeps books: which allocations live, which operation of a stream comes after
// which, what a capture has recorded.  Kernels do nothing.  Run with the name of a case;
// exits 0 if it holds (test_host_runtime.py).
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <random>
#include <set>
#include <string>
#include <thread>
#include <vector>

#include "bbp.h"
#include "bbp_kernels.cuh"
#include "bbp_primes.h"
#include "bbp_sieve.cuh"

namespace {

std::recursive_mutex mu;  // the serving engine has a thread of its own

struct Op {
  std::string what;
  std::vector<size_t> after;
  std::vector<const void*> reads;
  bool captured = false, complete = false;
};
struct Stream {
  long last = -1, last_real = -1;
  bool capturing = false;
};
struct Event {
  long op = -1;
};
std::vector<Op> ops;
std::set<Stream*> streams;
std::map<const void*, size_t> live;
int sms = 152;
thread_local cudaStreamCaptureMode mode = cudaStreamCaptureModeGlobal;
bool other_capture = false;                // a stream of some other code is captured in the default mode,
bool other_broken = false;                 // and a call of ours has ended that
uint32_t verdict = 0;                      // what the prime form's check says
std::map<std::string, int> calls, fail_at;  // fails from that call on (negative: that call alone)

#define REQUIRE(x)                                              \
  do {                                                          \
    if (!(x)) {                                                 \
      std::printf("line %d: %s does not hold\n", __LINE__, #x); \
      std::exit(1);                                             \
    }                                                           \
  } while (0)

// A call that a capture in the default mode forbids
bool forbidden() {
  if (!other_capture || mode == cudaStreamCaptureModeRelaxed) return false;
  other_broken = true;
  return true;
}

bool fails(const std::string& name) {
  std::lock_guard<std::recursive_mutex> l(mu);
  const int k = ++calls[name];
  const auto f = fail_at.find(name);
  return f != fail_at.end() && (f->second < 0 ? k == -f->second : k >= f->second);
}

Stream* of(cudaStream_t s) { return reinterpret_cast<Stream*>(s); }

cudaError_t add(cudaStream_t st, const std::string& what, std::vector<const void*> reads = {}, long also_after = -1) {
  std::lock_guard<std::recursive_mutex> l(mu);
  Stream* s = of(st);
  REQUIRE(streams.count(s));
  for (const void* p : reads) REQUIRE(!p || live.count(p));
  Op op;
  op.what = what;
  op.reads = reads;
  if (s->last >= 0) op.after.push_back(static_cast<size_t>(s->last));
  if (also_after >= 0) op.after.push_back(static_cast<size_t>(also_after));
  op.captured = s->capturing;
  ops.push_back(op);
  s->last = static_cast<long>(ops.size()) - 1;
  if (!s->capturing) s->last_real = s->last;
  return cudaSuccess;
}

std::vector<bool> before(long op) {  // the operations that have ended when `op` has
  std::vector<bool> in(ops.size(), false);
  std::vector<size_t> todo;
  if (op >= 0) todo.push_back(static_cast<size_t>(op));
  while (!todo.empty()) {
    const size_t i = todo.back();
    todo.pop_back();
    if (in[i]) continue;
    in[i] = true;
    for (size_t a : ops[i].after) todo.push_back(a);
  }
  return in;
}

cudaError_t wait_for(long op) {
  std::lock_guard<std::recursive_mutex> l(mu);
  const std::vector<bool> in = before(op);
  for (size_t i = 0; i < ops.size(); ++i)
    if (in[i]) ops[i].complete = true;
  return cudaSuccess;
}

// What torch.cuda.graph does around a call
void begin_capture(cudaStream_t s) {
  of(s)->capturing = true;
  of(s)->last = -1;
}
void end_capture() {
  for (Stream* s : streams) {
    s->capturing = false;
    s->last = s->last_real;
  }
}

size_t in_flight() {
  size_t n = 0;
  for (const Op& o : ops) n += !o.complete && !o.captured;
  return n;
}

}  // namespace

extern "C" {

cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  std::memset(p, 0, sizeof(*p));
  p->multiProcessorCount = sms;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetStreamPriorityRange(int* a, int* b) { *a = 0; *b = -5; return cudaSuccess; }

cudaError_t cudaMalloc(void** p, size_t n) {
  if (forbidden()) return cudaErrorStreamCaptureUnsupported;
  if (fails("cudaMalloc")) return cudaErrorMemoryAllocation;
  std::lock_guard<std::recursive_mutex> l(mu);
  *p = std::calloc(1, n ? n : 1);
  live[*p] = n;
  return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode* m) { std::swap(*m, mode); return cudaSuccess; }
cudaError_t cudaFree(void* p) {
  if (forbidden()) return cudaErrorStreamCaptureUnsupported;
  std::lock_guard<std::recursive_mutex> l(mu);
  if (!p) return cudaSuccess;
  REQUIRE(live.erase(p) == 1);
  for (Op& o : ops) o.complete |= !o.captured;  // waits for the device
  return cudaSuccess;  // the memory stays, so that no address comes back
}
cudaError_t cudaMallocHost(void** p, size_t n) { *p = std::calloc(1, n ? n : 1); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned int) { return cudaMallocHost(p, n); }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }

cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned int, int) {
  std::lock_guard<std::recursive_mutex> l(mu);
  Stream* n = new Stream();
  streams.insert(n);
  *s = reinterpret_cast<cudaStream_t>(n);
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned int) { return cudaStreamCreateWithPriority(s, 0, 0); }
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  std::lock_guard<std::recursive_mutex> l(mu);
  REQUIRE(streams.erase(of(s)) == 1);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return wait_for(of(s)->last_real); }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* c) {
  *c = of(s)->capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t e, unsigned int) {
  std::lock_guard<std::recursive_mutex> l(mu);
  const long op = reinterpret_cast<Event*>(e)->op;
  if (op < 0) return cudaSuccess;
  Stream* s = of(st);
  const bool captured = ops[static_cast<size_t>(op)].captured;
  if (captured && !s->capturing) {  // the stream joins the capture that is going on
    bool any = false;
    for (Stream* o : streams) any |= o->capturing;
    if (!any) return cudaErrorCapturedEvent;
    s->capturing = true;
    s->last = -1;
  }
  if (s->capturing && !captured) return cudaErrorStreamCaptureIsolation;
  return add(st, "wait", {}, op);
}

cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned int) {
  *e = reinterpret_cast<cudaEvent_t>(new Event());
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete reinterpret_cast<Event*>(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  std::lock_guard<std::recursive_mutex> l(mu);
  if (of(s)->last < 0) add(s, "nothing");
  reinterpret_cast<Event*>(e)->op = of(s)->last;
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) { return wait_for(reinterpret_cast<Event*>(e)->op); }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; return cudaSuccess; }

cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) {
  if (n && !of(s)->capturing) std::memset(p, v, n);
  return add(s, "memset");
}
cudaError_t cudaMemcpyAsync(void* d, const void* src, size_t n, cudaMemcpyKind, cudaStream_t s) {
  if (n && !of(s)->capturing) std::memcpy(d, src, n);
  return add(s, "memcpy");
}

cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
  begin_capture(s);
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
  of(s)->capturing = false;
  of(s)->last = of(s)->last_real;
  *g = reinterpret_cast<cudaGraph_t>(1);
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = reinterpret_cast<cudaGraphExec_t>(1);
  return cudaSuccess;
}
cudaError_t cudaGraphExecUpdate(cudaGraphExec_t, cudaGraph_t, cudaGraphExecUpdateResultInfo*) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) { return add(s, "graph"); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

}  // extern "C"

namespace bbp {

int head_lmax_for(int L, int bump) {
  if (fails("head_lmax_for")) return 0;
  for (int i = 0; i < kNumLmaxClasses; ++i)
    if (kLmaxClasses[i] >= L) return kLmaxClasses[std::min(i + bump, kNumLmaxClasses - 1)];
  return 0;
}
int head_occupancy(int, int, int, int) { return 2; }
int query_occupancy(int, int, int) { return 2; }
int queue_occupancy(int, int, int) { return 2; }
std::vector<int> head_paths;
cudaError_t launch_head(const HeadArgs& a, int path, int, int, int, cudaStream_t s, int) {
  head_paths.push_back(path);
  return add(s, "head", {a.slots});
}
cudaError_t launch_tail_set(const TailSet&, cudaStream_t s) { return add(s, "tails"); }
cudaError_t launch_query(const QuerySet& q, int, int, int, int, cudaStream_t s) { return add(s, "query", {q.slots}); }
cudaError_t launch_zero_slots(unsigned long long* p, int, cudaStream_t s, const uint32_t*) { return add(s, "zero", {p}); }
cudaError_t launch_fold_limbs(const unsigned long long* p, int, uint32_t*, cudaStream_t s) { return add(s, "fold", {p}); }
cudaError_t launch_finalize_bits(const unsigned long long* p, int, uint32_t, uint64_t, uint8_t*, uint32_t*, uint32_t*,
                                 cudaStream_t s, const uint32_t*) {
  return add(s, "finalize", {p});
}
std::vector<std::array<int, 2>> queues;  // tiles a hand-out, CTAs
cudaError_t launch_queue(const BatchDev& b, uint32_t, uint32_t, unsigned long long*, int, int, int, int blocks, cudaStream_t s) {
  queues.push_back({static_cast<int>(b.grab), blocks});
  return add(s, "queue", {b.accum});
}
cudaError_t launch_queue_tail(const BatchDev& b, uint32_t, uint32_t, unsigned long long*, int, cudaStream_t s) {
  return add(s, "queue tails", {b.accum});
}
cudaError_t launch_timestamp(unsigned long long*, cudaStream_t s) { return add(s, "time"); }
cudaError_t launch_imad_probe(int, int, int, int, unsigned long long*, uint32_t*, uint32_t*, cudaStream_t s) {
  return add(s, "probe");
}
cudaError_t launch_base_primes(uint32_t, uint32_t* p, SievePrime* sp, uint32_t* c, uint32_t*, cudaStream_t s) {
  return add(s, "base", {p, sp, c});
}
cudaError_t launch_sieve(const SieveArgs& a, int, cudaStream_t s) { return add(s, "sieve", {a.list}); }
cudaError_t launch_prime(const PrimeArgs& a, PrimeKernel, int, int, int, cudaStream_t s) {
  if (fails("launch_prime")) return cudaErrorLaunchOutOfResources;
  return add(s, "primes", {a.list});
}
cudaError_t launch_prime_check(const unsigned long long* slots, int, uint32_t, uint64_t, const uint32_t*, uint32_t, uint32_t,
                               uint8_t*, uint32_t*, uint32_t* redo, cudaStream_t s) {
  *redo = verdict;
  (void)slots;
  return add(s, "check");
}

}  // namespace bbp

using namespace bbp;

namespace {

struct Caller {
  bbp_plan plan = nullptr;
  cudaStream_t a = nullptr, b = nullptr;
  void* out = nullptr;
  Caller() {
    REQUIRE(bbp_plan_create(&plan, nullptr) == BBP_OK);
    cudaStreamCreateWithFlags(&a, 0);
    cudaStreamCreateWithFlags(&b, 0);
    cudaMalloc(&out, 256);
  }
  bbp_status async(uint64_t n, cudaStream_t s) {
    return bbp_bits_async(plan, BBP_BELLARD, n, 128, static_cast<uint8_t*>(out), nullptr, nullptr, s);
  }
  bbp_status bits(uint64_t n, bbp_formula f = BBP_BELLARD) {
    uint8_t bytes[160];
    return bbp_bits_formula(plan, f, n, 128, bytes, nullptr);
  }
};

// A captured query by primes, then larger ones that need longer lists, captured again and
// again: what the captures use is there until the plan goes, and goes with it.  What is held
// stays bounded.
void captured_lists_stay() {
  const size_t outside = 1;  // Caller::out
  Caller c;
  REQUIRE(c.bits(17'000'000) == BBP_OK);
  uint64_t largest = 0;
  for (uint64_t n = 17'000'000; n < 2'000'000'000; n += n / 9) {
    begin_capture(c.a);
    REQUIRE(c.async(n, c.a) == BBP_OK);
    end_capture();
    REQUIRE(c.bits(n + n / 9) == BBP_OK);
    for (const Op& o : ops)
      if (o.captured)
        for (const void* p : o.reads) REQUIRE(!p || live.count(p));
    size_t held = 0;
    for (const auto& m : live) held += m.second;
    largest = std::max<uint64_t>(largest, held);
  }
  size_t captured = 0;
  for (const Op& o : ops) captured += o.captured && o.what == "sieve";
  REQUIRE(captured > 0);
  REQUIRE(largest < 512ull << 20);  // two lists of 96 MB, and as much again of shorter ones
  REQUIRE(bbp_plan_destroy(c.plan) == BBP_OK);
  REQUIRE(live.size() == outside);
}

// Quotients of the sums' limits by primes from their square root on, from every single-precision
// estimate that the division's two ulps allow, up to the largest position of both formulas.
void sum_quotients() {
  std::mt19937_64 rng(7);
  for (int i = 0; i < 400000; ++i) {
    const int formula = i & 1;
    const uint64_t n = i < 1000 ? kPrimeMaxN - i : kPrimeMinN + rng() % (kPrimeMaxN - kPrimeMinN + 1);
    const PrimeLimits lim = prime_limits(formula, n - 1);
    const uint64_t root = static_cast<uint64_t>(std::sqrt(static_cast<double>(lim.A)));
    const uint64_t p = root + rng() % (i & 2 ? 100 : i & 4 ? root : 22 * root);
    uint64_t a[4] = {lim.A, lim.B, lim.C, n + 1280};
    a[3] -= rng() % p;
    a[0] = i & 8 ? a[0] / p * p - (i >> 4 & 1) : a[0];  // at a multiple, and one below
    for (uint64_t v : a) {
      const float near = static_cast<float>(v) / static_cast<float>(p);
      float q = std::nextafter(std::nextafter(near, 0.0f), 0.0f);
      for (int ulp = -2; ulp <= 2; ++ulp, q = std::nextafter(q, 1e30f))
        REQUIRE((formula ? corrected_quotient<1>(static_cast<uint32_t>(q), v, p)
                         : corrected_quotient<0>(static_cast<uint32_t>(q), v, p)) == v / p);
    }
  }
}

// The largest positions of both formulas, in lists of each length, on several numbers of SMs.
void largest_positions() {
  for (int n_sms : {120, 132, 148, 152, 160}) {
    sms = n_sms;
    Caller c;
    for (bbp_formula f : {BBP_BELLARD, BBP_BBP}) {
      const uint64_t n[2] = {kPrimeMaxN, kPrimeMaxN + 1};
      const uint32_t P[2] = {64, 64};
      uint8_t out[16];
      calls["launch_prime"] = 0;
      REQUIRE(bbp_bits_batch(c.plan, f, 1, n, P, out, 8, nullptr, nullptr) == BBP_OK);
      REQUIRE(calls["launch_prime"] > 10000);  // by primes
      if (n_sms == 152) REQUIRE(c.bits(kPrimeMaxN, f) == BBP_OK);
      ops.clear();
      for (Stream* s : streams) s->last = s->last_real = -1;
    }
    bbp_plan_destroy(c.plan);
  }
}

// A query whose lists cannot be planned is summed by its terms: alone, and in a batch.
void no_plan_no_primes() {
  Caller c;
  REQUIRE(c.bits(100'000'000) == BBP_OK);
  const int primes = calls["launch_prime"];
  calls["head_lmax_for"] = 0;
  fail_at["head_lmax_for"] = -10;  // the lists': after the query's, seven series' leftovers and their launch
  REQUIRE(c.bits(100'000'000) == BBP_OK);
  REQUIRE(calls["head_lmax_for"] > 10 && calls["launch_prime"] == primes);
  const uint64_t n[3] = {50'000'000, 1'000'000, 100'000'000};
  const uint32_t P[3] = {64, 64, 64};
  uint8_t out[24];
  double ms[3];
  calls["head_lmax_for"] = 0;
  fail_at["head_lmax_for"] = -4;  // three queries, then the first one's lists
  REQUIRE(bbp_bits_batch(c.plan, BBP_BELLARD, 3, n, P, out, 8, nullptr, ms) == BBP_OK);
  size_t graphs = 0;
  for (const Op& o : ops) graphs += o.what == "graph";
  REQUIRE(graphs == 2);  // the second pass
}

// A batch that fails among its prime forms has waited for all it queued when it returns.
void failed_batch_leaves_nothing() {
  Caller c;
  const uint64_t n[4] = {50'000'000, 1'000'000, 1'000'000'000, 100'000'000};
  const uint32_t P[4] = {64, 64, 64, 64};
  uint8_t out[32];
  for (int at = 1; at < 30; ++at) {
    calls["launch_prime"] = 0;
    fail_at["launch_prime"] = -at;
    REQUIRE(bbp_bits_batch(c.plan, BBP_BELLARD, 4, n, P, out, 8, nullptr, nullptr) == BBP_ECUDA);
    REQUIRE(calls["launch_prime"] >= at);
    REQUIRE(in_flight() == 0);
  }
}

bbp_status served(bbp_plan plan, bbp_ticket t) {
  uint8_t out[160];
  bbp_status st;
  while ((st = bbp_poll(plan, t, out, nullptr)) == BBP_PENDING) std::this_thread::yield();
  return st;
}

// A submitted query whose lists and then whose terms cannot be planned fails: no result is made
// of the few terms that the primes leave.
void unplanned_query_fails() {
  Caller c;
  bbp_ticket t = 0;
  calls["head_lmax_for"] = 0;
  fail_at["head_lmax_for"] = 2;  // after the submission's own
  REQUIRE(bbp_submit(c.plan, 100'000'000, 64, &t) == BBP_OK);
  REQUIRE(served(c.plan, t) == BBP_EINVAL);
  fail_at.clear();
  REQUIRE(bbp_submit(c.plan, 100'000'000, 64, &t) == BBP_OK);
  REQUIRE(served(c.plan, t) == BBP_OK);
  REQUIRE(bbp_plan_destroy(c.plan) == BBP_OK);
}

// An iteration that fails among its prime forms has ended when its queries are given back.
void failed_iteration_leaves_nothing() {
  for (int at : {1, 2, 3, 5, 9}) {
    Caller c;
    bbp_ticket t = 0;
    calls["launch_prime"] = 0;
    fail_at["launch_prime"] = -at;
    REQUIRE(bbp_submit(c.plan, 1'000'000'000, 64, &t) == BBP_OK);
    REQUIRE(served(c.plan, t) == BBP_ECUDA);
    {
      std::lock_guard<std::recursive_mutex> l(mu);
      REQUIRE(in_flight() == 0);
    }
    REQUIRE(bbp_submit(c.plan, 100'000'000, 64, &t) == BBP_OK);
    REQUIRE(served(c.plan, t) == BBP_OK);
    REQUIRE(bbp_plan_destroy(c.plan) == BBP_OK);
  }
}

// Stream queries beside a capture of some other stream, at a plan's first use and where its
// lists have to grow: the capture goes on, and the query runs by primes.
void beside_a_capture() {
  Caller c;
  other_capture = true;
  for (uint64_t n : {100'000'000, 1'000'000'000}) {
    const int primes = calls["launch_prime"];
    REQUIRE(c.async(n, c.a) == BBP_OK);
    REQUIRE(!other_broken && calls["launch_prime"] > primes);
    REQUIRE(mode == cudaStreamCaptureModeGlobal);
  }
}

// Queries on one stream after another, with captured ones between them: none sieves before
// those before it have used the workspace.
void runs_follow_one_another() {
  Caller c;
  auto uses = [](const Op& o) { return o.what == "base" || o.what == "sieve" || o.what == "primes" || o.what == "check"; };
  for (cudaStream_t s : {c.a, c.b, c.b, c.a, c.b}) {
    const size_t first = ops.size();
    REQUIRE(c.async(1'000'000'000, s) == BBP_OK);
    size_t sieve = first;
    while (ops[sieve].what != "sieve") ++sieve;
    const std::vector<bool> ended = before(static_cast<long>(sieve));
    for (size_t i = 0; i < first; ++i) REQUIRE(ended[i] || ops[i].captured || !uses(ops[i]));
    begin_capture(c.a);
    REQUIRE(c.async(1'000'000'000, c.a) == BBP_OK);
    end_capture();
  }
}

// A range across the line between two ladders is one launch while it is short, two when it is
// long enough on both sides.
void short_ranges_stay_whole() {
  Caller c;
  uint32_t limbs[10];
  for (uint64_t line : {kHalfMaxModulus, uint64_t{1} << 47}) {
    const uint64_t k = (line - 1) / 10 + 1;  // first k of series 10 k + 1 past it
    for (auto [below, above, launches] : {std::array<uint64_t, 3>{700, 700, 1}, {1000, 599'000, 1}, {1'000'000, 1'000'000, 1},
                                          {1000, 5'000'000, 1}, {1'500'000, 1'500'000, 2}, {5'000'000, 0, 1}, {0, 5'000'000, 1}}) {
      const size_t first = ops.size();
      REQUIRE(bbp_partial_sum(c.plan, BBP_BELLARD, 0, k - below, k + above, 100 * line, 256, limbs) == BBP_OK);
      uint64_t heads = 0;
      for (size_t i = first; i < ops.size(); ++i) heads += ops[i].what == "head";
      REQUIRE(heads == launches);
    }
  }
}

// Ranges of 47-bit moduli that leave SMs idle stay on the four-word path.
void short_47_bit_ranges() {
  Caller c;
  uint32_t limbs[6];
  for (auto [count, path] : {std::array<int, 2>{1000, 2}, {77'000, 2}, {78'000, kPath47}, {2'000'000, kPath47}}) {
    head_paths.clear();
    const uint64_t k = (uint64_t{1} << 46) / 10 + 10;
    REQUIRE(bbp_partial_sum(c.plan, BBP_BELLARD, 0, k, k + static_cast<uint64_t>(count), 1'000'000'000'000'000, 128, limbs) == BBP_OK);
    REQUIRE(head_paths == std::vector<int>{path});
  }
}

// Whole queries term by term (the raw sum wanted): one launch, but for many terms of 40 limbs.
void one_launch_by_size() {
  Caller c;
  void* limbs;
  cudaMalloc(&limbs, 256);
  for (auto [n, P, one] : {std::array<uint64_t, 3>{20'000'000, 1000, 1}, {40'000'000, 1000, 0}, {500'000'000, 1000, 0},
                           {500'000'000, 700, 1}, {500'000'000, 256, 1}}) {
    const size_t first = ops.size();
    REQUIRE(bbp_bits_async(c.plan, BBP_BELLARD, n, static_cast<uint32_t>(P), static_cast<uint8_t*>(c.out), nullptr,
                           static_cast<uint32_t*>(limbs), c.a) == BBP_OK);
    size_t queries = 0, heads = 0;
    for (size_t i = first; i < ops.size(); ++i) queries += ops[i].what == "query", heads += ops[i].what == "head";
    REQUIRE(queries == one && (heads == 0) == (one == 1));
  }
}

// A small batch is spread over the SMs, a large one takes what fits, four tiles at a time.
void small_groups_spread() {
  Caller c;
  std::vector<uint64_t> n(150, 1'000'000);
  std::vector<uint32_t> P(150, 64);
  std::vector<uint8_t> out(8 * 150);
  for (auto [count, grab, least, most] : {std::array<int, 4>{1, 1, sms, 2 * sms}, {150, 4, 2 * sms, 2 * sms}}) {
    queues.clear();
    REQUIRE(bbp_bits_batch(c.plan, BBP_BBP, static_cast<uint32_t>(count), n.data(), P.data(), out.data(), 8, nullptr, nullptr) == BBP_OK);
    REQUIRE(queues.size() == 1 && queues[0][0] == grab && queues[0][1] >= least && queues[0][1] <= most);
  }
  n[0] = 60;  // a handful of terms: a CTA for each tile
  queues.clear();
  REQUIRE(bbp_bits_batch(c.plan, BBP_BBP, 1, n.data(), P.data(), out.data(), 8, nullptr, nullptr) == BBP_OK);
  REQUIRE(queues.size() == 1 && queues[0][0] == 1 && queues[0][1] >= 1 && queues[0][1] < 32);
}

const std::map<std::string, void (*)()> kCases = {
    {"small_groups_spread", small_groups_spread},
    {"one_launch_by_size", one_launch_by_size},
    {"short_47_bit_ranges", short_47_bit_ranges},
    {"short_ranges_stay_whole", short_ranges_stay_whole},
    {"runs_follow_one_another", runs_follow_one_another},
    {"beside_a_capture", beside_a_capture},
    {"failed_iteration_leaves_nothing", failed_iteration_leaves_nothing},
    {"unplanned_query_fails", unplanned_query_fails},
    {"failed_batch_leaves_nothing", failed_batch_leaves_nothing},
    {"largest_positions", largest_positions},
    {"no_plan_no_primes", no_plan_no_primes},
    {"sum_quotients", sum_quotients},
    {"captured_lists_stay", captured_lists_stay},
};

}  // namespace

int main(int argc, char** argv) {
  const auto c = kCases.find(argc > 1 ? argv[1] : "");
  REQUIRE(c != kCases.end());
  c->second();
  return 0;
}
