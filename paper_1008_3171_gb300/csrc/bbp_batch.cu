// Batched queries: one persistent, graph-captured pass over a chunk queue.
//
// Every query of a batch is planned into jobs (bbp_planner.cpp): head jobs -- one
// range of head terms of one series, with the ladder parameters of its moduli --
// and tail jobs.  Queries are sorted by size and cut into waves whose work grows
// geometrically (the smallest queries first) up to 1/12 of the batch, so the
// largest queries finish over the last several waves rather than together at the
// end of one; a wave is one tail launch plus one
// persistent launch per kernel variant (limb capacity x modulus path) in which
// warps take `grab` tiles of the current job at a time (queue_kernel), so queries
// of very different sizes share the GPU at tile granularity and small ones finish
// early.  Each query's signed partial sums accumulate in its own carry-save
// slots; the warp that retires its last job finalizes it on the device and stamps
// the completion time.  The whole pass -- uploads, resets, launches, downloads --
// is captured once into a CUDA graph and replayed (the executable graph is updated
// in place when the next batch has the same shape).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <new>
#include <numeric>
#include <vector>

#include "bbp.h"
#include "bbp_kernels.cuh"
#include "bbp_planner.h"
#include "bbp_prime_run.h"
#include "bbp_primes.h"
#include "bbp_runtime.h"

using namespace bbp;

namespace {

constexpr int kVariants = kQueueVariants;
constexpr int kPrimeLanes = 4;
constexpr uint32_t kOutStride = kMaxWorkingBits / 8;  // bytes of output per query slot

int lmax_index(int lmax) {
  for (int i = 0; i < kNumLmaxClasses; ++i)
    if (kLmaxClasses[i] == lmax) return i;
  return -1;
}

template <typename T>
bool grow_device(T** p, size_t* cap, size_t want) {
  if (*cap >= want && *p) return true;
  cudaFree(*p);
  *p = nullptr;
  const size_t n = std::max<size_t>(want, 1) * 2;
  if (cudaMalloc(reinterpret_cast<void**>(p), n * sizeof(T)) != cudaSuccess) {
    *cap = 0;
    return false;
  }
  *cap = n;
  return true;
}

template <typename T>
bool grow_host(T** p, size_t* cap, size_t want) {
  if (*cap >= want && *p) return true;
  cudaFreeHost(*p);
  *p = nullptr;
  const size_t n = std::max<size_t>(want, 1) * 2;
  if (cudaMallocHost(reinterpret_cast<void**>(p), n * sizeof(T)) != cudaSuccess) {
    *cap = 0;
    return false;
  }
  *cap = n;
  return true;
}

}  // namespace

struct BatchState {
  // device buffers and their capacities (elements)
  HeadArgs* d_jobs = nullptr;               size_t c_jobs = 0;
  uint32_t* d_job_query = nullptr;          size_t c_job_query = 0;
  uint64_t* d_job_start = nullptr;          size_t c_job_start = 0;
  unsigned long long* d_job_done = nullptr; size_t c_job_done = 0;
  TailArgs* d_tails = nullptr;              size_t c_tails = 0;
  uint32_t* d_tail_query = nullptr;         size_t c_tail_query = 0;
  QueryDesc* d_queries = nullptr;           size_t c_queries = 0;
  unsigned long long* d_accum = nullptr;    size_t c_accum = 0;
  unsigned int* d_jobs_left = nullptr;      size_t c_jobs_left = 0;
  uint8_t* d_out = nullptr;                 size_t c_out = 0;
  uint32_t* d_valid = nullptr;              size_t c_valid = 0;
  unsigned long long* d_done = nullptr;     size_t c_done = 0;   // [0] = start time, [1 + q] = done
  unsigned long long* d_cursors = nullptr;  size_t c_cursors = 0;  // per wave: kVariants + 1 (tail)
  // pinned host staging
  HeadArgs* h_jobs = nullptr;               size_t hc_jobs = 0;
  uint32_t* h_job_query = nullptr;          size_t hc_job_query = 0;
  uint64_t* h_job_start = nullptr;          size_t hc_job_start = 0;
  TailArgs* h_tails = nullptr;              size_t hc_tails = 0;
  uint32_t* h_tail_query = nullptr;         size_t hc_tail_query = 0;
  QueryDesc* h_queries = nullptr;           size_t hc_queries = 0;
  unsigned int* h_jobs_left = nullptr;      size_t hc_jobs_left = 0;
  uint8_t* h_out = nullptr;                 size_t hc_out = 0;
  uint32_t* h_valid = nullptr;              size_t hc_valid = 0;
  unsigned long long* h_done = nullptr;     size_t hc_done = 0;
  // prime forms: the check's verdict per query, and the workspaces with their streams
  uint32_t* d_redo = nullptr;               size_t c_redo = 0;
  uint32_t* h_redo = nullptr;               size_t hc_redo = 0;
  PrimeState* lane[kPrimeLanes] = {};
  cudaStream_t lane_stream[kPrimeLanes] = {};
  cudaEvent_t lane_done[kPrimeLanes] = {};
  cudaGraphExec_t exec = nullptr;
  cudaStream_t stream = nullptr;  // capture needs a stream other than the legacy default stream
  cudaEvent_t ready = nullptr;
};

namespace bbp {

// Waits for everything a batch has queued: after a call that failed half way, no kernel may
// still add to the accumulators nor a copy read the staging that the next call fills.
static void wait_batch(BatchState* b) {
  if (b->stream) cudaStreamSynchronize(b->stream);
  for (int i = 0; i < kPrimeLanes; ++i) {
    if (b->lane_stream[i]) cudaStreamSynchronize(b->lane_stream[i]);
    wait_prime_state(b->lane[i]);
  }
}

void release_batch_state(bbp_plan p) {
  BatchState* b = p->batch;
  if (!b) return;
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->stream) cudaStreamDestroy(b->stream);
  if (b->ready) cudaEventDestroy(b->ready);
  for (int i = 0; i < kPrimeLanes; ++i) {
    release_prime_state(&b->lane[i]);
    if (b->lane_stream[i]) cudaStreamDestroy(b->lane_stream[i]);
    if (b->lane_done[i]) cudaEventDestroy(b->lane_done[i]);
  }
  cudaFree(b->d_redo);
  cudaFreeHost(b->h_redo);
  cudaFree(b->d_jobs);
  cudaFree(b->d_job_query);
  cudaFree(b->d_job_start);
  cudaFree(b->d_job_done);
  cudaFree(b->d_tails);
  cudaFree(b->d_tail_query);
  cudaFree(b->d_queries);
  cudaFree(b->d_accum);
  cudaFree(b->d_jobs_left);
  cudaFree(b->d_out);
  cudaFree(b->d_valid);
  cudaFree(b->d_done);
  cudaFree(b->d_cursors);
  cudaFreeHost(b->h_jobs);
  cudaFreeHost(b->h_job_query);
  cudaFreeHost(b->h_job_start);
  cudaFreeHost(b->h_tails);
  cudaFreeHost(b->h_tail_query);
  cudaFreeHost(b->h_queries);
  cudaFreeHost(b->h_jobs_left);
  cudaFreeHost(b->h_out);
  cudaFreeHost(b->h_valid);
  cudaFreeHost(b->h_done);
  delete b;
  p->batch = nullptr;
}

constexpr int kMaxWaves = 24;

// Plans `count` queries into the batch's pinned staging buffers.
struct BatchPlan {
  uint32_t njobs = 0, ntails = 0, nwaves = 0;
  uint32_t group_begin[kMaxWaves * kVariants + 1] = {};  // head jobs of (wave, variant)
  uint32_t tail_begin[kMaxWaves + 1] = {};               // tail jobs of a wave
  uint64_t terms = 0, head_terms = 0;
  double imad = 0;
  struct Prime { uint32_t q, W; uint64_t n, bound; bool planned; };
  std::vector<Prime> primes;  // queries by the prime form, smallest first
};

static bbp_status plan_batch(bbp_plan p, int f, uint32_t count, const uint64_t* n, const uint32_t* P,
                             BatchState* b, BatchPlan* bp, bool by_primes) {
  const FormulaDef& F = formula_def(f);
  std::vector<std::vector<HeadArgs>> vj(kVariants);
  std::vector<std::vector<uint32_t>> vq(kVariants);
  std::vector<std::vector<uint64_t>> vt(kVariants);
  std::vector<TailArgs> tails;
  std::vector<uint32_t> tail_q;
  std::vector<QueryDesc> queries(count);
  std::vector<unsigned int> jobs_left(count, 0);
  std::vector<uint64_t> qterms(count, 0);
  std::vector<TermRange> ranges;
  for (uint32_t q = 0; q < count; ++q) {
    uint32_t W;
    if (n[q] == 0 || !working_bits(P[q], p->guard, &W)) return BBP_EINVAL;
    const uint32_t L = W / 32;
    const int lmax = head_lmax_for(static_cast<int>(L));
    if (lmax == 0) return BBP_EINVAL;
    unsigned long long* slots = b->d_accum + static_cast<uint64_t>(q) * kMaxLimbs;
    ranges.clear();
    uint64_t N = 0;
    for (uint32_t j = 0; j < F.count; ++j) {
      const int st = plan_series(F, j, n[q], W, static_cast<uint32_t>(lmax), 0, UINT64_MAX, ranges, p->wide_min_bits);
      if (st == -6) return BBP_ERANGE;
      if (st != 0) return BBP_EINVAL;
      N += natural_end(F, j, n[q] - 1, W);
    }
    uint64_t qtiles = 0;
    for (const TermRange& r : ranges)
      if (!r.tail) qtiles += (r.count + tile_terms(p, r.path) - 1) / tile_terms(p, r.path);
    if (qtiles > kMaxQueueTiles) return BBP_ERANGE;  // carry-save limbs could pass 2^64
    const uint64_t bound = N + F.count + 1;
    const bool prime = by_primes && prime_form_serves(f, n[q], P[q], W, bound);
    for (const TermRange& r : ranges) {
      bp->terms += r.count;
      if (!r.tail) bp->head_terms += r.count;
      if (!r.tail && !prime) bp->imad += r.imad;
    }
    if (prime) {  // the queue takes what the prime form leaves
      const PrimeLimits lim = prime_limits(f, n[q] - 1);
      bp->imad += prime_form_imad(lim, static_cast<int>(L));
      bp->primes.push_back(BatchPlan::Prime{q, W, n[q], bound, true});
      ranges.clear();
      for (uint32_t j = 0; j < F.count; ++j)
        if (plan_series(F, j, n[q], W, static_cast<uint32_t>(lmax), prime_first_k(lim, j, n[q] - 1), UINT64_MAX, ranges,
                        p->wide_min_bits) != 0)
          return BBP_EINVAL;
      jobs_left[q] = 1;  // held: the check writes the result
    }
    for (const TermRange& r : ranges) {
      const SeriesDef& s = F.s[r.j];
      qterms[q] += r.count;
      if (r.tail) {
        TailArgs a{};
        a.d = n[q] - 1;
        a.k_begin = r.k_begin;
        a.count = r.count;
        a.a = s.a;
        a.b = s.b;
        a.c = s.c;
        a.step = F.step;
        a.W = W;
        a.L = L;
        a.alternating = F.alternating;
        a.negate = s.sign < 0 ? 1u : 0u;
        a.slots = slots;
        tails.push_back(a);
        tail_q.push_back(q);
      } else {
        HeadArgs a{};
        a.d = n[q] - 1;
        a.k_begin = r.k_begin;
        a.count = r.count;
        a.a = s.a;
        a.b = s.b;
        a.c = s.c;
        a.step = F.step;
        a.W = W;
        a.L = L;
        a.alternating = F.alternating;
        a.negate = ((s.sign < 0) != (F.alternating && (r.k_begin & 1ull))) ? 1u : 0u;
        // Short ranges take fewer terms per stream: 64 tiles where they can, so that a range is not
        // a few warps' long runs (but at least 8 terms: each run starts with a division).  With one
        // tile counter for all jobs (queue_kernel), 164 queries up to 1.6e7: 12.6 -> 5.1 ms.
        const uint64_t lanes = 32ull * static_cast<uint64_t>(head_streams(p, r.path));
        uint32_t run = static_cast<uint32_t>(p->run);
        while (run >= 16 && run % 4 == 0 && r.count < 64 * lanes * run) run /= 2;
        a.run = run;
        a.window = r.window;
        a.first = r.first;
        a.first_max = r.first_max;
        a.slots = slots;
        const int v = lmax_index(lmax) * kNumPaths + r.path;
        vj[v].push_back(a);
        vq[v].push_back(q);
        vt[v].push_back((r.count + lanes * run - 1) / (lanes * run));
      }
      jobs_left[q]++;
    }
    if (jobs_left[q] == 0) {  // no term at all: a zero-length tail job still retires it
      TailArgs a{};
      a.W = W;
      a.L = L;
      a.slots = slots;
      tails.push_back(a);
      tail_q.push_back(q);
      jobs_left[q] = 1;
    }
    QueryDesc& Q = queries[q];
    Q.bound = bound;
    Q.P = P[q];
    Q.L = L;
    Q.out_offset = q * kOutStride;
  }
  std::sort(bp->primes.begin(), bp->primes.end(),
            [](const BatchPlan::Prime& x, const BatchPlan::Prime& y) { return x.n != y.n ? x.n < y.n : x.q < y.q; });
  // waves: queries by size, each wave twice the work of the ones before it, at most 1/12 of the
  // total -- but at least kWaveTerms, some milliseconds: a launch lasts no less than a tile's 50 us,
  // whatever its size (164 queries up to 1.6e7, 2.5e8 terms: 19 ms in 24 waves, 12.6 in two)
  constexpr uint64_t kWaveTerms = 200'000'000;
  std::vector<uint32_t> qorder(count);
  std::iota(qorder.begin(), qorder.end(), 0u);
  std::stable_sort(qorder.begin(), qorder.end(), [&](uint32_t x, uint32_t y) { return qterms[x] < qterms[y]; });
  std::vector<uint32_t> wave_of(count, 0);
  {
    uint64_t total = 0;
    for (uint64_t t : qterms) total += t;
    const uint64_t first = std::max<uint64_t>(total / 4096, kWaveTerms);  // the first wave: 1/4096 of the work
    const uint64_t step_cap = std::max<uint64_t>(total / 12, kWaveTerms);  // no wave beyond 1/12 of the work
    uint64_t done = 0, target = first;
    uint32_t w = 0;
    for (uint32_t i = 0; i < count; ++i) {
      const uint32_t q = qorder[i];
      if (done >= target && w + 1 < static_cast<uint32_t>(kMaxWaves)) {
        ++w;
        target = std::min(std::max(target, done) * 2, done + step_cap);
      }
      wave_of[q] = w;
      done += qterms[q];
    }
    bp->nwaves = w + 1;
  }
  uint32_t nj = 0;
  for (int v = 0; v < kVariants; ++v) nj += static_cast<uint32_t>(vj[v].size());
  if (!grow_host(&b->h_jobs, &b->hc_jobs, nj) || !grow_host(&b->h_job_query, &b->hc_job_query, nj) ||
      !grow_host(&b->h_job_start, &b->hc_job_start, nj + 1) || !grow_host(&b->h_tails, &b->hc_tails, tails.size()) ||
      !grow_host(&b->h_tail_query, &b->hc_tail_query, tails.size()) ||
      !grow_host(&b->h_queries, &b->hc_queries, count) || !grow_host(&b->h_jobs_left, &b->hc_jobs_left, count))
    return BBP_ENOMEM;
  uint32_t at = 0;
  b->h_job_start[0] = 0;
  for (uint32_t w = 0; w < bp->nwaves; ++w) {
    for (int v = 0; v < kVariants; ++v) {
      bp->group_begin[w * kVariants + v] = at;
      std::vector<uint32_t> order;
      for (uint32_t i = 0; i < vj[v].size(); ++i)
        if (wave_of[vq[v][i]] == w) order.push_back(i);
      std::stable_sort(order.begin(), order.end(),
                       [&](uint32_t x, uint32_t y) { return qterms[vq[v][x]] < qterms[vq[v][y]]; });
      for (uint32_t i : order) {
        b->h_jobs[at] = vj[v][i];
        b->h_job_query[at] = vq[v][i];
        b->h_job_start[at + 1] = b->h_job_start[at] + vt[v][i];
        ++at;
      }
    }
  }
  bp->group_begin[bp->nwaves * kVariants] = at;
  uint32_t tat = 0;
  for (uint32_t w = 0; w < bp->nwaves; ++w) {
    bp->tail_begin[w] = tat;
    for (size_t i = 0; i < tails.size(); ++i)
      if (wave_of[tail_q[i]] == w) {
        b->h_tails[tat] = tails[i];
        b->h_tail_query[tat] = tail_q[i];
        ++tat;
      }
  }
  bp->tail_begin[bp->nwaves] = tat;
  bp->njobs = nj;
  bp->ntails = static_cast<uint32_t>(tails.size());
  std::copy(queries.begin(), queries.end(), b->h_queries);
  std::copy(jobs_left.begin(), jobs_left.end(), b->h_jobs_left);
  return BBP_OK;
}

}  // namespace bbp

#define BBP_TRY(expr)                              \
  do {                                             \
    if ((expr) != cudaSuccess) return BBP_ECUDA;   \
  } while (0)

namespace bbp {

// The prime form's workspaces for positions up to n; false if they cannot be had.
static bool prime_lanes(BatchState* b, uint64_t n, int lanes) {
  for (int i = 0; i < lanes; ++i) {
    if (!b->lane_stream[i] && cudaStreamCreateWithFlags(&b->lane_stream[i], cudaStreamNonBlocking) != cudaSuccess) return false;
    if (!b->lane_done[i] && cudaEventCreateWithFlags(&b->lane_done[i], cudaEventDisableTiming) != cudaSuccess) return false;
    if (!prime_workspace(&b->lane[i], n, kPrimeLaneListMax, b->lane_stream[i])) return false;
  }
  return true;
}

// One pass over the queries; by_primes: with the prime form where it serves.
static bbp_status run_batch(bbp_plan p, bbp_formula f, uint32_t count, const uint64_t* n, const uint32_t* P,
                            uint8_t* out, uint32_t out_stride, uint32_t* valid_bits, double* latency_ms,
                            bool by_primes) {
  BatchState* b = p->batch;
  // device buffers first (job descriptors hold accumulator addresses)
  if (!grow_device(&b->d_accum, &b->c_accum, static_cast<size_t>(count) * kMaxLimbs) ||
      !grow_device(&b->d_queries, &b->c_queries, count) || !grow_device(&b->d_jobs_left, &b->c_jobs_left, count) ||
      !grow_device(&b->d_out, &b->c_out, static_cast<size_t>(count) * kOutStride) ||
      !grow_device(&b->d_redo, &b->c_redo, count) || !grow_host(&b->h_redo, &b->hc_redo, count) ||
      !grow_device(&b->d_valid, &b->c_valid, count) || !grow_device(&b->d_done, &b->c_done, count + 1ull) ||
      !grow_host(&b->h_out, &b->hc_out, static_cast<size_t>(count) * kOutStride) ||
      !grow_host(&b->h_valid, &b->hc_valid, count) || !grow_host(&b->h_done, &b->hc_done, count + 1ull))
    return BBP_ENOMEM;
  if (!grow_device(&b->d_cursors, &b->c_cursors, static_cast<size_t>(kMaxWaves) * (kVariants + 1)))
    return BBP_ENOMEM;
  BatchPlan bp;
  bbp_status st = plan_batch(p, f, count, n, P, b, &bp, by_primes);
  if (st != BBP_OK) return st;
  const int lanes = static_cast<int>(std::min<size_t>(kPrimeLanes, bp.primes.size()));
  if (lanes > 0 && !prime_lanes(b, bp.primes.back().n, lanes)) {  // no memory for it: everything through the queue
    cudaGetLastError();
    bp = BatchPlan{};
    st = plan_batch(p, f, count, n, P, b, &bp, false);
    if (st != BBP_OK) return st;
  }
  if (!grow_device(&b->d_jobs, &b->c_jobs, bp.njobs) || !grow_device(&b->d_job_query, &b->c_job_query, bp.njobs) ||
      !grow_device(&b->d_job_start, &b->c_job_start, bp.njobs + 1ull) ||
      !grow_device(&b->d_job_done, &b->c_job_done, bp.njobs) ||
      !grow_device(&b->d_tails, &b->c_tails, bp.ntails) || !grow_device(&b->d_tail_query, &b->c_tail_query, bp.ntails))
    return BBP_ENOMEM;

  BatchDev dev{};
  dev.jobs = b->d_jobs;
  dev.job_query = b->d_job_query;
  dev.job_start = b->d_job_start;
  dev.job_done = b->d_job_done;
  dev.tails = b->d_tails;
  dev.tail_query = b->d_tail_query;
  dev.grab = static_cast<uint32_t>(p->grab);
  dev.queries = b->d_queries;
  dev.accum = b->d_accum;
  dev.jobs_left = b->d_jobs_left;
  dev.out = b->d_out;
  dev.valid = b->d_valid;
  dev.done_ns = b->d_done + 1;

  if (!b->stream && cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess) return BBP_ECUDA;
  if (!b->ready && cudaEventCreateWithFlags(&b->ready, cudaEventDisableTiming) != cudaSuccess) return BBP_ECUDA;
  // order after earlier work on the plan's stream, then run on the batch stream
  BBP_TRY(cudaEventRecord(b->ready, p->stream));
  BBP_TRY(cudaStreamWaitEvent(b->stream, b->ready, 0));
  cudaStream_t s = b->stream;
  // capture the pass
  cudaGraph_t graph = nullptr;
  BBP_TRY(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
  cudaError_t e = cudaSuccess;
  auto chk = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
  chk(cudaMemcpyAsync(b->d_jobs, b->h_jobs, sizeof(HeadArgs) * bp.njobs, cudaMemcpyHostToDevice, s));
  chk(cudaMemcpyAsync(b->d_job_query, b->h_job_query, sizeof(uint32_t) * bp.njobs, cudaMemcpyHostToDevice, s));
  chk(cudaMemcpyAsync(b->d_job_start, b->h_job_start, sizeof(uint64_t) * (bp.njobs + 1ull), cudaMemcpyHostToDevice, s));
  chk(cudaMemcpyAsync(b->d_tails, b->h_tails, sizeof(TailArgs) * bp.ntails, cudaMemcpyHostToDevice, s));
  chk(cudaMemcpyAsync(b->d_tail_query, b->h_tail_query, sizeof(uint32_t) * bp.ntails, cudaMemcpyHostToDevice, s));
  chk(cudaMemcpyAsync(b->d_queries, b->h_queries, sizeof(QueryDesc) * count, cudaMemcpyHostToDevice, s));
  chk(cudaMemcpyAsync(b->d_jobs_left, b->h_jobs_left, sizeof(unsigned int) * count, cudaMemcpyHostToDevice, s));
  chk(cudaMemsetAsync(b->d_job_done, 0, sizeof(unsigned long long) * bp.njobs, s));
  chk(cudaMemsetAsync(b->d_cursors, 0, sizeof(unsigned long long) * kMaxWaves * (kVariants + 1), s));
  chk(cudaMemsetAsync(b->d_accum, 0, sizeof(unsigned long long) * kMaxLimbs * count, s));
  chk(launch_timestamp(b->d_done, s));
  uint64_t launches = 1, head_launches = 0;
  for (uint32_t w = 0; w < bp.nwaves; ++w) {
    unsigned long long* cur = b->d_cursors + static_cast<size_t>(w) * (kVariants + 1);
    if (bp.tail_begin[w] < bp.tail_begin[w + 1]) {
      chk(launch_queue_tail(dev, bp.tail_begin[w], bp.tail_begin[w + 1], cur + kVariants, p->sm_count * 4, s));
      ++launches;
    }
    for (int v = 0; v < kVariants; ++v) {
      const uint32_t jb = bp.group_begin[w * kVariants + v], je = bp.group_begin[w * kVariants + v + 1];
      if (jb == je) continue;
      const int lmax = kLmaxClasses[v / kNumPaths], path = v % kNumPaths;
      // A small group: hand-outs for one CTA's warps an SM before they grow to `grab` tiles, and no more
      // CTAs than have hand-outs, but one an SM.  (With four tiles a hand-out and all CTAs that fit, the
      // first ones to come take everything, four CTAs on each of a few SMs.  One query of n = 1e6, P =
      // 448: Eq. 1 567 -> 212 us, Eq. 2 353 -> 149.)
      const uint64_t tiles = b->h_job_start[je] - b->h_job_start[jb], sms = static_cast<uint64_t>(p->sm_count);
      constexpr uint64_t kWarps = kHeadThreads / 32;
      BatchDev group = dev;
      group.grab = static_cast<uint32_t>(std::max<uint64_t>(1, std::min<uint64_t>(dev.grab, tiles / (kWarps * sms))));
      const uint64_t grabs = (tiles + group.grab - 1) / group.grab;
      const uint64_t want = std::max(std::min(sms, grabs), (grabs + kWarps - 1) / kWarps);
      const uint64_t fit = static_cast<uint64_t>(queue_occupancy(path, head_streams(p, path), lmax)) * sms;
      chk(launch_queue(group, jb, je, cur + v, path, head_streams(p, path), lmax, static_cast<int>(std::min(want, fit)), s));
      ++launches;
      ++head_launches;
    }
  }
  const cudaError_t ce = cudaStreamEndCapture(s, &graph);
  if (e != cudaSuccess || ce != cudaSuccess) {
    if (graph) cudaGraphDestroy(graph);
    return BBP_ECUDA;
  }
  bool updated = false;
  if (b->exec) {
    cudaGraphExecUpdateResultInfo info;
    updated = cudaGraphExecUpdate(b->exec, graph, &info) == cudaSuccess;
    if (!updated) {
      cudaGetLastError();
      cudaGraphExecDestroy(b->exec);
      b->exec = nullptr;
    }
  }
  if (!b->exec && cudaGraphInstantiate(&b->exec, graph, 0) != cudaSuccess) {
    cudaGraphDestroy(graph);
    b->exec = nullptr;
    return BBP_ECUDA;
  }
  cudaGraphDestroy(graph);
  if (p->profile) BBP_TRY(cudaEventRecord(p->ev0, s));
  BBP_TRY(cudaGraphLaunch(b->exec, s));
  if (!bp.primes.empty()) {
    BBP_TRY(cudaEventRecord(b->ready, s));
    const int used = static_cast<int>(std::min<size_t>(kPrimeLanes, bp.primes.size()));
    for (int i = 0; i < used; ++i) BBP_TRY(cudaStreamWaitEvent(b->lane_stream[i], b->ready, 0));
    for (size_t i = 0; i < bp.primes.size(); ++i) {
      BatchPlan::Prime& r = bp.primes[i];
      const int k = static_cast<int>(i % kPrimeLanes);
      const cudaStream_t to = b->lane_stream[k];
      PrimeRun run;
      r.planned = run.plan(b->lane[k], p->sm_count, f, r.n, r.W, b->d_accum + static_cast<uint64_t>(r.q) * kMaxLimbs) == BBP_OK;
      if (!r.planned) continue;  // by its terms, in the second pass
      bbp_status ls = run.begin(to);
      if (ls == BBP_OK) ls = run.run(0, run.lists(), to);
      if (ls == BBP_OK)
        ls = run.finish(P[r.q], r.bound, b->d_out + static_cast<size_t>(r.q) * kOutStride, b->d_valid + r.q,
                        b->d_redo + r.q, to);
      launches += run.launches();
      if (ls != BBP_OK) return ls;
      BBP_TRY(launch_timestamp(b->d_done + 1 + r.q, b->lane_stream[k]));
      ++launches;
    }
    for (int i = 0; i < used; ++i) {
      BBP_TRY(cudaEventRecord(b->lane_done[i], b->lane_stream[i]));
      BBP_TRY(cudaStreamWaitEvent(s, b->lane_done[i], 0));
    }
    BBP_TRY(cudaMemcpyAsync(b->h_redo, b->d_redo, sizeof(uint32_t) * count, cudaMemcpyDeviceToHost, s));
  }
  if (p->profile) BBP_TRY(cudaEventRecord(p->ev1, s));
  BBP_TRY(cudaMemcpyAsync(b->h_out, b->d_out, static_cast<size_t>(count) * kOutStride, cudaMemcpyDeviceToHost, s));
  BBP_TRY(cudaMemcpyAsync(b->h_valid, b->d_valid, sizeof(uint32_t) * count, cudaMemcpyDeviceToHost, s));
  BBP_TRY(cudaMemcpyAsync(b->h_done, b->d_done, sizeof(unsigned long long) * (count + 1ull), cudaMemcpyDeviceToHost, s));
  BBP_TRY(cudaStreamSynchronize(s));
  p->stats = bbp_stats{};
  p->stats.terms = bp.terms;
  p->stats.head_terms = bp.head_terms;
  p->stats.head_launches = head_launches;
  p->stats.kernel_launches = launches;
  p->stats.imad_model = bp.imad;
  if (p->profile) {
    float ms = 0;
    BBP_TRY(cudaEventElapsedTime(&ms, p->ev0, p->ev1));
    p->stats.head_ms = ms;
  }
  for (const BatchPlan::Prime& r : bp.primes)
    if (!r.planned) {  // nothing was written for it
      b->h_redo[r.q] = 1;
      b->h_done[1 + r.q] = b->h_done[0];
    }
  double last_ms = 0;
  for (uint32_t q = 0; q < count; ++q) {
    std::memcpy(out + static_cast<size_t>(q) * out_stride, b->h_out + static_cast<size_t>(q) * kOutStride,
                (P[q] + 7) / 8);
    valid_bits[q] = b->h_valid[q];
    latency_ms[q] = static_cast<double>(b->h_done[1 + q] - b->h_done[0]) * 1e-6;
    last_ms = std::max(last_ms, latency_ms[q]);
  }
  // queries that the check sends back to the terms: a second pass
  std::vector<uint32_t> again;
  for (const BatchPlan::Prime& r : bp.primes)
    if (b->h_redo[r.q]) again.push_back(r.q);
  if (!again.empty()) {
    const uint32_t m = static_cast<uint32_t>(again.size());
    std::vector<uint64_t> n2(m);
    std::vector<uint32_t> P2(m), valid2(m);
    std::vector<uint8_t> out2(static_cast<size_t>(m) * out_stride);
    std::vector<double> ms2(m);
    for (uint32_t i = 0; i < m; ++i) {
      n2[i] = n[again[i]];
      P2[i] = P[again[i]];
    }
    const bbp_stats first = p->stats;
    const bbp_status rs = run_batch(p, f, m, n2.data(), P2.data(), out2.data(), out_stride, valid2.data(), ms2.data(), false);
    if (rs != BBP_OK) return rs;
    const bbp_stats second = p->stats;
    p->stats = first;
    p->stats.head_launches += second.head_launches;
    p->stats.kernel_launches += second.kernel_launches;
    p->stats.imad_model += second.imad_model;
    p->stats.head_ms += second.head_ms;
    for (uint32_t i = 0; i < m; ++i) {
      const uint32_t q = again[i];
      std::memcpy(out + static_cast<size_t>(q) * out_stride, out2.data() + static_cast<size_t>(i) * out_stride,
                  (P[q] + 7) / 8);
      valid_bits[q] = valid2[i];
      latency_ms[q] = last_ms + ms2[i];
    }
  }
  return BBP_OK;
}

}  // namespace bbp

extern "C" bbp_status bbp_bits_batch(bbp_plan p, bbp_formula f, uint32_t count, const uint64_t* n, const uint32_t* P,
                                     uint8_t* out, uint32_t out_stride, uint32_t* valid_bits, double* latency_ms) {
  if (!p || (f != BBP_BELLARD && f != BBP_BBP) || (count && (!n || !P || !out))) return BBP_EINVAL;
  if (count == 0) return BBP_OK;
  if (count > kMaxQueueQueries) return BBP_EINVAL;
  uint32_t maxbytes = 0;
  for (uint32_t q = 0; q < count; ++q) maxbytes = std::max(maxbytes, (P[q] + 7) / 8);
  if (out_stride < maxbytes) return BBP_EINVAL;
  BBP_TRY(cudaSetDevice(p->device));
  if (!p->batch) {
    p->batch = new (std::nothrow) BatchState();
    if (!p->batch) return BBP_ENOMEM;
  }
  try {
    std::vector<uint32_t> valid(count);
    std::vector<double> ms(count);
    const bbp_status st = run_batch(p, f, count, n, P, out, out_stride, valid.data(), ms.data(), true);
    if (st != BBP_OK) {
      wait_batch(p->batch);
      return st;
    }
    if (valid_bits) std::copy(valid.begin(), valid.end(), valid_bits);
    if (latency_ms) std::copy(ms.begin(), ms.end(), latency_ms);
    if (p->strict)
      for (uint32_t q = 0; q < count; ++q)
        if (valid[q] < P[q]) return BBP_EINVALID_BITS;
  } catch (const std::bad_alloc&) {
    wait_batch(p->batch);
    return BBP_ENOMEM;
  }
  return BBP_OK;
}
