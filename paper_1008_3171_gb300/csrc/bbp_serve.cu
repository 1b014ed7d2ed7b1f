// Serving: continuous batching of bit-position queries (bbp_submit / bbp_poll).
//
// An engine thread owns a pool of device accumulator slots (admission is by free
// slots, i.e. by accumulator memory) and runs iterations.  Each iteration takes
// from every active query a piece of its remaining work -- at most a fair share of
// an iteration budget sized to a target duration from the measured throughput --
// so a long query is sliced over many iterations while short queries that arrive
// meanwhile join the next iteration and finish in one or two.  The pieces of an
// iteration are head-term ranges and tails of different queries, consumed by the
// same persistent queue kernels as a batch; each query's partial sums stay in its
// slot between iterations.  A query's job counter carries one extra hold while it
// has work left, so the device finalizes it (bits, certified count) exactly in the
// iteration that runs its last piece; the host then publishes the result to
// bbp_poll and frees the slot.
//
// Queries that the prime form serves (bbp_primes.h) run it instead: their tails go through
// the queue in their first iteration, their lists of primes through kServeLanes
// workspaces.  One that fits an iteration runs as a whole on the next free workspace; a
// longer one keeps a workspace, up to all but one of them, and runs some lists in each
// iteration.  A query whose check asks for the terms goes back to them.  48 queries of
// n = 10^6 ... 10^9 submitted together: 97 -> 13.7 ms.
//
// Iterations run one at a time: a query that
// arrives while one runs joins the next.  (Planning iteration i+1 while i runs was
// measured on the serving workload: the same terms/s, and every arrival waits one
// iteration longer, so the median latency rose from 46 to 72 ms.)
#include <cuda_runtime.h>

#include <algorithm>
#include <condition_variable>
#include <cstdint>
#include <cstring>
#include <deque>
#include <memory>
#include <mutex>
#include <new>
#include <thread>
#include <unordered_map>
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
constexpr uint32_t kOutStride = kMaxWorkingBits / 8;
constexpr double kIterTargetSeconds = 0.025;  // target duration of one iteration
constexpr double kInitialRate = 2.0e10;       // terms/s before the first measurement
constexpr int kServeLanes = 4;
// The work of a prime form in terms of the queue kernels: an eighth of its terms, and some
// 0.15 ms of launches and chains.
constexpr uint64_t kPrimeTermsPerTerm = 8, kPrimeFixedTerms = 6'000'000;

int lmax_index(int lmax) {
  for (int i = 0; i < kNumLmaxClasses; ++i)
    if (kLmaxClasses[i] == lmax) return i;
  return -1;
}

template <typename T>
bool grow_dev(T** p, size_t* cap, size_t want) {
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
bool grow_pinned(T** p, size_t* cap, size_t want) {
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

// A query's work: head ranges (HeadArgs without `slots`, with their tile count and
// kernel variant) and tail ranges, taken in order.
struct Work {
  bool tail;
  int variant;
  uint64_t tiles;  // head: warp tiles of the range
  uint64_t tile;   // head: terms per warp tile on the range's path
  HeadArgs head;
  TailArgs tailargs;
};

enum State { kPending = 0, kActive = 1, kDone = 2, kFailed = 3 };

struct Query {
  uint64_t ticket = 0;
  uint64_t n = 0;
  uint32_t P = 0, W = 0, L = 0;
  int slot = -1;
  int state = kPending;
  bbp_status error = BBP_OK;
  std::vector<Work> work;
  size_t next = 0;         // next work item
  uint64_t tile_off = 0;   // tiles of work[next] already handed out
  uint64_t bound = 0;      // N + J + 1
  uint64_t total_terms = 0;
  // prime form: `work` holds what it does not cover
  bool prime = false;
  std::unique_ptr<PrimeRun> run;  // once begun
  int lane = -1;                  // workspace kept between iterations
  size_t next_list = 0;
  uint64_t terms_done = 0;
  bbp_status broken = BBP_OK;     // could not be planned again: fails with this at the iteration's end
  bool final_in_flight = false;
  std::vector<uint8_t> out;
  uint32_t valid = 0;
};

}  // namespace

// Pinned host staging of one iteration: what it uploads, what it downloads, and
// the queries it finishes.
struct HostStage {
  HeadArgs* jobs = nullptr;          size_t c_jobs = 0;
  uint32_t* job_query = nullptr;     size_t c_job_query = 0;
  uint64_t* job_start = nullptr;     size_t c_job_start = 0;
  TailArgs* tails = nullptr;         size_t c_tails = 0;
  uint32_t* tail_query = nullptr;    size_t c_tail_query = 0;
  QueryDesc* queries = nullptr;      // one per slot
  unsigned int* jobs_left = nullptr; // one per slot
  uint8_t* out = nullptr;            // kOutStride bytes per slot
  uint32_t* valid = nullptr;         // one per slot
  uint32_t* redo = nullptr;          // one per slot (prime forms)
  cudaEvent_t start = nullptr, done = nullptr;
  std::vector<Query*> finishing;     // queries whose last piece runs in this iteration
  uint64_t terms = 0;                // terms of the iteration,
  uint64_t cost = 0;                 // and their work as queue terms
  bool in_flight = false;
};

struct ServeEngine {
  bbp_plan plan = nullptr;
  std::mutex mu;
  std::condition_variable cv;
  std::thread thread;
  bool stop = false;
  bool started = false;
  uint64_t next_ticket = 1;
  std::deque<Query*> pending;
  std::vector<Query*> active;        // admitted, with work left to hand out
  std::unordered_map<uint64_t, Query*> tickets;
  std::vector<int> free_slots;
  uint32_t max_slots = 0;
  double rate = kInitialRate;  // measured work, queue terms/s
  double terms_rate = kInitialRate;  // measured terms/s
  // prime forms
  PrimeState* lane[kServeLanes] = {};
  cudaStream_t lane_stream[kServeLanes] = {};
  cudaEvent_t lane_done[kServeLanes] = {};
  Query* lane_owner[kServeLanes] = {};
  bool no_lanes = false;             // workspaces could not be had: everything term by term
  uint32_t* d_redo = nullptr;
  std::vector<int> rezero;           // slots of queries that start again with their terms
  // device state (shared by consecutive iterations: stream order separates them)
  cudaStream_t stream = nullptr;
  cudaEvent_t queued = nullptr;      // the iteration's queue part, before its prime forms
  unsigned long long* d_accum = nullptr;
  QueryDesc* d_queries = nullptr;
  unsigned int* d_jobs_left = nullptr;
  uint8_t* d_out = nullptr;
  uint32_t* d_valid = nullptr;
  unsigned long long* d_done = nullptr;
  unsigned long long* d_cursors = nullptr;
  HeadArgs* d_jobs = nullptr;            size_t c_jobs = 0;
  uint32_t* d_job_query = nullptr;       size_t c_job_query = 0;
  uint64_t* d_job_start = nullptr;       size_t c_job_start = 0;
  unsigned long long* d_job_done = nullptr; size_t c_job_done = 0;
  TailArgs* d_tails = nullptr;           size_t c_tails = 0;
  uint32_t* d_tail_query = nullptr;      size_t c_tail_query = 0;
  HostStage stage;
  // statistics
  uint64_t iterations = 0;
  uint64_t terms_done = 0;
};

namespace {

// Host planning of one query into work items (the same ranges as bbp_bits); by_primes: only
// what the prime form leaves, where that serves.
bbp_status plan_query_work(bbp_plan p, uint64_t n, uint32_t P, Query* q, bool by_primes) {
  uint32_t W;
  if (n == 0 || !working_bits(P, p->guard, &W)) return BBP_EINVAL;
  const uint32_t L = W / 32;
  const int lmax = head_lmax_for(static_cast<int>(L));
  if (lmax == 0) return BBP_EINVAL;
  const FormulaDef& F = formula_def(BBP_BELLARD);
  std::vector<TermRange> ranges;
  uint64_t N = 0;
  for (uint32_t j = 0; j < F.count; ++j) {
    const int st = plan_series(F, j, n, W, static_cast<uint32_t>(lmax), 0, UINT64_MAX, ranges, p->wide_min_bits);
    if (st == -6) return BBP_ERANGE;
    if (st != 0) return BBP_EINVAL;
    N += natural_end(F, j, n - 1, W);
  }
  q->n = n;
  q->P = P;
  q->W = W;
  q->L = L;
  q->bound = N + F.count + 1;
  q->total_terms = 0;
  q->work.clear();
  uint64_t tiles = 0;
  for (const TermRange& r : ranges) {
    q->total_terms += r.count;
    if (!r.tail) tiles += (r.count + tile_terms(p, r.path) - 1) / tile_terms(p, r.path);
  }
  if (tiles > kMaxQueueTiles) return BBP_ERANGE;  // carry-save limbs could pass 2^64
  q->prime = by_primes && prime_form_serves(BBP_BELLARD, n, P, W, q->bound);
  if (q->prime) {
    const PrimeLimits lim = prime_limits(BBP_BELLARD, n - 1);
    ranges.clear();
    for (uint32_t j = 0; j < F.count; ++j)
      if (plan_series(F, j, n, W, static_cast<uint32_t>(lmax), prime_first_k(lim, j, n - 1), UINT64_MAX, ranges,
                      p->wide_min_bits) != 0)
        return BBP_EINVAL;
  }
  for (const TermRange& r : ranges) {
    const SeriesDef& s = F.s[r.j];
    Work w{};
    w.tail = r.tail != 0;
    if (w.tail) {
      TailArgs& a = w.tailargs;
      a.d = n - 1;
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
    } else {
      HeadArgs& a = w.head;
      a.d = n - 1;
      a.k_begin = r.k_begin;
      a.count = r.count;
      a.a = s.a;
      a.b = s.b;
      a.c = s.c;
      a.step = F.step;
      a.W = W;
      a.L = L;
      a.alternating = F.alternating;
      a.negate = s.sign < 0 ? 1u : 0u;  // the parity of the piece's first k is applied per piece
      a.run = static_cast<uint32_t>(p->run);
      a.window = r.window;
      a.first = r.first;
      a.first_max = r.first_max;
      w.tile = tile_terms(p, r.path);
      w.tiles = (r.count + w.tile - 1) / w.tile;
      w.variant = lmax_index(lmax) * kNumPaths + r.path;
    }
    q->work.push_back(w);
  }
  if (q->work.empty()) {  // nothing to sum: a zero-length tail still retires the query
    Work w{};
    w.tail = true;
    w.tailargs.W = W;
    w.tailargs.L = L;
    q->work.push_back(w);
  }
  return BBP_OK;
}

struct Piece {
  bool tail;
  int variant;
  uint64_t tiles;
  HeadArgs head;
  TailArgs tailargs;
  uint32_t slot;
};

// Takes about `budget_terms` terms (at least one item) of q's remaining work, in
// whole warp tiles of each range.
void take_pieces(ServeEngine* E, Query* q, uint64_t budget_terms, std::vector<Piece>& out, uint64_t* terms) {
  const FormulaDef& F = formula_def(BBP_BELLARD);
  unsigned long long* slots = E->d_accum + static_cast<uint64_t>(q->slot) * kMaxLimbs;
  bool first = true;
  while (q->next < q->work.size() && (first || budget_terms > 0)) {
    first = false;
    Work& w = q->work[q->next];
    Piece pc{};
    pc.slot = static_cast<uint32_t>(q->slot);
    pc.tail = w.tail;
    if (w.tail) {
      pc.tailargs = w.tailargs;
      pc.tailargs.slots = slots;
      *terms += w.tailargs.count;
      budget_terms = budget_terms > w.tailargs.count ? budget_terms - w.tailargs.count : 0;
      ++q->next;
      q->tile_off = 0;
    } else {
      const uint64_t tile = w.tile;
      const uint64_t avail = w.tiles - q->tile_off;
      const uint64_t take = std::max<uint64_t>(1, std::min(avail, budget_terms / tile));
      HeadArgs a = w.head;
      a.k_begin = w.head.k_begin + q->tile_off * tile;
      const uint64_t end = std::min(w.head.k_begin + w.head.count, a.k_begin + take * tile);
      a.count = end - a.k_begin;
      const bool neg_series = w.head.negate != 0;
      a.negate = (neg_series != (F.alternating && (a.k_begin & 1ull))) ? 1u : 0u;
      a.slots = slots;
      pc.head = a;
      pc.variant = w.variant;
      pc.tiles = (a.count + tile - 1) / tile;
      *terms += a.count;
      budget_terms = budget_terms > take * tile ? budget_terms - take * tile : 0;
      q->tile_off += take;
      if (q->tile_off >= w.tiles) {
        ++q->next;
        q->tile_off = 0;
      }
    }
    out.push_back(pc);
  }
}

bool alloc_engine(ServeEngine* E) {
  const size_t S = E->max_slots;
  bool ok = cudaStreamCreateWithFlags(&E->stream, cudaStreamNonBlocking) == cudaSuccess &&
            cudaEventCreateWithFlags(&E->queued, cudaEventDisableTiming) == cudaSuccess &&
            cudaMalloc(&E->d_accum, sizeof(unsigned long long) * kMaxLimbs * S) == cudaSuccess &&
            cudaMalloc(&E->d_queries, sizeof(QueryDesc) * S) == cudaSuccess &&
            cudaMalloc(&E->d_jobs_left, sizeof(unsigned int) * S) == cudaSuccess &&
            cudaMalloc(&E->d_out, static_cast<size_t>(kOutStride) * S) == cudaSuccess &&
            cudaMalloc(&E->d_valid, sizeof(uint32_t) * S) == cudaSuccess &&
            cudaMalloc(&E->d_redo, sizeof(uint32_t) * S) == cudaSuccess &&
            cudaMalloc(&E->d_done, sizeof(unsigned long long) * S) == cudaSuccess &&
            cudaMalloc(&E->d_cursors, sizeof(unsigned long long) * (kVariants + 1)) == cudaSuccess;
  {
    HostStage& h = E->stage;
    ok = ok && cudaMallocHost(&h.queries, sizeof(QueryDesc) * S) == cudaSuccess &&
         cudaMallocHost(&h.jobs_left, sizeof(unsigned int) * S) == cudaSuccess &&
         cudaMallocHost(&h.out, static_cast<size_t>(kOutStride) * S) == cudaSuccess &&
         cudaMallocHost(&h.valid, sizeof(uint32_t) * S) == cudaSuccess &&
         cudaMallocHost(&h.redo, sizeof(uint32_t) * S) == cudaSuccess &&
         cudaEventCreate(&h.start) == cudaSuccess && cudaEventCreate(&h.done) == cudaSuccess;
    if (ok) {
      std::memset(h.queries, 0, sizeof(QueryDesc) * S);
      std::memset(h.jobs_left, 0, sizeof(unsigned int) * S);
    }
  }
  return ok;
}

void free_engine(ServeEngine* E) {
  if (E->stream) cudaStreamSynchronize(E->stream);
  for (int i = 0; i < kServeLanes; ++i) {
    if (E->lane_stream[i]) cudaStreamSynchronize(E->lane_stream[i]);
    release_prime_state(&E->lane[i]);
    if (E->lane_stream[i]) cudaStreamDestroy(E->lane_stream[i]);
    if (E->lane_done[i]) cudaEventDestroy(E->lane_done[i]);
  }
  cudaFree(E->d_redo);
  cudaFree(E->d_accum);
  cudaFree(E->d_queries);
  cudaFree(E->d_jobs_left);
  cudaFree(E->d_out);
  cudaFree(E->d_valid);
  cudaFree(E->d_done);
  cudaFree(E->d_cursors);
  cudaFree(E->d_jobs);
  cudaFree(E->d_job_query);
  cudaFree(E->d_job_start);
  cudaFree(E->d_job_done);
  cudaFree(E->d_tails);
  cudaFree(E->d_tail_query);
  {
    HostStage& h = E->stage;
    cudaFreeHost(h.jobs);
    cudaFreeHost(h.job_query);
    cudaFreeHost(h.job_start);
    cudaFreeHost(h.tails);
    cudaFreeHost(h.tail_query);
    cudaFreeHost(h.queries);
    cudaFreeHost(h.jobs_left);
    cudaFreeHost(h.out);
    cudaFreeHost(h.valid);
    cudaFreeHost(h.redo);
    if (h.start) cudaEventDestroy(h.start);
    if (h.done) cudaEventDestroy(h.done);
  }
  if (E->queued) cudaEventDestroy(E->queued);
  if (E->stream) cudaStreamDestroy(E->stream);
}

uint64_t prime_cost(const Query* q) { return q->total_terms / kPrimeTermsPerTerm + kPrimeFixedTerms; }

// All workspaces, made when the first query needs one.
bool make_lanes(ServeEngine* E) {
  if (E->no_lanes) return false;
  for (int i = 0; i < kServeLanes; ++i) {
    if ((!E->lane_stream[i] && cudaStreamCreateWithFlags(&E->lane_stream[i], cudaStreamNonBlocking) != cudaSuccess) ||
        (!E->lane_done[i] && cudaEventCreateWithFlags(&E->lane_done[i], cudaEventDisableTiming) != cudaSuccess) ||
        !prime_workspace(&E->lane[i], kPrimeMaxN, kPrimeLaneListMax, E->lane_stream[i])) {
      cudaGetLastError();
      E->no_lanes = true;
      return false;
    }
  }
  return true;
}

// Back to the terms for a query that has not begun; if they cannot be planned it leaves with
// this iteration, without a result.
void plan_by_terms(ServeEngine* E, Query* q) {
  q->run.reset();
  q->broken = plan_query_work(E->plan, q->n, q->P, q, false);
  if (q->broken == BBP_OK) return;
  q->prime = false;
  q->work.clear();
}

// What an iteration does for one query by primes: its lists [first, last) on a workspace.
struct PrimePart {
  Query* q;
  int lane;
  size_t first, last;
};

// Chooses the iteration's parts, in the order of the active queries, for about
// `budget` queue terms; sets what it takes in each query.
void take_primes(ServeEngine* E, std::vector<Query*>& batch, uint64_t budget, std::vector<PrimePart>& parts,
                 std::vector<Query*>& begun, uint64_t* terms, uint64_t* cost) {
  uint64_t taken = 0;
  int turn = 0;
  for (Query* q : batch) {
    if (!q->prime) continue;
    const uint64_t whole = prime_cost(q);
    const bool is_long = whole > budget;
    if (q->lane < 0) {
      if (taken >= budget && !parts.empty()) continue;  // waits for the next iteration
      int free_lane = -1, held = 0;
      for (int k = 0; k < kServeLanes; ++k) {
        const int i = (turn + k) % kServeLanes;
        if (E->lane_owner[i]) ++held;
        else if (free_lane < 0) free_lane = i;
      }
      if (free_lane < 0 || (is_long && held >= kServeLanes - 1)) continue;
      q->run.reset(new (std::nothrow) PrimeRun());
      const uint64_t slot = static_cast<uint64_t>(q->slot);
      if (!q->run || q->run->plan(E->lane[free_lane], E->plan->sm_count, BBP_BELLARD, q->n, q->W,
                                  E->d_accum + slot * kMaxLimbs) != BBP_OK) {
        plan_by_terms(E, q);
        continue;
      }
      q->next_list = 0;
      turn = free_lane + 1;
      begun.push_back(q);
      if (is_long) {
        q->lane = free_lane;
        E->lane_owner[free_lane] = q;
      } else {
        parts.push_back(PrimePart{q, free_lane, 0, q->run->lists()});
        q->next_list = q->run->lists();
        *terms += q->total_terms;
        *cost += whole;
        taken += whole;
        continue;
      }
    }
    // some lists of a long query
    const size_t first = q->next_list;
    uint64_t part = 0;
    while (q->next_list < q->run->lists() && (part == 0 || part < budget / kServeLanes))
      part += std::max<uint64_t>(1, static_cast<uint64_t>(q->run->share(q->next_list++) * static_cast<double>(whole)));
    parts.push_back(PrimePart{q, q->lane, first, q->next_list});
    const uint64_t done = q->next_list == q->run->lists()
                              ? q->total_terms
                              : std::min(q->total_terms, q->terms_done + part * kPrimeTermsPerTerm);
    *terms += done - q->terms_done;
    q->terms_done = done;
    *cost += part;
    taken += part;
  }
}

// Plans one iteration over the active queries into staging H and enqueues it
// (uploads, launches, result download, events).  Queries whose
// last piece is in it move to H.finishing.  Returns false on a CUDA error.
bool enqueue_iteration(ServeEngine* E, HostStage& H, std::vector<Query*>& batch, std::vector<int>& fresh_slots) {
  bbp_plan p = E->plan;
  const uint64_t budget_terms = std::max<uint64_t>(1, static_cast<uint64_t>(E->rate * kIterTargetSeconds));
  std::vector<Piece> pieces;
  std::vector<PrimePart> parts;
  std::vector<Query*> begun;
  uint64_t terms = 0, cost = 0, prime_terms = 0;
  std::vector<uint32_t> npieces(batch.size(), 0);
  H.finishing.clear();
  bool primes = false;
  for (Query* q : batch) primes |= q->prime;
  if (primes && !make_lanes(E))
    for (Query* q : batch)
      if (q->prime) plan_by_terms(E, q);
  size_t by_terms = 0;
  for (Query* q : batch) by_terms += q->prime ? 0 : 1;
  // half of an iteration for either kind while there are both
  take_primes(E, batch, by_terms ? budget_terms / 2 : budget_terms, parts, begun, &prime_terms, &cost);
  const uint64_t share = std::max<uint64_t>(1, (budget_terms - std::min(cost, budget_terms / 2)) / std::max<size_t>(1, by_terms));
  for (size_t i = 0; i < batch.size(); ++i) {
    Query* q = batch[i];
    const size_t before = pieces.size();
    if (q->prime) {  // its few other terms with its first lists
      uint64_t few = 0;
      if (std::find(begun.begin(), begun.end(), q) != begun.end()) take_pieces(E, q, UINT64_MAX, pieces, &few);
      q->final_in_flight = q->run && q->next_list == q->run->lists();
    } else {
      take_pieces(E, q, share, pieces, &terms);
      q->final_in_flight = q->next >= q->work.size();
    }
    npieces[i] = static_cast<uint32_t>(pieces.size() - before);
    if (q->final_in_flight) H.finishing.push_back(q);
  }
  H.terms = terms + prime_terms;
  H.cost = terms + cost;
  // group head pieces by variant, tails apart
  std::vector<uint32_t> vb(kVariants + 1, 0);
  std::vector<const Piece*> heads, tails;
  for (int v = 0; v < kVariants; ++v) {
    vb[v] = static_cast<uint32_t>(heads.size());
    for (const Piece& pc : pieces)
      if (!pc.tail && pc.variant == v) heads.push_back(&pc);
  }
  vb[kVariants] = static_cast<uint32_t>(heads.size());
  for (const Piece& pc : pieces)
    if (pc.tail) tails.push_back(&pc);
  const size_t nh = heads.size(), nt = tails.size();
  if (!grow_pinned(&H.jobs, &H.c_jobs, nh) || !grow_pinned(&H.job_query, &H.c_job_query, nh) ||
      !grow_pinned(&H.job_start, &H.c_job_start, nh + 1) || !grow_pinned(&H.tails, &H.c_tails, nt) ||
      !grow_pinned(&H.tail_query, &H.c_tail_query, nt) || !grow_dev(&E->d_jobs, &E->c_jobs, nh) ||
      !grow_dev(&E->d_job_query, &E->c_job_query, nh) || !grow_dev(&E->d_job_start, &E->c_job_start, nh + 1) ||
      !grow_dev(&E->d_job_done, &E->c_job_done, nh) || !grow_dev(&E->d_tails, &E->c_tails, nt) ||
      !grow_dev(&E->d_tail_query, &E->c_tail_query, nt))
    return false;
  H.job_start[0] = 0;
  for (size_t i = 0; i < nh; ++i) {
    H.jobs[i] = heads[i]->head;
    H.job_query[i] = heads[i]->slot;
    H.job_start[i + 1] = H.job_start[i] + heads[i]->tiles;
  }
  for (size_t i = 0; i < nt; ++i) {
    H.tails[i] = tails[i]->tailargs;
    H.tail_query[i] = tails[i]->slot;
  }
  for (size_t i = 0; i < batch.size(); ++i) {
    Query* q = batch[i];
    QueryDesc& Q = H.queries[q->slot];
    Q.bound = q->bound;
    Q.P = q->P;
    Q.L = q->L;
    Q.out_offset = static_cast<uint32_t>(q->slot) * kOutStride;
    // held while work remains, and for a prime form, whose check writes the result
    H.jobs_left[q->slot] = npieces[i] + (q->final_in_flight && !q->prime ? 0u : 1u);
  }
  cudaStream_t s = E->stream;
  cudaError_t e = cudaSuccess;
  auto chk = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
  chk(cudaEventRecord(H.start, s));
  for (int slot : fresh_slots)
    chk(cudaMemsetAsync(E->d_accum + static_cast<uint64_t>(slot) * kMaxLimbs, 0,
                        sizeof(unsigned long long) * kMaxLimbs, s));
  // the whole slot tables in two copies (slots not in this iteration have no jobs)
  chk(cudaMemcpyAsync(E->d_queries, H.queries, sizeof(QueryDesc) * E->max_slots, cudaMemcpyHostToDevice, s));
  chk(cudaMemcpyAsync(E->d_jobs_left, H.jobs_left, sizeof(unsigned int) * E->max_slots, cudaMemcpyHostToDevice, s));
  chk(cudaMemcpyAsync(E->d_jobs, H.jobs, sizeof(HeadArgs) * nh, cudaMemcpyHostToDevice, s));
  chk(cudaMemcpyAsync(E->d_job_query, H.job_query, sizeof(uint32_t) * nh, cudaMemcpyHostToDevice, s));
  chk(cudaMemcpyAsync(E->d_job_start, H.job_start, sizeof(uint64_t) * (nh + 1), cudaMemcpyHostToDevice, s));
  chk(cudaMemcpyAsync(E->d_tails, H.tails, sizeof(TailArgs) * nt, cudaMemcpyHostToDevice, s));
  chk(cudaMemcpyAsync(E->d_tail_query, H.tail_query, sizeof(uint32_t) * nt, cudaMemcpyHostToDevice, s));
  chk(cudaMemsetAsync(E->d_job_done, 0, sizeof(unsigned long long) * std::max<size_t>(nh, 1), s));
  chk(cudaMemsetAsync(E->d_cursors, 0, sizeof(unsigned long long) * (kVariants + 1), s));
  BatchDev dev{};
  dev.jobs = E->d_jobs;
  dev.job_query = E->d_job_query;
  dev.job_start = E->d_job_start;
  dev.job_done = E->d_job_done;
  dev.tails = E->d_tails;
  dev.tail_query = E->d_tail_query;
  dev.grab = 1;  // short iterations: hand out single tiles so every launch ends evenly
  dev.queries = E->d_queries;
  dev.accum = E->d_accum;
  dev.jobs_left = E->d_jobs_left;
  dev.out = E->d_out;
  dev.valid = E->d_valid;
  dev.done_ns = E->d_done;
  chk(launch_queue_tail(dev, 0, static_cast<uint32_t>(nt), E->d_cursors + kVariants, p->sm_count * 4, s));
  for (int v = 0; v < kVariants; ++v) {
    if (vb[v] == vb[v + 1]) continue;
    const int lmax = kLmaxClasses[v / kNumPaths], path = v % kNumPaths;
    const int blocks = queue_occupancy(path, head_streams(p, path), lmax) * p->sm_count;
    chk(launch_queue(dev, vb[v], vb[v + 1], E->d_cursors + v, path, head_streams(p, path), lmax, blocks, s));
  }
  if (!parts.empty()) {
    bool used[kServeLanes] = {};
    chk(cudaEventRecord(E->queued, s));
    for (const PrimePart& part : parts) {
      const cudaStream_t to = E->lane_stream[part.lane];
      const size_t slot = static_cast<size_t>(part.q->slot);
      PrimeRun& run = *part.q->run;
      if (!used[part.lane]) chk(cudaStreamWaitEvent(to, E->queued, 0));
      used[part.lane] = true;
      bool ok = part.first != 0 || run.begin(to) == BBP_OK;
      ok = ok && run.run(part.first, part.last, to) == BBP_OK;
      if (part.last == run.lists())
        ok = ok && run.finish(part.q->P, part.q->bound, E->d_out + slot * kOutStride, E->d_valid + slot,
                              E->d_redo + slot, to) == BBP_OK;
      if (!ok) chk(cudaErrorUnknown);
    }
    for (int i = 0; i < kServeLanes; ++i) {
      if (!used[i]) continue;
      chk(cudaEventRecord(E->lane_done[i], E->lane_stream[i]));
      chk(cudaStreamWaitEvent(s, E->lane_done[i], 0));
    }
    chk(cudaMemcpyAsync(H.redo, E->d_redo, sizeof(uint32_t) * E->max_slots, cudaMemcpyDeviceToHost, s));
  }
  if (!H.finishing.empty()) {  // results of the queries that finish in this iteration
    chk(cudaMemcpyAsync(H.out, E->d_out, static_cast<size_t>(kOutStride) * E->max_slots, cudaMemcpyDeviceToHost, s));
    chk(cudaMemcpyAsync(H.valid, E->d_valid, sizeof(uint32_t) * E->max_slots, cudaMemcpyDeviceToHost, s));
  }
  chk(cudaEventRecord(H.done, s));
  H.in_flight = e == cudaSuccess;
  return e == cudaSuccess;
}

// Waits for an enqueued iteration and publishes the queries it finished (under
// E->mu, which bbp_poll and bbp_serve_stats take too).
bool finish_iteration(ServeEngine* E, HostStage& H) {
  if (!H.in_flight) return true;
  H.in_flight = false;
  if (cudaEventSynchronize(H.done) != cudaSuccess) return false;
  float ms = 0;
  const bool timed = cudaEventElapsedTime(&ms, H.start, H.done) == cudaSuccess && ms > 0.1f && H.terms > 0;
  std::lock_guard<std::mutex> lock(E->mu);
  if (timed) {
    // a short iteration is mostly launches: it says little about the rate of a full one
    const double w = 0.3 * std::min(1.0, ms / 5.0);
    E->rate = (1.0 - w) * E->rate + w * (static_cast<double>(H.cost) / (1e-3 * ms));
    E->terms_rate = 0.7 * E->terms_rate + 0.3 * (static_cast<double>(H.terms) / (1e-3 * ms));
  }
  E->iterations++;
  E->terms_done += H.terms;
  for (Query* q : H.finishing) {
    if (q->lane >= 0) E->lane_owner[q->lane] = nullptr;
    q->lane = -1;
    q->run.reset();
    if (q->prime && H.redo[q->slot] != 0) {  // too close to a carry: the terms decide
      E->terms_done -= q->total_terms;
      q->next = 0;
      q->tile_off = 0;
      q->final_in_flight = false;
      plan_by_terms(E, q);
      if (q->broken == BBP_OK) {
        E->rezero.push_back(q->slot);
        E->active.push_back(q);
        continue;
      }
    }
    if (q->broken != BBP_OK) {
      q->state = kFailed;
      q->error = q->broken;
      E->free_slots.push_back(q->slot);
      q->slot = -1;
      continue;
    }
    q->out.assign(H.out + static_cast<size_t>(q->slot) * kOutStride,
                  H.out + static_cast<size_t>(q->slot) * kOutStride + (q->P + 7) / 8);
    q->valid = H.valid[q->slot];
    q->state = kDone;
    E->free_slots.push_back(q->slot);
    q->slot = -1;
    q->work.clear();
    q->work.shrink_to_fit();
  }
  H.finishing.clear();
  return true;
}

// An iteration could not be enqueued or did not complete: every admitted query
// fails (bbp_poll returns BBP_ECUDA) and gives its slot back, so that later
// submissions are admitted again (a fresh slot is zeroed on admission).  What the iteration
// has queued ends first: none of it may add to a slot that has a new query.
void fail_all(ServeEngine* E) {
  cudaStreamSynchronize(E->stream);
  for (int i = 0; i < kServeLanes; ++i) {
    if (E->lane_stream[i]) cudaStreamSynchronize(E->lane_stream[i]);
    wait_prime_state(E->lane[i]);
  }
  std::lock_guard<std::mutex> lock(E->mu);
  auto fail = [&](Query* q) {
    q->state = kFailed;
    q->error = BBP_ECUDA;
    if (q->slot >= 0) E->free_slots.push_back(q->slot);
    q->slot = -1;
    if (q->lane >= 0) E->lane_owner[q->lane] = nullptr;
    q->lane = -1;
    q->run.reset();
    q->work.clear();
  };
  for (Query* q : E->stage.finishing) fail(q);
  E->stage.finishing.clear();
  E->stage.in_flight = false;
  for (Query* q : E->active) fail(q);
  E->active.clear();
}

void engine_main(ServeEngine* E) {
  cudaSetDevice(E->plan->device);
  for (;;) {
    std::vector<Query*> batch;
    std::vector<int> fresh;
    {
      std::unique_lock<std::mutex> lock(E->mu);
      E->cv.wait(lock, [&] { return E->stop || !E->pending.empty() || !E->active.empty(); });
      if (E->stop) return;
      while (!E->pending.empty() && !E->free_slots.empty()) {  // admission by free accumulator slots
        Query* q = E->pending.front();
        E->pending.pop_front();
        q->slot = E->free_slots.back();
        E->free_slots.pop_back();
        q->state = kActive;
        E->active.push_back(q);
        fresh.push_back(q->slot);
      }
      fresh.insert(fresh.end(), E->rezero.begin(), E->rezero.end());
      E->rezero.clear();
      batch = E->active;
    }
    bool ok = enqueue_iteration(E, E->stage, batch, fresh);
    {
      std::lock_guard<std::mutex> lock(E->mu);  // queries handed out completely leave the active list
      std::vector<Query*> still;
      for (Query* q : E->active)
        if (!q->final_in_flight) still.push_back(q);
      E->active.swap(still);
    }
    ok = ok && finish_iteration(E, E->stage);
    if (!ok) fail_all(E);
  }
}

ServeEngine* engine_of(bbp_plan p, bbp_status* st) {
  *st = BBP_OK;
  if (p->serve) return p->serve;
  ServeEngine* E = new (std::nothrow) ServeEngine();
  if (!E) {
    *st = BBP_ENOMEM;
    return nullptr;
  }
  E->plan = p;
  const size_t per_slot = sizeof(unsigned long long) * kMaxLimbs + kOutStride + 64;
  E->max_slots = static_cast<uint32_t>(
      std::max<size_t>(1, std::min<size_t>({p->max_slots, p->accum_budget / per_slot, kMaxQueueQueries})));
  cudaSetDevice(p->device);
  if (!alloc_engine(E)) {
    free_engine(E);
    delete E;
    *st = BBP_ENOMEM;
    return nullptr;
  }
  for (int s = static_cast<int>(E->max_slots) - 1; s >= 0; --s) E->free_slots.push_back(s);
  E->thread = std::thread(engine_main, E);
  E->started = true;
  p->serve = E;
  return E;
}

}  // namespace

namespace bbp {

void release_serve_state(bbp_plan p) {
  ServeEngine* E = p->serve;
  if (!E) return;
  {
    std::lock_guard<std::mutex> lock(E->mu);
    E->stop = true;
  }
  E->cv.notify_all();
  if (E->thread.joinable()) E->thread.join();
  if (E->stream) cudaStreamSynchronize(E->stream);
  for (auto& kv : E->tickets) delete kv.second;
  free_engine(E);
  delete E;
  p->serve = nullptr;
}

}  // namespace bbp

extern "C" {

bbp_status bbp_submit(bbp_plan p, uint64_t n, uint32_t P, bbp_ticket* t) {
  if (!p || !t) return BBP_EINVAL;
  Query* q = new (std::nothrow) Query();
  if (!q) return BBP_ENOMEM;
  const bbp_status ps = plan_query_work(p, n, P, q, true);
  if (ps != BBP_OK) {
    delete q;
    return ps;
  }
  bbp_status st;
  ServeEngine* E = engine_of(p, &st);
  if (!E) {
    delete q;
    return st;
  }
  {
    std::lock_guard<std::mutex> lock(E->mu);
    // admission: a query waits for a slot only while the queue is shorter than the pool
    if (E->pending.size() >= E->max_slots) {
      delete q;
      return BBP_EBUSY;
    }
    q->ticket = E->next_ticket++;
    E->tickets[q->ticket] = q;
    E->pending.push_back(q);
    *t = q->ticket;
  }
  E->cv.notify_all();
  return BBP_OK;
}

bbp_status bbp_poll(bbp_plan p, bbp_ticket t, uint8_t* out, uint32_t* valid_bits) {
  if (!p) return BBP_EINVAL;
  ServeEngine* E = p->serve;
  if (!E) return BBP_ENOTFOUND;
  std::lock_guard<std::mutex> lock(E->mu);
  auto it = E->tickets.find(t);
  if (it == E->tickets.end()) return BBP_ENOTFOUND;
  Query* q = it->second;
  if (q->state == kPending || q->state == kActive) return BBP_PENDING;
  const bbp_status st = q->state == kFailed ? q->error : BBP_OK;
  if (st == BBP_OK) {
    if (out) std::memcpy(out, q->out.data(), q->out.size());
    if (valid_bits) *valid_bits = q->valid;
  }
  E->tickets.erase(it);
  delete q;
  return st;
}

bbp_status bbp_serve_stats(bbp_plan p, bbp_serve_info* info) {
  if (!p || !info) return BBP_EINVAL;
  std::memset(info, 0, sizeof(*info));
  ServeEngine* E = p->serve;
  if (!E) return BBP_OK;
  std::lock_guard<std::mutex> lock(E->mu);
  info->pending = E->pending.size();
  info->active = E->active.size();
  info->slots = E->max_slots;
  info->iterations = E->iterations;
  info->terms = E->terms_done;
  info->terms_per_s = E->terms_rate;
  return BBP_OK;
}

}  // extern "C"
