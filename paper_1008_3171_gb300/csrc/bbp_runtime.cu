// C ABI of libbbp (include/bbp.h): plans, single-query paths and statistics.
//
// A query (Sze, arXiv:1008.3171, Sec. 3) is planned on the host into term ranges
// (bbp_planner.cpp), each range is one kernel launch (bbp_kernels.cu) that folds
// its signed partial sum into L carry-save 64-bit accumulators on the device, and
// a finalize kernel turns the accumulators into the W-bit sum, the certified bit
// count and the top P bits.  Nothing of the arithmetic runs on the host.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "bbp.h"
#include "bbp_kernels.cuh"
#include "bbp_planner.h"
#include "bbp_prime_run.h"
#include "bbp_primes.h"
#include "bbp_runtime.h"

using namespace bbp;

namespace bbp {

bbp_status cuda_status(cudaError_t e) { return e == cudaSuccess ? BBP_OK : BBP_ECUDA; }

}  // namespace bbp

#define BBP_CUDA(expr)                                  \
  do {                                                  \
    cudaError_t e_ = (expr);                            \
    if (e_ != cudaSuccess) return BBP_ECUDA;            \
  } while (0)

namespace {

constexpr uint32_t kDefaultGuard = 64;
constexpr int kDefaultRun = 64;

bool valid_formula(int f) { return f == BBP_BELLARD || f == BBP_BBP; }

int pick_lmax(uint32_t W, int bump) { return head_lmax_for(static_cast<int>(W / 32), bump); }

}  // namespace

extern "C" {

uint32_t bbp_abi_version(void) { return BBP_ABI_VERSION; }

const char* bbp_status_str(bbp_status s) {
  switch (s) {
    case BBP_OK: return "ok";
    case BBP_PENDING: return "pending";
    case BBP_EINVAL: return "invalid argument";
    case BBP_ENOMEM: return "out of memory";
    case BBP_ECUDA: return "CUDA error";
    case BBP_EBUSY: return "busy: no slot or accumulator memory free";
    case BBP_ETIMEOUT: return "bounded device wait expired";
    case BBP_ERANGE: return "position out of range (modulus would reach 2^60)";
    case BBP_EINVALID_BITS: return "fewer bits certified than requested";
    case BBP_ENOTFOUND: return "unknown ticket";
    case BBP_ESCRATCH: return "working precision exceeds the fixed scratch of the no-allocation entry point";
  }
  return "unknown status";
}

void bbp_plan_opts_default(bbp_plan_opts* o) {
  if (!o) return;
  std::memset(o, 0, sizeof(*o));
  o->guard_bits = kDefaultGuard;
}

bbp_status bbp_plan_create(bbp_plan* out, const bbp_plan_opts* opts) {
  if (!out) return BBP_EINVAL;
  *out = nullptr;
  bbp_plan_opts o;
  bbp_plan_opts_default(&o);
  if (opts) o = *opts;
  if (o.guard_bits == 0) o.guard_bits = kDefaultGuard;
  if (o.guard_bits % 32 != 0 || o.guard_bits >= kMaxWorkingBits) return BBP_EINVAL;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) return BBP_ECUDA;
  if (o.device < 0 || o.device >= ndev) return BBP_EINVAL;
  BBP_CUDA(cudaSetDevice(o.device));
  bbp_plan p = new (std::nothrow) bbp_plan_s();
  if (!p) return BBP_ENOMEM;
  p->device = o.device;
  p->guard = o.guard_bits;
  p->profile = o.profile != 0;
  p->strict = o.strict != 0;
  p->accum_budget = o.accum_mem_budget ? o.accum_mem_budget : (64u << 20);
  p->max_slots = o.max_slots ? o.max_slots : 4096u;
  p->run = kDefaultRun;
  p->streams = 0;
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, o.device) != cudaSuccess) {
    delete p;
    return BBP_ECUDA;
  }
  p->sm_count = prop.multiProcessorCount;
  if (o.stream) {
    p->stream = static_cast<cudaStream_t>(o.stream);
    p->own_stream = false;
  } else {
    if (cudaStreamCreateWithFlags(&p->stream, cudaStreamNonBlocking) != cudaSuccess) {
      delete p;
      return BBP_ECUDA;
    }
    p->own_stream = true;
  }
  bool ok = cudaMalloc(&p->d_slots, sizeof(unsigned long long) * kMaxLimbs) == cudaSuccess &&
            cudaMalloc(&p->d_limbs, sizeof(uint32_t) * kMaxLimbs) == cudaSuccess &&
            cudaMalloc(&p->d_query, sizeof(unsigned long long) * (kMaxLimbs + 1)) == cudaSuccess &&
            cudaMalloc(&p->d_redo, sizeof(uint32_t)) == cudaSuccess &&
            cudaMallocHost(&p->h_stage, 4096) == cudaSuccess &&
            cudaEventCreate(&p->ev0) == cudaSuccess && cudaEventCreate(&p->ev1) == cudaSuccess &&
            cudaEventCreate(&p->ev2) == cudaSuccess;
  if (!ok) {
    bbp_plan_destroy(p);
    return BBP_ENOMEM;
  }
  if (o.tune_table) load_tune_table(p, o.tune_table);
  *out = p;
  return BBP_OK;
}

bbp_status bbp_plan_destroy(bbp_plan p) {
  if (!p) return BBP_OK;
  cudaSetDevice(p->device);
  release_serve_state(p);
  if (p->stream) cudaStreamSynchronize(p->stream);
  release_batch_state(p);
  release_prime_state(&p->primes);
  cudaFree(p->d_slots);
  cudaFree(p->d_limbs);
  cudaFree(p->d_query);
  cudaFree(p->d_redo);
  cudaFreeHost(p->h_stage);
  if (p->ev0) cudaEventDestroy(p->ev0);
  if (p->ev1) cudaEventDestroy(p->ev1);
  if (p->ev2) cudaEventDestroy(p->ev2);
  if (p->own_stream && p->stream) cudaStreamDestroy(p->stream);
  delete p;
  return BBP_OK;
}

uint32_t bbp_working_bits(bbp_plan p, uint32_t P) {
  uint32_t W = 0;
  if (!p || !working_bits(P, p->guard, &W)) return 0;
  return W;
}

bbp_status bbp_series_extent(bbp_formula f, uint32_t denominator, uint64_t n, uint32_t W, uint64_t* he,
                             uint64_t* ne) {
  if (!valid_formula(f) || n == 0 || W == 0 || W % 32 != 0) return BBP_EINVAL;
  const FormulaDef& F = formula_def(f);
  if (denominator >= F.count) return BBP_EINVAL;
  if (he) *he = head_end(F, denominator, n - 1);
  if (ne) *ne = natural_end(F, denominator, n - 1, W);
  return BBP_OK;
}

bbp_status bbp_plan_stats(bbp_plan p, bbp_stats* out) {
  if (!p || !out) return BBP_EINVAL;
  *out = p->stats;
  return BBP_OK;
}

}  // extern "C"

namespace bbp {

namespace {

HeadArgs head_args(const FormulaDef& F, const TermRange& r, uint64_t n, uint32_t W) {
  const SeriesDef& s = F.s[r.j];
  HeadArgs a{};
  a.d = n - 1;
  a.k_begin = r.k_begin;
  a.count = r.count;
  a.a = s.a;
  a.b = s.b;
  a.c = s.c;
  a.step = F.step;
  a.W = W;
  a.L = W / 32;
  a.alternating = F.alternating;
  a.negate = ((s.sign < 0) != (F.alternating && (r.k_begin & 1ull))) ? 1u : 0u;
  a.window = r.window;
  a.first = r.first;
  a.first_max = r.first_max;
  return a;
}

TailArgs tail_args(const FormulaDef& F, const TermRange& r, uint64_t n, uint32_t W, unsigned long long* slots) {
  const SeriesDef& s = F.s[r.j];
  TailArgs a{};
  a.d = n - 1;
  a.k_begin = r.k_begin;
  a.count = r.count;
  a.a = s.a;
  a.b = s.b;
  a.c = s.c;
  a.step = F.step;
  a.W = W;
  a.L = W / 32;
  a.alternating = F.alternating;
  a.negate = s.sign < 0 ? 1u : 0u;
  a.slots = slots;
  return a;
}

// Consecutive terms per stream: the plan's, less while `count_tiles(run)` tiles are fewer than
// four for each resident warp (with one, a warp with two tiles doubles the time; n = 1e7,
// P = 256: 174 -> 148 us).
template <typename F>
uint32_t run_for(uint32_t run, uint64_t resident_warps, F count_tiles) {
  while (run % 4 == 0 && count_tiles(run) < 4 * resident_warps) run /= 2;
  return run;
}

}  // namespace

// Of 40 limbs no more head terms go into one launch: its kernel is 5 to 18 % slower a term than the
// ranges' own, which pays for eight launches up to n = 2e7 (P = 1000: 562 us in one, 579 in nine; 4e7:
// 1124 and 1057; 5e8: 14.6 and 12.3 ms).  Of fewer limbs one launch is the faster one throughout.
constexpr uint64_t kOneLaunchTerms40 = 20'000'000;

// run_for on path 2 up to 10 limbs, whose threads have two terms, four CTAs an SM, and start a
// run in a third of a term's time: the longest run that fills the resident warps, unless the
// shorter ones' waves, the last one whole, are less work (P = 256: 1e6 terms 97 us by this, 103 by
// shorter runs; 3e6 terms 268 and 233).  Of more limbs the shorter ones are the faster throughout.
template <typename F>
uint32_t run_for_path2(uint32_t run, uint64_t resident_warps, F count_tiles) {
  const uint32_t fine = run_for(run, resident_warps, count_tiles);
  while (run % 4 == 0 && count_tiles(run) < resident_warps) run /= 2;
  auto work = [&](uint32_t r) { return (count_tiles(r) + resident_warps - 1) / resident_warps * (3 * r + 1); };
  return 49 * work(run) <= 50 * work(fine) ? run : fine;
}

// Queues a whole query as one launch if all its head ranges are on modulus path 0 (n up
// to 2^29); *done says whether it did.
bbp_status launch_one(bbp_plan p, int f, uint64_t n, uint32_t W, uint32_t P, const std::vector<TermRange>& ranges,
                      uint64_t bound, uint8_t* out, uint32_t* valid, uint32_t* limbs, cudaStream_t st, bool* done) {
  *done = false;
  const FormulaDef& F = formula_def(f);
  const int lmax = pick_lmax(W, p->limb_bump);
  if (lmax == 0) return BBP_EINVAL;
  uint32_t heads = 0, tails = 0;
  uint64_t head_terms = 0;
  for (const TermRange& r : ranges) {
    if (!r.tail && r.path != 0) return BBP_OK;
    ++(r.tail ? tails : heads);
    head_terms += r.tail ? 0 : r.count;
  }
  if (lmax == 40 && head_terms > kOneLaunchTerms40) return BBP_OK;
  if (heads > static_cast<uint32_t>(kMaxQueryRanges) || tails > static_cast<uint32_t>(kMaxTailSet)) return BBP_OK;
  QuerySet q{};
  q.slots = p->d_query;
  q.finished = reinterpret_cast<unsigned int*>(p->d_query + kMaxLimbs);
  q.bound = bound;
  q.L = W / 32;
  q.P = P;
  q.out = out;
  q.valid = valid;
  q.limbs = limbs;
  const int streams = head_streams(p, 0);
  const int warps_per_block = p->cta / 32;
  const uint64_t cap = static_cast<uint64_t>(query_occupancy(streams, lmax, p->cta)) * p->sm_count;
  auto tiles_of = [&](uint64_t count, uint32_t run) { return (count + 32ull * streams * run - 1) / (32ull * streams * run); };
  auto count_tiles = [&](uint32_t run) {
    uint64_t total = 0;
    for (const TermRange& r : ranges) total += r.tail ? 0 : tiles_of(r.count, run);
    return total;
  };
  const uint32_t run = run_for(static_cast<uint32_t>(p->run), cap * warps_per_block, count_tiles);
  uint64_t tail_terms = 0;
  p->stats = bbp_stats{};
  for (const TermRange& r : ranges) {
    p->stats.terms += r.count;
    if (r.tail) {
      q.tails.a[q.tails.n++] = tail_args(F, r, n, W, q.slots);
      tail_terms += r.count;
    } else {
      HeadArgs& a = q.head[q.n];
      a = head_args(F, r, n, W);
      a.run = run;
      q.start[q.n + 1] = q.start[q.n] + tiles_of(r.count, run);
      ++q.n;
      p->stats.head_terms += r.count;
      p->stats.imad_model += r.imad;
    }
  }
  q.tail_blocks = static_cast<uint32_t>((tail_terms + p->cta - 1) / p->cta);
  const uint64_t want = (q.start[q.n] + warps_per_block - 1) / warps_per_block;
  const int blocks = static_cast<int>(std::max<uint64_t>(q.tail_blocks ? 0 : 1, std::min(want, cap)));
  BBP_CUDA(cudaMemsetAsync(p->d_query, 0, sizeof(unsigned long long) * (kMaxLimbs + 1), st));
  if (p->profile) BBP_CUDA(cudaEventRecord(p->ev0, st));
  BBP_CUDA(launch_query(q, streams, lmax, blocks, p->cta, st));
  p->stats.kernel_launches = 1;
  p->stats.head_launches = 1;
  if (p->profile) {
    BBP_CUDA(cudaEventRecord(p->ev1, st));
    BBP_CUDA(cudaEventSynchronize(p->ev1));
    float ms = 0;
    BBP_CUDA(cudaEventElapsedTime(&ms, p->ev0, p->ev1));
    p->stats.head_ms = ms;
  }
  *done = true;
  return BBP_OK;
}

// A range that crosses the line between two ladders is split where that pays: a second launch
// costs some 13 us (600,000 terms across 2^47: 70 us in one, 72 to 85 in two; across 1.02e12 58, 61
// to 73), and the cheaper ladder saves 9 to 17 % of its part.  From 2^21 terms on two are as fast
// or faster (3e6 terms across 2^47: 199 to 236 us, 255 before the ladders), with few terms below
// the line one (1000 of 4e6: 292, 306 in two).
constexpr uint64_t kSplitTerms = 1u << 21, kSplitBelow = 1u << 17;

// Launches every range of `ranges` (all of one query, same W) into `slots`.
bbp_status launch_ranges(bbp_plan p, int f, uint64_t n, uint32_t W, const std::vector<TermRange>& ranges,
                         unsigned long long* slots, cudaStream_t st, const uint32_t* gate) {
  const FormulaDef& F = formula_def(f);
  const int lmax = pick_lmax(W, p->limb_bump);
  if (lmax == 0) return BBP_EINVAL;
  float total_ms = 0;
  TailSet tails{};
  tails.gate = gate;
  for (const TermRange& r : ranges) {
    if (r.tail) {  // collected, and launched together once the set is full or the ranges end
      tails.a[tails.n++] = tail_args(F, r, n, W, slots);
      p->stats.terms += r.count;
      if (tails.n == kMaxTailSet) {
        BBP_CUDA(launch_tail_set(tails, st));
        p->stats.kernel_launches++;
        tails.n = 0;
      }
      continue;
    }
    // parts of paths 1 and 2 that have a ladder of their own
    TermRange parts[2] = {r, r};
    int paths[2] = {r.path, r.path};
    parts[1].count = 0;
    if ((r.path == 1 && p->wide_min_bits == kWideMinBits) || r.path == 2) {
      const SeriesDef& s = F.s[r.j];
      const uint64_t top = r.path == 1 ? kHalfMaxModulus : (1ull << (kSmallMaxBits + 1)) - 1;
      const uint64_t first_above = top < s.b ? 0 : (top - s.b) / s.a + 1;  // first k past `top`
      const uint64_t below = first_above > r.k_begin ? std::min(r.count, first_above - r.k_begin) : 0;
      const bool whole = below == r.count && (r.path == 1 || r.count >= k47Terms);
      if (whole || (below >= kSplitBelow && r.count >= kSplitTerms)) {
        parts[0].count = below;
        parts[1].k_begin = r.k_begin + below;
        parts[1].count = r.count - below;
        paths[0] = r.path == 1 ? kPathHalf : kPath47;
        uint8_t window;
        window_params(1, bitlen(static_cast<uint64_t>(s.a) * (r.k_begin + below - 1) + s.b), &window, &parts[0].first,
                      &parts[0].first_max);
        parts[0].window = 4;
      }
    }
    for (int i = 0; i < 2; ++i) {
      const TermRange& part = parts[i];
      if (part.count == 0) continue;
      HeadArgs a = head_args(F, part, n, W);
      a.slots = slots;
      a.gate = gate;
      const int streams = head_streams(p, paths[i]);
      const int path = roomy_path(paths[i], streams, lmax, part.count);
      const int warps_per_block = p->cta / 32;
      const int occ = head_occupancy(path, streams, lmax, p->cta);
      const uint64_t resident_warps = static_cast<uint64_t>(occ) * p->sm_count * warps_per_block;
      // a short range takes fewer consecutive terms per stream, so that its tiles
      // spread over the GPU's resident warps instead of a few warps running long runs
      auto tiles_for = [&](uint32_t rn) { return (part.count + 32ull * streams * rn - 1) / (32ull * streams * rn); };
      const uint32_t run = path == 2 && lmax <= 10 ? run_for_path2(static_cast<uint32_t>(p->run), resident_warps, tiles_for)
                                                   : run_for(static_cast<uint32_t>(p->run), resident_warps, tiles_for);
      a.run = run;
      const uint64_t ntiles = tiles_for(run);
      const uint64_t want = (ntiles + warps_per_block - 1) / warps_per_block;
      const int blocks = static_cast<int>(std::max<uint64_t>(1, std::min<uint64_t>(want, uint64_t(occ) * p->sm_count)));
      if (p->profile) BBP_CUDA(cudaEventRecord(p->ev0, st));
      BBP_CUDA(launch_head(a, path, streams, lmax, blocks, st, p->cta));
      if (p->profile) {
        BBP_CUDA(cudaEventRecord(p->ev1, st));
        BBP_CUDA(cudaEventSynchronize(p->ev1));
        float ms = 0;
        BBP_CUDA(cudaEventElapsedTime(&ms, p->ev0, p->ev1));
        total_ms += ms;
      }
      p->stats.kernel_launches++;
      p->stats.head_launches++;
      p->stats.terms += part.count;
      p->stats.head_terms += part.count;
    }
    p->stats.imad_model += r.imad;
  }
  if (tails.n > 0) {
    BBP_CUDA(launch_tail_set(tails, st));
    p->stats.kernel_launches++;
  }
  p->stats.head_ms += total_ms;
  return BBP_OK;
}

bbp_status plan_query(bbp_plan p, int f, uint64_t n, uint32_t W, int j_only, uint64_t k_lo, uint64_t k_hi,
                      std::vector<TermRange>& ranges, uint64_t* n_terms) {
  const FormulaDef& F = formula_def(f);
  const int lmax = pick_lmax(W, p->limb_bump);
  uint64_t N = 0;
  for (uint32_t j = 0; j < F.count; ++j) {
    if (j_only >= 0 && static_cast<int>(j) != j_only) continue;
    const int st = plan_series(F, j, n, W, static_cast<uint32_t>(lmax), k_lo, k_hi, ranges, p->wide_min_bits);
    if (st == -6) return BBP_ERANGE;
    if (st != 0) return BBP_EINVAL;
    N += natural_end(F, j, n - 1, W);
  }
  if (n_terms) *n_terms = N;
  return BBP_OK;
}

}  // namespace bbp

namespace {

// How a whole query is summed: term by term; by the prime form, whose check may ask for
// the terms (the caller reads the flag); or by the prime form with the term kernels
// queued behind it, which do nothing unless the check asks for them.
enum Form { kTerms, kPrimeOnly, kPrimeOrTerms };

// Queues a whole query.  kPrimeOnly: *redo says whether the terms are wanted, 0 unless
// the prime form runs.  Outputs may be in pinned host memory.
bbp_status enqueue_bits(bbp_plan p, int f, uint64_t n, uint32_t P, uint32_t W, uint8_t* d_out, uint32_t* d_valid,
                        uint32_t* d_limbs, cudaStream_t s, Form form, uint32_t* redo) {
  if (!redo) redo = p->d_redo;
  const FormulaDef& F = formula_def(f);
  std::vector<TermRange> ranges;
  uint64_t N = 0;
  const bbp_status st = plan_query(p, f, n, W, -1, 0, UINT64_MAX, ranges, &N);
  if (st != BBP_OK) return st;
  BBP_CUDA(cudaSetDevice(p->device));
  const int L = static_cast<int>(W / 32);
  const uint64_t bound = N + F.count + 1;  // |S - exact| < N + J + 1 units
  // The raw sum itself depends on every term's rounding: only the terms give it.
  const uint32_t* gate = nullptr;
  uint64_t prime_launches = 0;
  float prime_ms = 0;
  p->stats = bbp_stats{};
  if (form != kTerms && !d_limbs && prime_form_serves(f, n, P, W, bound) && prime_workspace(&p->primes, n, kPrimeListMax, s)) {
    const PrimeLimits lim = prime_limits(f, n - 1);
    std::vector<TermRange> rest;  // tails, and a head term past the limits
    for (uint32_t j = 0; j < F.count; ++j) {
      const bbp_status rs = plan_query(p, f, n, W, static_cast<int>(j), prime_first_k(lim, j, n - 1), UINT64_MAX, rest, nullptr);
      if (rs != BBP_OK) return rs;
    }
    if (p->profile) BBP_CUDA(cudaEventRecord(p->ev2, s));
    BBP_CUDA(launch_zero_slots(p->d_slots, L, s));
    const bbp_status ls = launch_ranges(p, f, n, W, rest, p->d_slots, s);
    if (ls != BBP_OK) return ls;
    PrimeRun run;
    if (run.plan(p->primes, p->sm_count, f, n, W, p->d_slots) == BBP_OK) {  // else all by terms
      bbp_status ps = run.begin(s);
      if (ps == BBP_OK) ps = run.run(0, run.lists(), s);
      if (ps == BBP_OK) ps = run.finish(P, bound, d_out, d_valid, redo, s);
      prime_launches = run.launches();
      if (ps != BBP_OK) return ps;
      if (p->profile) {
        BBP_CUDA(cudaEventRecord(p->ev1, s));
        BBP_CUDA(cudaEventSynchronize(p->ev1));
        BBP_CUDA(cudaEventElapsedTime(&prime_ms, p->ev2, p->ev1));
      }
      prime_launches += p->stats.kernel_launches + 1;
      gate = redo;
    }
  }
  if (!gate) {
    bool done = false;
    const bbp_status os = launch_one(p, f, n, W, P, ranges, bound, d_out, d_valid, d_limbs, s, &done);
    if (os != BBP_OK || done) return os;
  }
  if (gate && form == kPrimeOnly) {
    p->stats = bbp_stats{};
    for (const TermRange& r : ranges) {
      p->stats.terms += r.count;
      if (!r.tail) p->stats.head_terms += r.count;
    }
    p->stats.imad_model = prime_form_imad(prime_limits(f, n - 1), L);
    p->stats.head_launches = prime_launches;
    p->stats.kernel_launches = prime_launches;
    p->stats.head_ms = prime_ms;
    return BBP_OK;
  }
  p->stats = bbp_stats{};
  BBP_CUDA(launch_zero_slots(p->d_slots, L, s, gate));
  const bbp_status ls = launch_ranges(p, f, n, W, ranges, p->d_slots, s, gate);
  if (ls != BBP_OK) return ls;
  BBP_CUDA(launch_finalize_bits(p->d_slots, L, P, bound, d_out, d_valid, d_limbs, s, gate));
  p->stats.kernel_launches += 2 + prime_launches;
  p->stats.head_launches += prime_launches;
  p->stats.head_ms += prime_ms;
  if (gate) p->stats.imad_model = prime_form_imad(prime_limits(f, n - 1), L);
  return BBP_OK;
}

}  // namespace

extern "C" {

bbp_status bbp_partial_sum_async(bbp_plan p, bbp_formula f, uint32_t denominator, uint64_t k_begin,
                                 uint64_t k_end, uint64_t n, uint32_t P, uint32_t* d_out_limbs, void* stream) {
  if (!p || !valid_formula(f) || n == 0 || P == 0 || k_begin > k_end || !d_out_limbs) return BBP_EINVAL;
  if (denominator >= formula_def(f).count) return BBP_EINVAL;
  uint32_t W;
  if (!working_bits(P, p->guard, &W)) return BBP_EINVAL;
  std::vector<TermRange> ranges;
  const bbp_status st = plan_query(p, f, n, W, static_cast<int>(denominator), k_begin, k_end, ranges, nullptr);
  if (st != BBP_OK) return st;
  BBP_CUDA(cudaSetDevice(p->device));
  cudaStream_t s = stream ? static_cast<cudaStream_t>(stream) : p->stream;
  p->stats = bbp_stats{};
  BBP_CUDA(launch_zero_slots(p->d_slots, static_cast<int>(W / 32), s));
  const bbp_status ls = launch_ranges(p, f, n, W, ranges, p->d_slots, s);
  if (ls != BBP_OK) return ls;
  BBP_CUDA(launch_fold_limbs(p->d_slots, static_cast<int>(W / 32), d_out_limbs, s));
  p->stats.kernel_launches += 2;
  return BBP_OK;
}

bbp_status bbp_partial_sum(bbp_plan p, bbp_formula f, uint32_t denominator, uint64_t k_begin, uint64_t k_end,
                           uint64_t n, uint32_t P, uint32_t* out_limbs) {
  if (!p || !out_limbs) return BBP_EINVAL;
  bbp_status st = bbp_partial_sum_async(p, f, denominator, k_begin, k_end, n, P, p->d_limbs, p->stream);
  if (st != BBP_OK) return st;
  const uint32_t L = bbp_working_bits(p, P) / 32;
  BBP_CUDA(cudaMemcpyAsync(p->h_stage, p->d_limbs, sizeof(uint32_t) * L, cudaMemcpyDeviceToHost, p->stream));
  BBP_CUDA(cudaStreamSynchronize(p->stream));
  std::memcpy(out_limbs, p->h_stage, sizeof(uint32_t) * L);
  return BBP_OK;
}

bbp_status bbp_bits_async(bbp_plan p, bbp_formula f, uint64_t n, uint32_t P, uint8_t* d_out, uint32_t* d_valid,
                          uint32_t* d_limbs, void* stream) {
  if (!p || !valid_formula(f) || n == 0 || P == 0 || !d_out) return BBP_EINVAL;
  uint32_t W;
  if (!working_bits(P, p->guard, &W)) return BBP_EINVAL;
  return enqueue_bits(p, f, n, P, W, d_out, d_valid, d_limbs, stream ? static_cast<cudaStream_t>(stream) : p->stream,
                      kPrimeOrTerms, nullptr);
}

bbp_status bbp_shard_range(bbp_formula f, uint32_t denominator, uint64_t n, uint32_t W, uint32_t shard,
                           uint32_t nshards, uint64_t* k_begin, uint64_t* k_end) {
  if (!valid_formula(f) || n == 0 || W == 0 || W % 32 != 0 || nshards == 0 || shard >= nshards) return BBP_EINVAL;
  const FormulaDef& F = formula_def(f);
  if (denominator >= F.count) return BBP_EINVAL;
  uint64_t kb = 0, ke = 0;
  shard_range(F, denominator, n, W, shard, nshards, &kb, &ke);
  if (k_begin) *k_begin = kb;
  if (k_end) *k_end = ke;
  return BBP_OK;
}

bbp_status bbp_explain(bbp_formula f, uint64_t n, uint32_t P, uint32_t guard_bits, uint32_t wide_min_bits,
                       bbp_range* out, uint32_t cap, uint32_t* count, uint64_t* terms) {
  uint32_t W;
  if (!valid_formula(f) || n == 0 || !count || (cap > 0 && !out) || !working_bits(P, guard_bits, &W))
    return BBP_EINVAL;
  if (wide_min_bits < static_cast<uint32_t>(kWideFloorBits) || wide_min_bits > static_cast<uint32_t>(kWideMinBits))
    return BBP_EINVAL;
  const FormulaDef& F = formula_def(f);
  const int lmax = head_lmax_for(static_cast<int>(W / 32));
  if (lmax == 0) return BBP_EINVAL;
  std::vector<TermRange> ranges;
  for (uint32_t j = 0; j < F.count; ++j) {
    const int st = plan_series(F, j, n, W, static_cast<uint32_t>(lmax), 0, UINT64_MAX, ranges,
                               static_cast<int>(wide_min_bits));
    if (st == -6) return BBP_ERANGE;
    if (st != 0) return BBP_EINVAL;
  }
  uint64_t total = 0;
  for (size_t i = 0; i < ranges.size(); ++i) {
    const TermRange& r = ranges[i];
    total += r.count;
    if (i < cap) {
      bbp_range& o = out[i];
      o.denominator = r.j;
      o.tail = r.tail;
      o.path = r.path;
      o.window = r.window;
      o.first = r.first;
      o.first_max = r.first_max;
      o.k_begin = r.k_begin;
      o.count = r.count;
      o.imad = r.imad;
    }
  }
  *count = static_cast<uint32_t>(ranges.size());
  if (terms) *terms = total;
  return BBP_OK;
}

bbp_status bbp_accumulate_async(bbp_plan p, bbp_formula f, uint64_t n, uint32_t P, uint32_t shard, uint32_t nshards,
                                unsigned long long* d_slots, void* stream) {
  if (!p || !valid_formula(f) || n == 0 || P == 0 || !d_slots || nshards == 0 || shard >= nshards)
    return BBP_EINVAL;
  uint32_t W;
  if (!working_bits(P, p->guard, &W)) return BBP_EINVAL;
  const FormulaDef& F = formula_def(f);
  std::vector<TermRange> ranges;
  for (uint32_t j = 0; j < F.count; ++j) {
    uint64_t kb, ke;
    shard_range(F, j, n, W, shard, nshards, &kb, &ke);
    const bbp_status st = plan_query(p, f, n, W, static_cast<int>(j), kb, ke, ranges, nullptr);
    if (st != BBP_OK) return st;
  }
  BBP_CUDA(cudaSetDevice(p->device));
  cudaStream_t s = stream ? static_cast<cudaStream_t>(stream) : p->stream;
  p->stats = bbp_stats{};
  return launch_ranges(p, f, n, W, ranges, d_slots, s);
}

bbp_status bbp_finalize_async(bbp_plan p, bbp_formula f, uint64_t n, uint32_t P, const unsigned long long* d_slots,
                              uint8_t* d_out, uint32_t* d_valid, uint32_t* d_limbs, void* stream) {
  if (!p || !valid_formula(f) || n == 0 || P == 0 || !d_slots || !d_out) return BBP_EINVAL;
  uint32_t W;
  if (!working_bits(P, p->guard, &W)) return BBP_EINVAL;
  uint64_t N = 0;
  const FormulaDef& F = formula_def(f);
  for (uint32_t j = 0; j < F.count; ++j) N += natural_end(F, j, n - 1, W);
  BBP_CUDA(cudaSetDevice(p->device));
  cudaStream_t s = stream ? static_cast<cudaStream_t>(stream) : p->stream;
  BBP_CUDA(launch_finalize_bits(d_slots, static_cast<int>(W / 32), P, N + F.count + 1, d_out, d_valid, d_limbs, s));
  return BBP_OK;
}

bbp_status bbp_bits_formula(bbp_plan p, bbp_formula f, uint64_t n, uint32_t P, uint8_t* out, uint32_t* valid_bits) {
  if (!p || !out) return BBP_EINVAL;
  uint32_t W;
  if (!valid_formula(f) || n == 0 || P == 0 || !working_bits(P, p->guard, &W)) return BBP_EINVAL;
  // the kernels write their results to pinned host memory: no copies behind them
  uint8_t* h = static_cast<uint8_t*>(p->h_stage);
  uint32_t* h_valid = reinterpret_cast<uint32_t*>(h + 2048);
  uint32_t* h_redo = h_valid + 1;
  for (Form form = kPrimeOnly;; form = kTerms) {
    *h_redo = 0;
    const bbp_status st = enqueue_bits(p, f, n, P, W, h, h_valid, nullptr, p->stream, form, h_redo);
    if (st != BBP_OK) return st;
    BBP_CUDA(cudaStreamSynchronize(p->stream));
    if (*reinterpret_cast<volatile uint32_t*>(h_redo) == 0) break;
  }
  std::memcpy(out, h, (P + 7) / 8);
  const uint32_t valid = *reinterpret_cast<volatile uint32_t*>(h_valid);
  if (valid_bits) *valid_bits = valid;
  if (p->strict && valid < P) return BBP_EINVALID_BITS;
  return BBP_OK;
}

bbp_status bbp_bits(bbp_plan p, uint64_t n, uint32_t P, uint8_t* out, uint32_t* valid_bits) {
  return bbp_bits_formula(p, BBP_BELLARD, n, P, out, valid_bits);
}

bbp_status bbp_imad_probe(bbp_plan p, int kind, double* lanes_per_clk_per_sm) {
  if (!p || !lanes_per_clk_per_sm || kind < 0 || kind > 6) return BBP_EINVAL;
  BBP_CUDA(cudaSetDevice(p->device));
  const int blocks = p->sm_count;
  const int threads = 1024;
  const int iters = 4096;
  unsigned long long* d_cycles = nullptr;
  uint32_t* d_smid = nullptr;
  uint32_t* d_sink = nullptr;
  BBP_CUDA(cudaMalloc(&d_cycles, sizeof(unsigned long long) * blocks));
  BBP_CUDA(cudaMalloc(&d_smid, sizeof(uint32_t) * blocks));
  BBP_CUDA(cudaMalloc(&d_sink, sizeof(uint32_t)));
  cudaError_t e = launch_imad_probe(kind, blocks, threads, iters, d_cycles, d_smid, d_sink, p->stream);
  std::vector<unsigned long long> cycles(blocks);
  if (e == cudaSuccess) e = cudaMemcpyAsync(cycles.data(), d_cycles, sizeof(unsigned long long) * blocks,
                                            cudaMemcpyDeviceToHost, p->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(p->stream);
  cudaFree(d_cycles);
  cudaFree(d_smid);
  cudaFree(d_sink);
  if (e != cudaSuccess) return BBP_ECUDA;
  std::sort(cycles.begin(), cycles.end());
  const double med = static_cast<double>(cycles[cycles.size() / 2]);
  const double ops = static_cast<double>(threads) * iters * 64.0;
  *lanes_per_clk_per_sm = med > 0 ? ops / med : 0.0;
  return BBP_OK;
}

}  // extern "C"
