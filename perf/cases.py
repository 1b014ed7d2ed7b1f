"""Performance cases of the library: the calls a user makes, over the range of sizes they make them at.

A case is a dict of plain values.  ``prepare(case, seed)`` builds what a program holds before the
call (a plan with its stream, device buffers, the list of queries), ``run(state)`` is one pass
through the public entry points.  The position of a query is drawn from the seed just below the
case's ``n`` (within 0.1 %), so another seed is another position with the same amount of work;
ranges of terms start at a point drawn from the seed too.

Kinds of case:

* ``bits``     one blocking query through ``Plan`` handles: bits n .. n+P-1 of pi and the certified
               count, as host bytes.  The everyday call.
* ``device``   the same query with its outputs in the caller's device memory on the caller's
               stream (``bbp_bits_async``), with or without the raw W-bit sum.
* ``slice``    ``bbp_partial_sum``: one series over a range of terms, the unit by which a query is
               spread over machines or verified by pieces.
* ``shard``    ``bbp_accumulate_async`` of one shard of a long query and ``bbp_finalize_async``:
               what a checkpointed long run does for each of its shards, and at its end.
* ``noalloc``  ``bbp_partial_sum_noalloc``: the plan-less entry point on the caller's stream.
* ``batch``    ``bbp_bits_batch`` over a list of queries whose positions are log-uniform.
* ``serve``    the serving engine: every query of a list submitted, then polled until it is done.
"""

import math
import random
import time

import numpy as np
import torch

import paper_1008_3171_gb300 as bbp

# (a, b, sign, c) of each series: sign (-1)^(alternating k) 2^(n - 1 + c - step k) / (a k + b)
FORMULAS = {
    0: (10, True, [(10, 1, 1, 2), (10, 3, -1, 0), (10, 5, -1, -4), (10, 7, -1, -4), (10, 9, 1, -6),
                   (4, 1, -1, -1), (4, 3, -1, -6)]),
    1: (4, False, [(8, 1, 1, 2), (2, 1, -1, -1), (8, 5, -1, 0), (4, 3, -1, -1)]),
}


def listed():
    return [
        # smallest ordinary query: the position where a cluster of CPUs is not needed; launches count
        dict(name="bits_1e6_p64", kind="bits", n=10**6, P=64, guard=32, formula=0),
        # a device-side caller that wants the raw sum too, at a position of a few milliseconds' work
        dict(name="device_1e7_p256_limbs", kind="device", n=10**7, P=256, guard=64, formula=0, limbs=True),
        # one-limb moduli throughout: the printed table rows' first position, 128 bits
        dict(name="bits_1e9_p128", kind="bits", n=10**9, P=128, guard=64, formula=0),
        # the original BBP formula, run as the independent check of a result
        dict(name="bits_eq1_1e9_p64", kind="bits", n=10**9, P=64, guard=64, formula=1),
        # long outputs, 1000 bits at an odd width (34 limbs)
        dict(name="bits_3e8_p1000", kind="bits", n=3 * 10**8, P=1000, guard=64, formula=0),
        # the headline query's shape (256 bits, mostly two-limb moduli) at the largest size a pass allows
        dict(name="bits_4e10_p256", kind="bits", n=4 * 10**10, P=256, guard=64, formula=0),
        # pieces of the long queries: 40-bit moduli, and 47-bit moduli past the three-word square
        dict(name="slice_1e12_p256", kind="slice", n=10**12, P=256, guard=64, formula=0, j=0,
             k_frac=0.5, count=2 * 10**8),
        dict(name="slice_1e14_p256", kind="slice", n=10**14, P=256, guard=64, formula=0, j=3,
             k_frac=0.85, count=2 * 10**8),
        # one shard of a checkpointed 1e13 run
        dict(name="shard_1e13_p256", kind="shard", n=10**13, P=256, guard=64, formula=0, nshards=4096),
        # a short piece without a plan, for callers that may not allocate
        dict(name="noalloc_3e7_p128", kind="noalloc", n=3 * 10**7, P=128, guard=64, formula=0, j=5,
             k_frac=0.3, count=150_001),
        # many queries of very different sizes at once
        dict(name="batch_256_1e4_1e9", kind="batch", count=256, lo=4.0, hi=9.0, guard=64, formula=0),
        # queries arriving together at the serving engine
        dict(name="serve_48_1e6_1e9", kind="serve", count=48, lo=6.0, hi=9.0, guard=64, formula=0),
    ]


def _log(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    kind = rng.choice(["bits", "bits", "bits", "device", "slice", "slice", "shard", "noalloc", "batch", "serve"])
    guard = 64
    if kind == "bits":
        n, P = _log(rng, 10**5, 4 * 10**10), rng.choice([32, 64, 64, 128, 200, 256, 256, 448, 1000])
        if n > 2 * 10**10:
            P = min(P, 256)
        if n < 10**7:
            guard = rng.choice([32, 64])
        # the original formula has 1.43 times the terms: keep it below the largest listed query
        formula = rng.choice([0, 0, 0, 1]) if n < 2 * 10**10 else 0
        return dict(kind=kind, n=n | rng.randrange(2), P=P, guard=guard, formula=formula)
    if kind == "device":
        return dict(kind=kind, n=_log(rng, 10**5, 2 * 10**9), P=rng.choice([64, 100, 256]), guard=guard,
                    formula=0, limbs=rng.random() < 0.5)
    if kind in ("slice", "noalloc"):
        big = kind == "slice"
        formula = rng.choice([0, 0, 1])
        return dict(kind=kind, n=_log(rng, 10**7, 10**15 if big else 10**10), P=rng.choice([64, 128, 256]),
                    guard=guard, formula=formula, j=rng.randrange(len(FORMULAS[formula][2])),
                    k_frac=rng.uniform(0.01, 0.95), count=_log(rng, 10**3, 10**9 if big else 10**7))
    if kind == "shard":
        n = _log(rng, 10**9, 10**14)
        return dict(kind=kind, n=n, P=rng.choice([64, 256]), guard=guard, formula=0,
                    nshards=max(16, n // _log(rng, 10**8, 3 * 10**9)))
    return dict(kind=kind, count=_log(rng, 3, 256 if kind == "batch" else 48), lo=4.0 if kind == "batch" else 6.0,
                hi=rng.uniform(7.0, 9.0), guard=guard, formula=0)


# ---------------------------------------------------------------- inputs

def _position(case, rng):
    n = case["n"]
    return n - rng.randrange(max(1, n // 1000))


def _queries(case, rng):
    """Positions log-uniform in 10^lo .. 10^hi, one in each equal part of it, so that every seed has
    about the same work; in random order, the three ordinary precisions in turn."""
    lo, hi, count = case["lo"], case["hi"], case["count"]
    parts = list(range(count))
    rng.shuffle(parts)
    ns = [int(10.0 ** (lo + (hi - lo) * (i + 0.45 + 0.1 * rng.random()) / count)) for i in parts]
    return ns, [(64, 128, 256)[q % 3] for q in range(count)]


def _range_of_terms(case, n, rng):
    step, _, series = FORMULAS[case["formula"]]
    head = (n - 1 + series[case["j"]][3]) // step + 1
    count = min(case["count"], head // 2)
    k0 = min(int(head * case["k_frac"]), head - count)
    k0 -= rng.randrange(k0 // 1000 + 1)
    return k0, k0 + count


class State:
    """What the user's program holds; the plan goes with it."""

    def __init__(self, case, seed):
        self.case = case
        self.kind = case["kind"]
        rng = random.Random(seed * 1_000_003 + 17)
        self.device = torch.device("cuda", 0)
        self.stream = torch.cuda.current_stream(self.device).cuda_stream
        self.plan = None
        if self.kind != "noalloc":
            self.plan = bbp.Plan(device=0, guard_bits=case["guard"])
        if self.kind in ("batch", "serve"):
            self.ns, self.Ps = _queries(case, rng)
            return
        self.n = _position(case, rng)
        P = case["P"]
        L = ((P + 31) // 32 * 32 + case["guard"]) // 32
        if self.kind in ("slice", "noalloc"):
            self.k0, self.k1 = _range_of_terms(case, self.n, rng)
        if self.kind == "shard":
            self.shard = rng.randrange(case["nshards"])
        if self.kind in ("device", "shard", "noalloc"):
            self.out = torch.zeros((P + 7) // 8, dtype=torch.uint8, device=self.device)
            self.valid = torch.zeros(1, dtype=torch.int32, device=self.device)
            self.limbs = torch.zeros(L, dtype=torch.int32, device=self.device)
            self.slots = torch.zeros(L, dtype=torch.int64, device=self.device)


def prepare(case, seed):
    return State(case, seed)


# ---------------------------------------------------------------- one pass

def run(state):
    c = state.case
    if state.kind == "bits":
        raw, valid = bbp.bbp_bits_formula(state.plan.handle, c["formula"], state.n, c["P"])
        return [np.frombuffer(raw, dtype=np.uint8), valid]
    if state.kind == "device":
        bbp.bbp_bits_async(state.plan.handle, c["formula"], state.n, c["P"], state.out.data_ptr(),
                           state.valid.data_ptr(), state.limbs.data_ptr() if c["limbs"] else 0, state.stream)
        return [state.out, state.valid] + ([state.limbs] if c["limbs"] else [])
    if state.kind == "slice":
        return np.array(bbp.bbp_partial_sum(state.plan.handle, c["formula"], c["j"], state.k0, state.k1, state.n,
                                            c["P"]), dtype=np.int64)
    if state.kind == "shard":
        state.slots.zero_()
        bbp.bbp_accumulate_async(state.plan.handle, c["formula"], state.n, c["P"], state.shard, c["nshards"],
                                 state.slots.data_ptr(), state.stream)
        bbp.bbp_finalize_async(state.plan.handle, c["formula"], state.n, c["P"], state.slots.data_ptr(),
                               state.out.data_ptr(), state.valid.data_ptr(), state.limbs.data_ptr(), state.stream)
        return [state.out, state.valid, state.limbs]
    if state.kind == "noalloc":
        bbp.bbp_partial_sum_noalloc(c["formula"], c["j"], state.k0, state.k1, state.n, c["P"], c["guard"],
                                    state.limbs.data_ptr(), state.stream)
        return state.limbs
    if state.kind == "batch":
        values, valid, _ = bbp.bbp_bits_batch(state.plan.handle, c["formula"], state.ns, state.Ps)
        return [_value_bytes(values, state.Ps), np.array(valid, dtype=np.int64)]
    tickets = [bbp.bbp_submit(state.plan.handle, n, P) for n, P in zip(state.ns, state.Ps)]
    done = [None] * len(tickets)
    left = list(range(len(tickets)))
    while left:
        still = []
        for q in left:
            done[q] = bbp.bbp_poll(state.plan.handle, tickets[q], state.Ps[q])
            if done[q] is None:
                still.append(q)
        left = still
        if left:
            time.sleep(0.0005)
    return [_value_bytes([v for v, _ in done], state.Ps), np.array([k for _, k in done], dtype=np.int64)]


def _value_bytes(values, Ps):
    return np.frombuffer(b"".join(v.to_bytes((P + 7) // 8, "big") for v, P in zip(values, Ps)), dtype=np.uint8)


# ---------------------------------------------------------------- what a pass amounts to

def _terms_and_limbs(case):
    def whole(n, formula):
        step, _, series = FORMULAS[formula]
        return len(series) * n / step

    W = (case.get("P", 150) + 31) // 32 * 32 + case["guard"]
    if case["kind"] in ("batch", "serve"):
        lo, hi = case["lo"], case["hi"]
        mean = (10.0**hi - 10.0**lo) / ((hi - lo) * math.log(10.0))
        return case["count"] * whole(mean, case["formula"]), W / 32
    if case["kind"] in ("slice", "noalloc"):
        step = FORMULAS[case["formula"]][0]
        return min(case["count"], case["n"] // step // 2), W / 32
    terms = whole(case["n"], case["formula"])
    return (terms / case["nshards"] if case["kind"] == "shard" else terms), W / 32


def work(case):
    """A sum of `terms` fractions of W bits: one multiplication and one addition per term and limb.
    Nothing is read but the query; the result is a few limbs."""
    terms, limbs = _terms_and_limbs(case)
    queries = case.get("count", 1) if case["kind"] in ("batch", "serve") else 1
    return {"bytes": queries * (16 + 4 * limbs), "flops": 2.0 * terms * limbs}


# ---------------------------------------------------------------- exact values of the small cases

def _partial(formula, j, k0, k1, n, W):
    """sign_j sum over k0 <= k < k1 of (-1)^k floor(2^(W + e) / m) mod 2^W, as the definition reads."""
    step, alternating, series = FORMULAS[formula]
    a, b, sign, c = series[j]
    total = 0
    for k in range(k0, k1):
        m, e = a * k + b, n - 1 + c - step * k
        if e >= 0:
            t = (pow(2, e, m) << W) // m
        else:
            t = ((1 << (W + e)) // m) if W + e >= 0 else 0
            if t == 0:
                break
        total += -t if alternating and k & 1 else t
    return sign * total % (1 << W)


def exact(case, seed):
    rng = random.Random(seed * 1_000_003 + 17)
    if case["kind"] in ("batch", "serve"):
        return None
    n, P = _position(case, rng), case["P"]
    W = (P + 31) // 32 * 32 + case["guard"]
    L = W // 32
    if case["kind"] in ("slice", "noalloc"):
        if case["count"] > 10**6:
            return None
        k0, k1 = _range_of_terms(case, n, rng)
        S = _partial(case["formula"], case["j"], k0, k1, n, W)
        limbs = np.array([(S >> (32 * i)) & 0xFFFFFFFF for i in range(L)], dtype=np.int64)
        return limbs.astype(np.uint32).view(np.int32) if case["kind"] == "noalloc" else limbs
    if case["kind"] == "shard" or n > 2 * 10**6:
        return None
    S, terms = 0, 0
    step, _, series = FORMULAS[case["formula"]]
    for j, (a, b, sign, c) in enumerate(series):
        end = (n - 1 + c) // step + 1 + W // step + 2
        S += _partial(case["formula"], j, 0, end, n, W)
        p = lambda k: W + n - 1 + c - step * k
        while end > 0 and (p(end - 1) < 0 or (1 << min(p(end - 1), 4096)) < a * (end - 1) + b):
            end -= 1
        terms += end
    S %= 1 << W
    # certified bits: the sum is within `bound` units of the value, so the top b bits stand when the
    # rest is at least that far from both ends
    bound, valid = terms + len(series) + 1, 0
    for b in range(P, -1, -1):
        low = S & ((1 << (W - b)) - 1)
        if bound <= low <= (1 << (W - b)) - bound:
            valid = b
            break
    nbytes = (P + 7) // 8
    raw = np.frombuffer(((S >> (W - P)) << (8 * nbytes - P)).to_bytes(nbytes, "big"), dtype=np.uint8)
    if case["kind"] == "bits":
        return [raw, valid]
    limbs = np.array([(S >> (32 * i)) & 0xFFFFFFFF for i in range(L)], dtype=np.int64).astype(np.uint32).view(np.int32)
    return [raw, np.array([valid], dtype=np.int32)] + ([limbs] if case["limbs"] else [])
