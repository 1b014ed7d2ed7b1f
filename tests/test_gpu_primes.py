"""Whole queries summed by primes (bbp_bits, bbp_bits_async without the raw sum) against the
term-by-term kernels (bbp_accumulate_async + bbp_finalize_async): the same bits and the same
certified count, tolerance 0, at positions where the prime form's limits, classes, lists and
words change, and where its check sends the query back to the terms."""

import time

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def bbp():
    import paper_1008_3171_gb300 as m

    return m


@pytest.fixture(scope="module")
def plans(bbp):
    ps = {G: bbp.Plan(device=0, guard_bits=G) for G in (32, 64)}
    yield ps
    for p in ps.values():
        p.close()


def by_terms(bbp, plan, n, P, formula=0):
    L = plan.working_bits(P) // 32
    slots = torch.zeros(L, dtype=torch.int64, device="cuda")
    out = torch.zeros((P + 7) // 8, dtype=torch.uint8, device="cuda")
    valid = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    bbp.bbp_accumulate_async(plan.handle, formula, n, P, 0, 1, slots.data_ptr())
    bbp.bbp_finalize_async(plan.handle, formula, n, P, slots.data_ptr(), out.data_ptr(), valid.data_ptr())
    torch.cuda.synchronize()
    return int.from_bytes(bytes(out.cpu().numpy()), "big") >> (8 * len(out) - P), int(valid[0])


def by_async(bbp, plan, n, P):
    out = torch.zeros((P + 7) // 8, dtype=torch.uint8, device="cuda")
    valid = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    bbp.bbp_bits_async(plan.handle, 0, n, P, out.data_ptr(), valid.data_ptr())
    torch.cuda.synchronize()
    return int.from_bytes(bytes(out.cpu().numpy()), "big") >> (8 * len(out) - P), int(valid[0])


# the smallest position that takes primes and its neighbours (n - 1 and n - 2 even and odd, A a
# multiple of 5 or not), 2^27, 2^29 and 2^31 (word and path changes above and below the moduli),
# A / 23 past 2^31 (sums in two words), several lists
@pytest.mark.parametrize("n,P", [(16 * 10**6 - 1, 64), (16 * 10**6, 64), (16 * 10**6 + 1, 100),
                                 (16 * 10**6 + 3, 256), (16 * 10**6 + 4, 448), (16 * 10**6 + 5, 1000), (10**8 + 6, 64), (2**27 + 1, 704), (2**29 - 1, 128), (2**29 + 3, 32),
                                 (2**31 - 1, 64), (2**31 + 2, 256), (23 * 2**29 + 7, 128), (23 * 2**31 + 11, 256)])
def test_equals_the_terms(bbp, plans, n, P):
    assert plans[64].bits(n, P) == by_terms(bbp, plans[64], n, P)


# the BBP formula: residues of n - 1 mod 4, moduli up to 2 n past 2^29 and 2^31, sums in two words
@pytest.mark.parametrize("n,P", [(16 * 10**6, 64), (16 * 10**6 + 1, 256), (16 * 10**6 + 2, 1000), (16 * 10**6 + 3, 32),
                                 (2**28 - 1, 100), (2**28 + 2, 448), (2**30 - 2, 64), (2**30 + 1, 704),
                                 (23 * 2**30 + 5, 128)])
def test_bbp_formula_equals_the_terms(bbp, plans, n, P):
    assert plans[64].bits(n, P, 1) == by_terms(bbp, plans[64], n, P, 1)


def test_check_sends_uncertain_positions_to_the_terms(bbp, plans):
    """G = 32 and P = 60: 36 bits below the output for a bound of 2^26.1 units, so about one
    position in 160 lies within three bounds of a carry.  Those and the others agree."""
    plan, P = plans[32], 60
    redone, checked = 0, {}
    for n in range(10**8 + 1, 10**8 + 801):
        got = plan.bits(n, P)
        terms_run = plan.stats()["imad_model"] > 4e9   # 7.5e9 for the terms, about 1e9 for the primes
        redone += terms_run
        if terms_run or n % 64 == 0:
            checked[n] = by_terms(bbp, plan, n, P)
            assert got == checked[n], n
            assert by_async(bbp, plan, n, P) == checked[n], n
    assert 0 < redone < 40   # 5 expected
    # in one batch, some of them through its second pass
    ns = list(checked)
    vals, valid, lat = bbp.bbp_bits_batch(plan.handle, 0, ns, [P] * len(ns))
    assert dict(zip(ns, zip(vals, valid))) == checked
    assert all(v > 0 for v in lat)
    # and through the serving engine, where they go back to its queue
    tickets = {n: bbp.bbp_submit(plan.handle, n, P) for n in ns}
    got, t_end = {}, time.time() + 60
    while len(got) < len(ns) and time.time() < t_end:
        for n in ns:
            if n not in got:
                r = bbp.bbp_poll(plan.handle, tickets[n], P)
                if r is not None:
                    got[n] = r
        time.sleep(0.001)
    assert got == checked


def test_batch_of_both_kinds(bbp, plans):
    """Queries of both kinds around the smallest position that takes primes, and the same batch
    again: each as alone, term by term."""
    plan = plans[64]
    ns = [10**4, 16 * 10**6 + 9, 12_345, 16 * 10**6 - 1, 10**8 + 21, 1, 3 * 10**7 + 2, 16 * 10**6, 10**6 + 1]
    Ps = [64, 128, 256, 64, 448, 8, 100, 256, 1000]
    want = [by_terms(bbp, plan, n, P) for n, P in zip(ns, Ps)]
    for _ in range(2):
        vals, valid, _ = bbp.bbp_bits_batch(plan.handle, 0, ns, Ps)
        assert list(zip(vals, valid)) == want
    vals, valid, _ = bbp.bbp_bits_batch(plan.handle, 1, ns, Ps)
    assert list(zip(vals, valid)) == [by_terms(bbp, plan, n, P, 1) for n, P in zip(ns, Ps)]


def test_async_on_a_stream_and_under_capture(bbp, plans):
    """Queued on a caller's stream, captured into a graph and replayed; a plan whose workspace is
    not there yet is captured term by term."""
    n, P = 10**8 + 77, 128
    want = by_terms(bbp, plans[64], n, P)
    for fresh in (True, False):
        plan = bbp.Plan(device=0, guard_bits=64)
        if not fresh:
            plan.bits(n, P)
        out = torch.zeros(P // 8, dtype=torch.uint8, device="cuda")
        valid = torch.zeros(1, dtype=torch.int32, device="cuda")
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            bbp.bbp_bits_async(plan.handle, 0, n, P, out.data_ptr(), valid.data_ptr(), 0, stream.cuda_stream)
        for _ in range(2):
            out.zero_()
            valid.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert (int.from_bytes(bytes(out.cpu().numpy()), "big"), int(valid[0])) == want
        del graph
        plan.close()
