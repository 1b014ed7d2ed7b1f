"""Calls by primes beside other uses of a plan and of the device, each against the
term-by-term kernels or the printed rows, tolerance 0."""

import pytest

from test_gpu_primes import bbp, by_terms, plans  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def value(out, P):
    return int.from_bytes(bytes(out.cpu().numpy()), "big") >> (8 * len(out) - P)


def test_graph_replayed_after_a_longer_query(bbp, plans):  # noqa: F811
    """Captured at 1e8, then a query of 6e8 whose lists do not fit the captured ones, replayed."""
    n, P = 10**8 + 79, 128
    plan = bbp.Plan(device=0, guard_bits=64)
    plan.bits(n, P)
    out = torch.zeros(P // 8, dtype=torch.uint8, device="cuda")
    valid = torch.zeros(1, dtype=torch.int32, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        bbp.bbp_bits_async(plan.handle, 0, n, P, out.data_ptr(), valid.data_ptr(), 0, stream.cuda_stream)
    want = by_terms(bbp, plans[64], n, P)
    longer = by_terms(bbp, plans[64], 6 * 10**8 + 1, P)
    free = torch.cuda.mem_get_info()[0]
    assert plan.bits(6 * 10**8 + 1, P) == longer
    # the longer lists came on top of the captured ones: two of 24 M primes
    assert free - torch.cuda.mem_get_info()[0] >= 2 * 4 * (24 << 20)
    out.zero_()
    valid.zero_()
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    assert (value(out, P), int(valid[0])) == want
    assert plan.bits(6 * 10**8 + 1, P) == longer
    del graph
    plan.close()


def test_beside_a_capture_of_another_stream(bbp, plans):  # noqa: F811
    """A plan's first query by primes, and one whose lists grow, on one stream while another is
    captured in the default mode: both are right."""
    plan = bbp.Plan(device=0, guard_bits=64)
    queries = [(10**8 + 81, 128), (4 * 10**8 + 3, 64)]
    outs = [torch.zeros(P // 8, dtype=torch.uint8, device="cuda") for _, P in queries]
    valid = torch.zeros(2, dtype=torch.int32, device="cuda")
    x = torch.zeros(1024, device="cuda")
    side, stream = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="global"):
        x.add_(1)
        for i, (n, P) in enumerate(queries):
            bbp.bbp_bits_async(plan.handle, 0, n, P, outs[i].data_ptr(), valid.data_ptr() + 4 * i, 0, side.cuda_stream)
    graph.replay()
    torch.cuda.synchronize()
    assert float(x.sum()) == 1024
    for i, (n, P) in enumerate(queries):
        assert (value(outs[i], P), int(valid[i])) == by_terms(bbp, plans[64], n, P)
    del graph
    plan.close()


def test_primes_past_the_half_reduced_ladder(bbp, plans, pins):  # noqa: F811
    """Primes past 1.02e12 take the plain two-word ladder: the printed row at 1e13 + 1 by Eq. 2
    (half a minute), and Eq. 1, whose moduli reach 2 n, against Eq. 2 at 6e11."""
    row = pins["table2_m13"]
    want = int(row["hex"], 16) >> (len(row["hex"]) * 4 - 256)
    assert plans[64].bits(10**13 + 1, 256) == (want, 256)
    n = 6 * 10**11 + 7
    assert plans[64].bits(n, 128, 1) == plans[64].bits(n, 128)
