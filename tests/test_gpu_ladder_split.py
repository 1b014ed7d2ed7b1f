"""Ranges of terms that reach, leave or cross a line between two ladders (moduli of 1.02e12 and
2^47), whole below the sizes from which a crossing one is split and in two from there on,
against the oracle, tolerance 0."""

import pytest

import oracle
from oracle import bbp_oracle as o1

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")

TERMS, BELOW = 1 << 21, 1 << 17


@pytest.fixture(scope="module")
def plan():
    import paper_1008_3171_gb300 as bbp

    with bbp.Plan(device=0, guard_bits=64) as p:
        yield p


@pytest.mark.parametrize("line,n,formula,j", [(1_020_000_000_000, 3 * 10**12 + 1, 0, 0), (2**47, 10**15 + 4, 0, 3),
                                              (1_020_000_000_000, 2 * 10**13, 1, 2)])
def test_ranges_at_a_line(plan, line, n, formula, j):
    s = o1.FORMULAS[formula].series[j]
    k = (line - s.b) // s.a + 1            # first k past the line
    for i, (below, above) in enumerate([(700, 0), (0, 700), (1, 1), (701, 4000), (4000, 701), (76 * 1024 - 1, 0), (76 * 1024, 0),
                                        (BELOW, TERMS - BELOW - 1), (BELOW - 1, TERMS - BELOW + 1),
                                        (BELOW, TERMS - BELOW), (TERMS - 1, 1), (TERMS, 0), (0, TERMS)]):
        P = (64, 256, 100)[i % 3]
        assert plan.partial_sum(formula, j, k - below, k + above, n, P) == \
            oracle.c_partial_sum(formula, j, k - below, k + above, n, P, 64), (below, above, P)


@pytest.mark.parametrize("streams", [0, 1])
@pytest.mark.parametrize("P", [256, 170, 64])
def test_kernels_of_ten_limbs_by_length(P, streams, tmp_path):
    """Moduli of 42 and 47 bits, at the length from which ranges of 10 limbs take other kernels."""
    import paper_1008_3171_gb300 as bbp

    table = tmp_path / "tune.json"
    table.write_text('{"streams": %d}' % streams if streams else "{}")
    with bbp.Plan(device=0, guard_bits=64, tune_table=str(table)) as p:
        for m, n in ((3 * 10**12, 10**14 + 1), (10**14, 10**15)):
            for count in (2**19 - 1, 2**19):
                k = m // 10 + count
                assert p.partial_sum(0, 0, k, k + count, n, P) == oracle.c_partial_sum(0, 0, k, k + count, n, P, 64)
