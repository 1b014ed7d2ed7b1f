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
    for i, (below, above) in enumerate([(700, 0), (0, 700), (1, 1), (701, 4000), (4000, 701),
                                        (BELOW, TERMS - BELOW - 1), (BELOW - 1, TERMS - BELOW + 1),
                                        (BELOW, TERMS - BELOW), (TERMS - 1, 1), (TERMS, 0), (0, TERMS)]):
        P = (64, 256, 100)[i % 3]
        assert plan.partial_sum(formula, j, k - below, k + above, n, P) == \
            oracle.c_partial_sum(formula, j, k - below, k + above, n, P, 64), (below, above, P)
