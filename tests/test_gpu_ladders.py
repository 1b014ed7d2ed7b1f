"""Partial sums where the head kernels change ladders inside a modulus path -- moduli up to
and past 1.02e12, moduli of 46, 47 and 48 bits -- and where exponents are smallest and
largest for them, against the oracle, tolerance 0: one and two term pairs a thread, several
widths, both formulas, and the entry point without a plan."""

import json

import pytest

import oracle
from oracle import bbp_oracle as o1

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

HALF = 1_020_000_000_000


def first_k(value, s):
    return max(0, (value - s.b) // s.a)


def cases():
    for formula, j in ((0, 0), (0, 5), (0, 8 % 7), (1, 0), (1, 1)):
        f = o1.FORMULAS[formula]
        s = f.series[j]
        for n, value in ((3 * 10**12, HALF), (3 * 10**13, HALF), (10**14 + 1, 2**46), (10**15 + 3, 2**47),
                         (2**43 - 1, HALF)):
            k = first_k(value, s)
            if k + 700 < o1.head_end(f, s, n - 1):
                yield formula, j, n, k - 700, k + 700
        # the smallest exponents that 40- and 47-bit moduli meet, and the head's last terms
        for n in (3 * 10**11 + 7, 9 * 10**13 + 2):
            he = o1.head_end(f, s, n - 1)
            yield formula, j, n, he - 1300, he + 2
        # exponents around the powers of 4 and 2 where the number of pairs changes
        for e in (64 * 4**18 // 3, 64 * 4**17 // 3, 2**39):
            n = 9 * 10**11 + 5
            k = (n - 1 - e) // f.step
            if 0 < k and s.a * k + s.b < HALF:
                yield formula, j, n, k - 300, k + 300


@pytest.mark.parametrize("streams", [1, 2])
def test_ladder_changes(streams, tmp_path):
    import paper_1008_3171_gb300 as bbp

    table = tmp_path / "tune.json"
    table.write_text(json.dumps({"streams": streams}))
    with bbp.Plan(device=0, guard_bits=64, tune_table=str(table)) as plan:
        for i, (formula, j, n, kb, ke) in enumerate(cases()):
            P = (64, 256, 1000, 128)[i % 4]
            assert plan.partial_sum(formula, j, kb, ke, n, P) == oracle.c_partial_sum(formula, j, kb, ke, n, P, 64), \
                (formula, j, n, kb, ke, P)


def test_ladder_changes_without_a_plan():
    import paper_1008_3171_gb300 as bbp

    for formula, j, n, kb, ke in list(cases())[::3]:
        P = 200
        out = torch.zeros(9, dtype=torch.int32, device="cuda")
        bbp.bbp_partial_sum_noalloc(formula, j, kb, ke, n, P, 64, out.data_ptr())
        torch.cuda.synchronize()
        got = sum((int(v) & 0xFFFFFFFF) << (32 * i) for i, v in enumerate(out.cpu().tolist()))
        assert got == oracle.c_partial_sum(formula, j, kb, ke, n, P, 64), (formula, j, n, kb, ke)
