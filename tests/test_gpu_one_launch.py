"""Queries in one launch (every modulus below 2^29) against the oracle: positions around the
head/tail boundary, one and several tiles, ranges whose signs differ, widths of each limb
class, both formulas, settings of the plan, and results that go to device memory with the raw
sum or without the certified count.  Tolerance 0."""

import json

import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("table", [None, {"run": 2, "streams": 2, "cta": 32, "limb_bump": 2}, {"run": 128, "cta": 224}])
def test_positions_and_widths(table, tmp_path):
    import paper_1008_3171_gb300 as bbp

    path = None
    if table:
        path = tmp_path / "tune.json"
        path.write_text(json.dumps(table))
    for G in (32, 64):
        with bbp.Plan(device=0, guard_bits=G, tune_table=str(path) if path else None) as plan:
            for formula in (0, 1):
                for n, P in ((1, 8), (2, 64), (11, 96), (12, 1000), (65, 32), (4097, 448), (99_999, 250), (10**6 + 3, 64)):
                    assert plan.bits(n, P, formula) == oracle.c_bits(n, P, G, formula=formula), (n, P, G, formula)


def test_device_outputs():
    import paper_1008_3171_gb300 as bbp

    plan = bbp.Plan(device=0, guard_bits=64)
    n, P = 123_457, 200
    L = plan.working_bits(P) // 32
    for with_valid, with_limbs in ((True, True), (False, True), (True, False), (False, False)):
        out = torch.zeros(P // 8, dtype=torch.uint8, device="cuda")
        valid = torch.zeros(1, dtype=torch.int32, device="cuda")
        limbs = torch.zeros(L, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        bbp.bbp_bits_async(plan.handle, 0, n, P, out.data_ptr(), valid.data_ptr() if with_valid else 0,
                           limbs.data_ptr() if with_limbs else 0)
        torch.cuda.synchronize()
        want = oracle.c_bits(n, P, 64)
        assert int.from_bytes(bytes(out.cpu().numpy()), "big") == want[0]
        assert int(valid[0]) == (want[1] if with_valid else 0)
        if with_limbs:
            S = sum((int(v) & 0xFFFFFFFF) << (32 * i) for i, v in enumerate(limbs.cpu().tolist()))
            parts = sum(oracle.c_partial_sum(0, j, 0, None, n, P, 64) for j in range(7)) % (1 << (32 * L))
            assert S == parts
    plan.close()
