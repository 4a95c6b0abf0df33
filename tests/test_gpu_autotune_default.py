"""The tuner measures the library's own default schedule (budget 0: the default grouping) among
its candidates: where schedules tie it keeps that one, the time it reports as the default's is
that schedule's, and plans of a context it left at budget 0 group as an untuned context's do."""
import pytest

from paper_2512_18345_gb300 import inputs

pytestmark = pytest.mark.gpu


def context():
    import torch
    from paper_2512_18345_gb300 import binding
    P = inputs.workload_params("hrotate_N65536_L24_tc")
    ctx = binding.Context.from_params(P)
    ctx.set_bconv(binding.FHE_BCONV_TC)
    ctx.set_relin_key(torch.randint(0, 1 << 20, (P.dnum, 2, P.L + P.K, P.N), dtype=torch.int32, device="cuda"))
    return P, ctx


def plan_groups(P, ctx, n, level):
    import torch
    from paper_2512_18345_gb300 import binding
    d = torch.zeros(level, P.N, dtype=torch.int32, device="cuda")
    out = torch.empty(2, level, P.N, dtype=torch.int32, device="cuda")
    plan = ctx.batch_plan([dict(op=binding.FHE_OP_KS, level=level, rot=binding.FHE_RELIN_KEY, out=out, **{"in": d})] * n, 0)
    groups = plan.groups
    plan.close()
    return groups


def test_ties_keep_the_default_grouping(fhe_lib):
    P, ctx = context()
    r = ctx.autotune(4, 1)  # one item: every budget gives the same plan
    assert r["l2_budget_bytes"] == 0 and r["max_group"] == 0
    tuned = plan_groups(P, ctx, 48, 4)
    ctx.set_batch(0, 0, r["lanes"])
    assert tuned == plan_groups(P, ctx, 48, 4)
    ctx.close()


def test_the_default_is_a_candidate(fhe_lib, tmp_path):
    P, ctx = context()
    path = tmp_path / "tune.txt"
    r = ctx.autotune(4, 48, cache=str(path))  # groups of 12 by default, of at most 8 with a budget
    assert 0 < r["us_per_ks"] <= r["default_us_per_ks"]
    tuned = plan_groups(P, ctx, 48, 4)
    assert r["n_groups"] == len(tuned)
    _, fresh = context()
    if r["l2_budget_bytes"] == 0:
        assert max(tuned) > 8
        fresh.set_batch(0, 0, r["lanes"])
        assert tuned == plan_groups(P, fresh, 48, 4)
    # served from the file with the same choice
    again = fresh.autotune(4, 48, cache=str(path))
    assert again["candidates"] == 0 and again["l2_budget_bytes"] == r["l2_budget_bytes"]
    # an entry recorded under the candidates without the default is not taken over
    line = path.read_text().splitlines()[0]
    assert line.startswith("sched=2 ")
    path.write_text(line[len("sched=2 "):] + "\n")
    assert fresh.autotune(4, 48, cache=str(path))["candidates"] >= 2
    ctx.close()
    fresh.close()
