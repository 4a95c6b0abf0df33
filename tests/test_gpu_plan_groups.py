"""Default grouping of a plan's items: one group while the working set is small, equal groups on
every lane above that, the smaller groups where the context's memory limit is short of the
default's; an explicit cap is kept.  Every grouping gives the single calls' residues."""
import numpy as np
import pytest

from paper_2512_18345_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,lo,limit,batch,want", [
    (2, 24, 0, None, [2]), (8, 24, 0, None, [4, 4]), (8, 24, 0, (0, 3, 2), [3, 3, 2]),
    (33, 3, 0, None, None), (33, 3, 16, None, None),
])
def test_groups(fhe_lib, n, lo, limit, batch, want):
    import torch
    from paper_2512_18345_gb300 import binding
    P = inputs.workload_params("hrotate_N65536_L24_tc")
    ctx = binding.Context.from_params(P)
    ctx.set_bconv(binding.FHE_BCONV_TC)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)

    def residues(primes, *lead):
        q = torch.tensor(primes, dtype=torch.int64, device="cuda")[:, None]
        return (torch.randint(0, 1 << 62, (*lead, len(primes), P.N), generator=g, device="cuda") % q).to(torch.int32)

    ctx.set_rot_key(5, residues(P.primes, P.dnum, 2))
    ctx.set_relin_key(residues(P.primes, P.dnum, 2))
    if batch:
        ctx.set_batch(*batch)
    items = []
    for i in range(n):
        l = lo + (i * 7) % (P.L + 1 - lo)
        it = dict(op=binding.FHE_OP_ROTATE if i % 2 else binding.FHE_OP_RELIN, level=l, rot=5)
        it["in"], it["in2"] = residues(P.q[:l], 2), residues(P.q[:l], 2)
        it["out"] = torch.zeros_like(it["in"])
        items.append(it)
    if limit:  # room for the keys and `limit` workspace slots beyond the first
        i = ctx.info()
        ctx.set_memory_limit(2 * i["key_bytes"] + (limit + 1) * i["workspace_bytes"])
    plan = ctx.batch_plan(items)
    if want:
        assert plan.groups == want
    assert sum(plan.groups) == n
    if n == 33:  # two lanes of up to 8 items are what fits 16 further slots
        assert max(plan.groups) <= 8 if limit else max(plan.groups) > 8
    ctx.set_memory_limit(0)
    plan.launch()
    ctx.sync()
    for it in items:
        ref = ctx.rotate(it["in"], it["level"], 5) if it["op"] == binding.FHE_OP_ROTATE else ctx.hmult(it["in"], it["in2"], it["level"])
        assert torch.equal(ref, it["out"]), it["level"]
    plan.close()
    ctx.close()
