"""What a default plan may hold: groups stay within a bound whatever the mix of levels, a context
with a memory limit keeps the smaller groups (room that later calls need), and a share that comes
out empty falls back to them.  Every grouping gives the single calls' residues."""
import pytest

from paper_2512_18345_gb300 import inputs

pytestmark = pytest.mark.gpu


def context():
    import torch
    from paper_2512_18345_gb300 import binding
    P = inputs.workload_params("hrotate_N65536_L24_tc")
    ctx = binding.Context.from_params(P)
    ctx.set_bconv(binding.FHE_BCONV_TC)
    g = torch.Generator(device="cuda")
    g.manual_seed(11)

    def residues(primes, *lead):
        q = torch.tensor(primes, dtype=torch.int64, device="cuda")[:, None]
        return (torch.randint(0, 1 << 62, (*lead, len(primes), P.N), generator=g, device="cuda") % q).to(torch.int32)

    ctx.set_rot_key(5, residues(P.primes, P.dnum, 2))
    return P, ctx, residues


def rotations(P, residues, levels):
    import torch
    from paper_2512_18345_gb300 import binding
    items = []
    for l in levels:
        it = dict(op=binding.FHE_OP_ROTATE, level=l, rot=5)
        it["in"] = residues(P.q[:l], 2)
        it["out"] = torch.zeros_like(it["in"])
        items.append(it)
    return items


def check(ctx, plan, items):
    import torch
    plan.launch()
    ctx.sync()
    for it in items:
        assert torch.equal(ctx.rotate(it["in"], it["level"], 5), it["out"]), it["level"]
    plan.close()


@pytest.mark.parametrize("lanes,most", [(0, 24), (1, 24), (3, 16), (4, 12)])
def test_groups_are_bounded_for_uneven_levels(fhe_lib, lanes, most):
    P, ctx, residues = context()
    ctx.set_batch(0, 0, lanes)
    items = rotations(P, residues, [24] * 10 + [1] * 54)
    plan = ctx.batch_plan(items)
    assert sum(plan.groups) == 64 and 8 < max(plan.groups) <= most, plan.groups
    check(ctx, plan, items)
    ctx.close()


def test_empty_share_falls_back(fhe_lib):
    P, ctx, residues = context()
    ctx.set_batch(0, 0, 4)
    items = rotations(P, residues, [24, 24, 24, 1, 1])
    plan = ctx.batch_plan(items)
    assert sum(plan.groups) == 5 and min(plan.groups) > 0
    check(ctx, plan, items)
    ctx.close()


def test_a_limit_leaves_room_for_later_calls(fhe_lib):
    """A limit that holds what a plan of 33 items takes without one, and less than a transform's
    scratch beside it: the limited plan takes less, and the transform finds room."""
    import torch
    P, ctx, residues = context()
    info, level, baby, giant = ctx.info(), 6, 1, 2
    items = rotations(P, residues, [3 + (k * 7) % 22 for k in range(33)])
    rk = residues(P.primes, P.dnum, 2)
    ct, diags = residues(P.q[:level], 2), residues(P.q[:level], baby * giant)
    plan = ctx.batch_plan(items)
    slots = 2 * max(plan.groups)
    assert slots > 16
    check(ctx, plan, items)
    ctx.set_rot_key(1, rk)
    want = ctx.linear_transform(ct, level, diags, baby, giant)
    ctx.close()
    P, ctx, _ = context()
    ctx.set_rot_key(1, rk)
    ctx.set_memory_limit(2 * info["key_bytes"] + slots * info["workspace_bytes"] + 2 * level * P.N * 4)
    plan = ctx.batch_plan(items)
    assert max(plan.groups) <= 8
    assert torch.equal(ctx.linear_transform(ct, level, diags, baby, giant), want)
    ctx.set_memory_limit(0)
    check(ctx, plan, items)
    ctx.close()
