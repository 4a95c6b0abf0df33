"""Both linear transforms queued back to back on changing inputs: their dependent launches share
one scratch buffer and the workspace slots, so a read of the call before would show.  The same
calls under tracing, where every launch is an ordinary one, give what is expected.  Up to four
giant steps and more, with the inner products inside the kernels that use them and outside, on
both rings, and on two contexts and streams at once."""
import pytest

from paper_2512_18345_gb300 import inputs

pytestmark = pytest.mark.gpu

BABY, FEW, MANY = (0, 1, 3), (0, 7, 9), (0, 7, 9, 11, 12)


def setup(logn, staged, seed):
    import torch
    from paper_2512_18345_gb300 import binding
    P = inputs.make_params(1 << logn, 4, 2, 2, 31)
    ctx = binding.Context.from_params(P)
    ctx.set_kernel_shape(ip_staged_gather=staged)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def residues(primes, *lead):
        q = torch.tensor(primes, dtype=torch.int64, device="cuda")[:, None]
        return (torch.randint(0, 1 << 62, (*lead, len(primes), P.N), generator=g, device="cuda") % q).to(torch.int32)

    for r in {r for r in (*BABY, *MANY, 2, 4, 6) if r}:
        ctx.set_rot_key(r, residues(P.primes, P.dnum, 2))
    level = 3
    sets = [(residues(P.q[:level], 2), residues(P.q[:level], 8), residues(tuple(P.q[:level]) + tuple(P.p), 3))
            for _ in range(3)]
    return ctx, level, sets


def calls(ctx, level, ct, dense, diags):
    idx = [[(g + b) % 4 - 1 for b in range(len(BABY))] for g in range(len(MANY))]
    return [ctx.linear_transform_dh(ct, level, BABY, FEW, diags, idx[: len(FEW)]),
            ctx.linear_transform(ct, level, dense, 2, 4),
            ctx.linear_transform_dh(ct, level, BABY, MANY, diags, idx),
            ctx.linear_transform(ct, level, dense, 2, 1)]


def traced(ctx, level, sets):
    ctx.trace(True)  # no dependent launches
    want = [[x.clone() for x in calls(ctx, level, *s)] for s in sets]
    ctx.sync()
    ctx.trace(False)
    return want


@pytest.mark.parametrize("logn,staged", [(12, 1), (12, 0), (16, 1), (16, 0)])
def test_back_to_back(fhe_lib, logn, staged):
    import torch
    ctx, level, sets = setup(logn, staged, 3)
    want = traced(ctx, level, sets)
    for rep in range(3):
        got = [calls(ctx, level, *sets[i % 3]) for i in range(6)]
        ctx.sync()
        for i, g in enumerate(got):
            for k, (x, y) in enumerate(zip(g, want[i % 3])):
                assert torch.equal(x, y), (rep, i, k)
    ctx.close()


def test_two_contexts_on_two_streams(fhe_lib):
    import torch
    work = []
    for logn, seed in ((12, 4), (16, 5)):
        ctx, level, sets = setup(logn, 1, seed)
        work.append((ctx, level, sets, traced(ctx, level, sets), torch.cuda.Stream()))
    torch.cuda.synchronize()
    got = []
    for rep in range(6):
        for ctx, level, sets, want, st in work:
            with torch.cuda.stream(st):
                got.append((calls(ctx, level, *sets[rep % 3]), want[rep % 3]))
    torch.cuda.synchronize()
    for g, w in got:
        assert all(torch.equal(x, y) for x, y in zip(g, w))
