"""Single calls launch their stage kernels as dependents of one another; the same calls under
tracing, in a caller's captured graph and in a plan do not.  Every form must give the same
residues: queued back to back on changing inputs (so that a stale read would show), on two
contexts and streams at once, at the levels where launches are smallest and largest."""
import numpy as np
import pytest

from paper_2512_18345_gb300 import inputs

pytestmark = pytest.mark.gpu

SMALL, BIG, WIDE = "hmult_relin_rescale_N4096_L4", "hrotate_N65536_L24_tc", "paper_ks_N65536_L48_a12"


def setup(name, seed, tc):
    import torch
    from paper_2512_18345_gb300 import binding
    P = inputs.workload_params(name)
    ctx = binding.Context.from_params(P)
    ctx.set_bconv(binding.FHE_BCONV_TC if tc else binding.FHE_BCONV_SCALAR)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def residues(primes, *lead):
        q = torch.tensor(primes, dtype=torch.int64, device="cuda")[:, None]
        return (torch.randint(0, 1 << 62, (*lead, len(primes), P.N), generator=g, device="cuda") % q).to(torch.int32)

    ctx.set_relin_key(residues(P.primes, P.dnum, 2))
    for r in (1, 2, 5):
        ctx.set_rot_key(r, residues(P.primes, P.dnum, 2))
    return P, ctx, residues


def calls(ctx, level, a, b):
    out = [ctx.rotate(a, level, 5), ctx.keyswitch(a[0].contiguous(), level), ctx.hmult(a, b, level)]
    out += ctx.rotate_hoisted(a, level, [1, 0, 2])
    out += [ctx.modup(a[1].contiguous(), level)]
    out += [ctx.moddown(out[-1][0].contiguous(), level), ctx.bconv(a[0, :1].contiguous(), [0], list(range(1, ctx.L + ctx.K)))]
    return out + ([ctx.rescale(out[2], level)] if level > 1 else [])


@pytest.mark.parametrize("name,level,tc", [(SMALL, 1, False), (SMALL, 4, False), (SMALL, 3, True), (BIG, 1, True),
                                           (BIG, 9, False), (BIG, 24, True), (WIDE, 48, True)])
def test_back_to_back_calls(fhe_lib, name, level, tc):
    import torch
    P, ctx, residues = setup(name, 5, tc)
    sets = [(residues(P.q[:level], 2), residues(P.q[:level], 2)) for _ in range(3)]
    ctx.trace(True)  # no dependent launches
    want = [[x.clone() for x in calls(ctx, level, *s)] for s in sets]
    ctx.sync()
    ctx.trace(False)
    for rep in range(4):
        got = [calls(ctx, level, *sets[i % 3]) for i in range(6)]
        ctx.sync()
        for i, g in enumerate(got):
            for k, (x, y) in enumerate(zip(g, want[i % 3])):
                assert torch.equal(x, y), (rep, i, k)
    # a product written over its own factor (the factors are read before the last kernel writes)
    for k in (0, 1):
        ab = [x.clone() for x in sets[1]]
        assert torch.equal(ctx.hmult(ab[0], ab[1], level, out=ab[k]), want[1][2])
    sq = sets[2][0].clone()
    assert torch.equal(ctx.hmult(sq, sq, level, out=sq), ctx.hmult(sets[2][0], sets[2][0], level))
    # a caller's own capture of the same calls, replayed on other inputs
    a, b = (x.clone() for x in sets[0])
    torch.cuda.synchronize()
    graph, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(st):  # the context's last calls are on the capturing stream
        ctx.rotate(a, level, 5)
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=st):
        out = [ctx.rotate(a, level, 5), ctx.hmult(a, b, level)]
    for i in (1, 2):
        a.copy_(sets[i][0])
        b.copy_(sets[i][1])
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out[0], want[i][0]) and torch.equal(out[1], want[i][2])


def test_two_contexts_on_two_streams(fhe_lib):
    import torch
    pairs = [setup(SMALL, 1, False), setup(BIG, 2, True)]
    work = []
    for P, ctx, residues in pairs:
        level = P.L
        s = (residues(P.q[:level], 2), residues(P.q[:level], 2))
        ctx.trace(True)
        want = [x.clone() for x in calls(ctx, level, *s)]
        ctx.sync()
        ctx.trace(False)
        work.append((ctx, level, s, want, torch.cuda.Stream()))
    torch.cuda.synchronize()
    got = []
    for rep in range(6):
        for i, (ctx, level, s, want, st) in enumerate(work):
            with torch.cuda.stream(st):
                got.append((i, calls(ctx, level, *s)))
    torch.cuda.synchronize()
    for i, g in got:
        assert all(torch.equal(x, y) for x, y in zip(g, work[i][3])), i
