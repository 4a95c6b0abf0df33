"""The linear transforms reserve what the form that runs stores: a memory limit that holds
exactly that is enough, one byte less is refused, and the residues are those of the forms that
store the baby rotations and the key switches too (which need, and get, the larger scratch)."""
import pytest

from paper_2512_18345_gb300 import inputs

pytestmark = pytest.mark.gpu


def setup(logn, L, K, dnum, rots):
    import torch
    from paper_2512_18345_gb300 import binding
    P = inputs.make_params(1 << logn, L, K, dnum, 31)
    ctx = binding.Context.from_params(P)
    g = torch.Generator(device="cuda")
    g.manual_seed(L)

    def residues(primes, *lead):
        q = torch.tensor(primes, dtype=torch.int64, device="cuda")[:, None]
        return (torch.randint(0, 1 << 62, (*lead, len(primes), P.N), generator=g, device="cuda") % q).to(torch.int32)

    for r in rots:
        ctx.set_rot_key(r, residues(P.primes, P.dnum, 2))
    i = ctx.info()
    return P, ctx, residues, len(rots) * i["key_bytes"], i["workspace_bytes"]


def exactly(ctx, nbytes, call):
    from paper_2512_18345_gb300 import binding
    ctx.set_memory_limit(nbytes - 1)
    with pytest.raises(binding.FheError) as e:
        call()
    assert e.value.code == binding.FHE_ENOMEM
    ctx.set_memory_limit(nbytes)
    out = call().clone()
    ctx.sync()
    return out


# bab: the extended ciphertexts stored for the rotating baby steps; every rotating giant step's key
# switch is stored with the staged gather off only
@pytest.mark.parametrize("logn", [12, 16])
@pytest.mark.parametrize("baby,giant,bab", [
    ((0, 1, 3), (0, 7, 9), 0),          # one kernel for the baby steps, one for the giant steps
    ((0, 1, 3), (0, 1, 7, 9, 11), 2),  # more than four giant steps: the baby rotations are stored
    ((1, 3), (0,), 0),               # no rotating giant step: nothing is key-switched
    ((0,), (0, 7), 0),               # no rotating baby step
])
def test_double_hoisted(fhe_lib, logn, baby, giant, bab):
    import torch
    level = 3
    rots = sorted({r for r in (*baby, *giant) if r})
    P, ctx, residues, keys, slot = setup(logn, 4, 2, 2, rots)
    xct = 2 * (level + P.K) * P.N * 4
    ng = sum(1 for r in giant if r)
    ct, diags = residues(P.q[:level], 2), residues(tuple(P.q[:level]) + tuple(P.p), 2)
    idx = [[(g + b) % 2 for b in range(len(baby))] for g in range(len(giant))]
    call = lambda: ctx.linear_transform_dh(ct, level, baby, giant, diags, idx)  # noqa: E731
    slots = max(2, 1 + ng)  # the shared ModUp's, one per rotating giant step, the last ModDown's
    nbytes = keys + slots * slot + (bab + len(giant) + 1) * xct + ng * level * P.N * 4
    got = exactly(ctx, nbytes, call)
    ctx.set_memory_limit(0)
    ctx.set_kernel_shape(ip_staged_gather=0)
    assert torch.equal(call(), got)
    ctx.set_kernel_shape(ip_staged_gather=1)
    assert torch.equal(call(), got)
    ctx.close()


@pytest.mark.parametrize("logn,baby,giant,grot", [(16, 2, 4, False), (16, 3, 1, False), (12, 2, 3, True)])
def test_dense(fhe_lib, logn, baby, giant, grot):
    import torch
    from paper_2512_18345_gb300 import binding
    level = 3
    rots = sorted(set(range(1, baby)) | {baby * g for g in range(1, giant)})
    P, ctx, residues, keys, slot = setup(logn, 4, 2, 2, rots)
    one = 2 * level * P.N * 4
    ct, diags = residues(P.q[:level], 2), residues(P.q[:level], baby * giant)
    call = lambda: ctx.linear_transform(ct, level, diags, baby, giant)  # noqa: E731
    slots = max(baby, giant - 1)  # the shared ModUp's and one per baby rotation; one per giant rotation
    nbytes = keys + slots * slot + (baby + giant + (giant - 1 if grot else 0)) * one
    got = exactly(ctx, nbytes, call)
    ctx.set_memory_limit(0)
    ctx.set_ntt(binding.FHE_NTT_OTF)  # separate ModDowns: the giant rotations are stored
    assert torch.equal(call(), got)
    ctx.set_ntt(0)
    assert torch.equal(call(), got)
    ctx.close()
