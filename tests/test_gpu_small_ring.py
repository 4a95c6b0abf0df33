"""The small ring's whole-limb stages (one CTA per 4096-coefficient limb): digits and special
primes from one limb to sixteen (the folds of the conversion's accumulators fall after every
third input), partial last digits, maximal residues, rotations read through the automorphism in
single calls, hoisted sets, plans and the double-hoisted transform.  Oracle: the C
implementation, residue for residue."""
import numpy as np
import pytest

import oracle
from oracle import bootstrap_lt as blt
from paper_2512_18345_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,K,dnum,bits,level,fill", [
    (1, 1, 1, 31, 1, "random"), (4, 2, 2, 30, 3, "max"), (5, 3, 2, 31, 4, "random"), (7, 4, 1, 31, 7, "max"),
    (16, 16, 1, 31, 16, "max"), (16, 13, 1, 31, 13, "random"), (24, 6, 4, 31, 19, "max"), (30, 10, 3, 30, 30, "random"),
])
def test_every_call(fhe_lib, L, K, dnum, bits, level, fill):
    from paper_2512_18345_gb300 import binding
    P = inputs.make_params(1 << 12, L, K, dnum, bits)
    OP = oracle.OracleParams.from_params(P)
    g = inputs.rng(100 + L * K)
    ctx = binding.Context.from_params(P)
    dev, host = binding.to_device, binding.to_numpy

    def res(primes):
        if fill == "max":
            return np.stack([np.full(P.N, q - 1, np.uint32) for q in primes])
        return inputs.uniform_residues(g, primes, P.N)

    def key():
        return np.stack([np.stack([res(P.primes) for _ in range(2)]) for _ in range(P.dnum)])

    def ct():
        x = np.stack([res(P.q[:level]) for _ in range(2)])
        x[:, :, ::3] = np.stack([inputs.uniform_residues(g, P.q[:level], P.N) for _ in range(2)])[:, :, ::3]
        return x

    rk, keys = key(), {r: key() for r in (1, 3, 1024, -7)}
    ctx.set_relin_key(dev(rk))
    for r, k in keys.items():
        ctx.set_rot_key(r, dev(k))
    a, b = ct(), ct()
    da, db = dev(a), dev(b)
    hm = oracle.hmult(OP, a, b, level, rk)
    assert np.array_equal(host(ctx.keyswitch(da[1].contiguous(), level)), oracle.keyswitch(OP, a[1], level, rk))
    got = ctx.hmult(da, db, level)
    assert np.array_equal(host(got), hm)
    if level > 1:
        assert np.array_equal(host(ctx.rescale(got, level)), oracle.rescale(OP, hm, level))
    rots = {r: oracle.rotate(OP, a, level, r, k) for r, k in keys.items()}
    for r, want in rots.items():
        assert np.array_equal(host(ctx.rotate(da, level, r)), want), r
    hoisted = oracle.rotate_hoisted(OP, a, level, list(keys), [keys[r] for r in keys])
    for r, x, y in zip(keys, ctx.rotate_hoisted(da, level, list(keys)), hoisted):
        assert np.array_equal(host(x), y), r
    plan = [dict(op=binding.FHE_OP_ROTATE, level=level, rot=r, out=binding.empty(a.shape), **{"in": da}) for r in keys]
    plan.append(dict(op=binding.FHE_OP_RELIN, level=level, in2=db, out=binding.empty(a.shape), **{"in": da}))
    p = ctx.batch_plan(plan)
    p.launch()
    ctx.sync()
    for it, want in zip(plan, list(rots.values()) + [hm]):
        assert np.array_equal(host(it["out"]), want)
    p.close()
    baby, giant, idx = (0, 1, 3), (0, 1024), ((0, 1, -1), (2, -1, 0))
    diags = np.stack([res(tuple(P.q[:level]) + tuple(P.p)) for _ in range(3)])
    want = blt.lt_double_hoisted(OP, a, level, baby, giant, diags, idx, keys)
    assert np.array_equal(host(ctx.linear_transform_dh(da, level, baby, giant, dev(diags), idx)), want)
    ctx.close()
