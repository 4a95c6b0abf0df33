"""Contexts whose digit count exceeds four although ceil(L / alpha) does not (L = 7, dnum = 5:
alpha = 2, four digits and an empty fifth in the keys): every call with an inner product, on both
rings, in the fused and the plain pipeline, with every form of the inner product.  Oracle: the C
implementation, residue for residue."""
import numpy as np
import pytest

import oracle
from oracle import bootstrap_lt as blt
from paper_2512_18345_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logn,L,K,dnum,level,mode", [
    (16, 7, 2, 5, 7, "fused"), (16, 7, 2, 6, 5, "fused"), (16, 6, 2, 5, 6, "staged_off"), (16, 7, 2, 5, 6, "ip_moddown"),
    (16, 8, 2, 7, 7, "plain"), (12, 7, 2, 5, 7, "fused"), (12, 16, 4, 5, 15, "plain"), (12, 12, 3, 5, 12, "otf"),
])
def test_every_call(fhe_lib, logn, L, K, dnum, level, mode):
    from paper_2512_18345_gb300 import binding
    P = inputs.make_params(1 << logn, L, K, dnum, 31)
    assert P.beta(L) <= 4 < dnum
    OP = oracle.OracleParams.from_params(P)
    g = inputs.rng(900 + 10 * L + level)
    ctx = binding.Context.from_params(P)
    dev, host = binding.to_device, binding.to_numpy
    if mode == "plain":
        ctx.set_fused(False)
    elif mode == "otf":
        ctx.set_ntt(binding.FHE_NTT_OTF)
    elif mode == "ip_moddown":
        ctx.set_kernel_shape(fuse_ip_moddown=1)
    elif mode == "staged_off":
        ctx.set_kernel_shape(ip_staged_gather=0)

    def key():
        return np.stack([np.stack([inputs.uniform_residues(g, P.primes, P.N) for _ in range(2)]) for _ in range(P.dnum)])

    def poly(*lead):
        return np.stack([inputs.uniform_residues(g, P.q[:level], P.N) for _ in range(lead[0])])

    rk, keys = key(), {r: key() for r in (1, 2, 4)}
    ctx.set_relin_key(dev(rk))
    for r, k in keys.items():
        ctx.set_rot_key(r, dev(k))
    a, b = poly(2), poly(2)
    da, db = dev(a), dev(b)
    hm, rot = oracle.hmult(OP, a, b, level, rk), oracle.rotate(OP, a, level, 4, keys[4])
    assert np.array_equal(host(ctx.keyswitch(da[1].contiguous(), level)), oracle.keyswitch(OP, a[1], level, rk))
    assert np.array_equal(host(ctx.hmult(da, db, level)), hm)
    assert np.array_equal(host(ctx.rotate(da, level, 4)), rot)
    want = oracle.rotate_hoisted(OP, a, level, [1, 2], [keys[1], keys[2]])
    for x, y in zip(ctx.rotate_hoisted(da, level, [1, 2]), want):
        assert np.array_equal(host(x), y)
    plan = [dict(op=binding.FHE_OP_ROTATE, level=level, rot=4, out=binding.empty(a.shape), **{"in": da}),
            dict(op=binding.FHE_OP_RELIN, level=level, in2=db, out=binding.empty(a.shape), **{"in": da})]
    p = ctx.batch_plan(plan)
    p.launch()
    ctx.sync()
    assert np.array_equal(host(plan[0]["out"]), rot) and np.array_equal(host(plan[1]["out"]), hm)
    p.close()
    diags = poly(4)
    assert np.array_equal(host(ctx.linear_transform(da, level, dev(diags), 2, 2)),
                          oracle.bsgs_linear_transform(OP, a, level, diags, 2, 2, keys))
    xd = np.stack([inputs.uniform_residues(g, tuple(P.q[:level]) + tuple(P.p), P.N) for _ in range(2)])
    baby, giant, idx = (0, 1), (0, 4), ((0, 1), (1, 0))
    assert np.array_equal(host(ctx.linear_transform_dh(da, level, baby, giant, dev(xd), idx)),
                          blt.lt_double_hoisted(OP, a, level, baby, giant, xd, idx, keys))
    ctx.close()
