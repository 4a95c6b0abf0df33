"""The block pass whose half-warps each own a 256-element block: the rotation's input blocks
are staged in memory order and permuted on the way out, so every residue class of the Galois
element has to land right -- odd and even steps, block-preserving ones, negative ones, at both
ring degrees, in a plan that mixes a rotation with items read unpermuted, and the combine and
rescale endings.  Oracle: the C key switch, residue for residue."""
import numpy as np
import pytest

import oracle
from paper_2512_18345_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,level,rots", [
    ("hmult_relin_rescale_N4096_L4", 3, (1, 2, 7, 16, 255, 1024, 2047, -5)),
    ("hrotate_N65536_L24_tc", 2, (1, 4096, 32767, -129)),
])
def test_rotations_and_mixed_plan(fhe_lib, name, level, rots):
    from paper_2512_18345_gb300 import binding
    P = inputs.workload_params(name)
    OP = oracle.OracleParams.from_params(P)
    g = inputs.rng(77)
    ctx = binding.Context.from_params(P)

    def key():
        return np.stack([np.stack([inputs.uniform_residues(g, P.primes, P.N) for _ in range(2)]) for _ in range(P.dnum)])

    def ct():
        return np.stack([inputs.uniform_residues(g, P.q[:level], P.N) for _ in range(2)])

    rk = key()
    ctx.set_relin_key(binding.to_device(rk))
    a, b = ct(), ct()
    a[:, 0, :] = P.q[0] - 1
    da, db = binding.to_device(a), binding.to_device(b)
    plan, want = [], []
    for r in rots:
        k = key()
        ctx.set_rot_key(r, binding.to_device(k))
        w = oracle.rotate(OP, a, level, r, k)
        assert np.array_equal(binding.to_numpy(ctx.rotate(da, level, r)), w), r
        plan.append(dict(op=binding.FHE_OP_ROTATE, level=level, rot=r, out=binding.empty((2, level, P.N)), **{"in": da}))
        want.append(w)
    plan.append(dict(op=binding.FHE_OP_RELIN, level=level, in2=db, out=binding.empty((2, level, P.N)), **{"in": da}))
    want.append(oracle.hmult(OP, a, b, level, rk))
    p = ctx.batch_plan(plan)
    p.launch()
    ctx.sync()
    for it, w in zip(plan, want):
        assert np.array_equal(binding.to_numpy(it["out"]), w), it["rot"] if it["op"] else "relin"
    m = binding.to_numpy(ctx.rescale(binding.to_device(want[-1]), level))
    assert np.array_equal(m, oracle.rescale(OP, want[-1], level))
