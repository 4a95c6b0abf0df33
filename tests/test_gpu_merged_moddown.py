"""The dense transform's giant rotations with their ModDowns merged into one transform: one and
two rotations, as many as a program holds and more (a further program adds to the output), both
base conversions, full and partial last digits, maximal residues, and the on-the-fly NTT mode,
which keeps the separate ModDowns.  Oracle: the composition of separate rotations, residue for
residue."""
import numpy as np
import pytest

import oracle
from paper_2512_18345_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,K,dnum,level,baby,giant,tc,fill", [
    (6, 2, 3, 6, 2, 2, True, "random"), (6, 2, 3, 5, 2, 3, False, "max"), (6, 2, 3, 3, 1, 16, True, "max"),
    (8, 2, 4, 7, 2, 16, False, "random"), (3, 3, 1, 3, 3, 12, True, "random"), (12, 12, 1, 11, 2, 4, True, "max"),
])
def test_transform(fhe_lib, L, K, dnum, level, baby, giant, tc, fill):
    from paper_2512_18345_gb300 import binding
    P = inputs.make_params(1 << 16, L, K, dnum, 31)
    OP = oracle.OracleParams.from_params(P)
    g = inputs.rng(7 * L + giant)

    def res(primes):
        if fill == "max":
            return np.stack([np.full(P.N, q - 1, np.uint32) for q in primes])
        return inputs.uniform_residues(g, primes, P.N)

    ctx = binding.Context.from_params(P)
    ctx.set_bconv(binding.FHE_BCONV_TC if tc else binding.FHE_BCONV_SCALAR)
    keys = {r: np.stack([np.stack([res(P.primes) for _ in range(2)]) for _ in range(P.dnum)])
            for r in sorted(set(range(1, baby)) | {baby * x for x in range(1, giant)})}
    for r, k in keys.items():
        ctx.set_rot_key(r, binding.to_device(k))
    ct = np.stack([inputs.uniform_residues(g, P.q[:level], P.N) for _ in range(2)])
    diags = np.stack([res(P.q[:level]) for _ in range(baby * giant)])
    want = oracle.bsgs_linear_transform(OP, ct, level, diags, baby, giant, keys)
    args = (binding.to_device(ct), level, binding.to_device(diags), baby, giant)
    for mode in (0, binding.FHE_NTT_OTF):
        ctx.set_ntt(mode)
        for _ in range(2):
            got = ctx.linear_transform(*args)
        ctx.sync()
        assert np.array_equal(binding.to_numpy(got), want), mode
    ctx.close()
