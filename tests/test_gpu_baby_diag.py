"""The double-hoisted transform's baby rotations and diagonals in one kernel (at most four giant
steps) and in two (more), and its giant steps' key switches and sum in one, up to 16 of them: one to four digits, partial last digits, one to 32 baby steps, identity
and repeated baby steps, special limbs that meet no step, sparse and full index tables, maximal
residues (the folds of the accumulators).  Residue for residue against the C oracle on the small
ring, and on the large one against the two-kernel form, which the oracle checks elsewhere."""
import numpy as np
import pytest

from oracle import bootstrap_lt as blt
import oracle
from paper_2512_18345_gb300 import inputs

pytestmark = pytest.mark.gpu


def setup(logn, L, K, dnum, level, baby, giant, keep, fill):
    P = inputs.make_params(1 << logn, L, K, dnum, 31)
    g = inputs.rng(5200 + 100 * L + level + len(baby))

    def res(primes):
        if fill == "max":
            return np.stack([np.full(P.N, q - 1, np.uint32) for q in primes])
        return inputs.uniform_residues(g, primes, P.N)

    keys = {r: np.stack([np.stack([res(P.primes) for _ in range(2)]) for _ in range(P.dnum)])
            for r in sorted(set(baby) | set(giant)) if r % (P.N // 2)}
    ct = np.stack([inputs.uniform_residues(g, P.q[:level], P.N) for _ in range(2)])
    diags = np.stack([res(tuple(P.q[:level]) + tuple(P.p)) for _ in range(3)])
    idx = [[(i * 5 + b) % 3 if keep(i, b) else -1 for b in range(len(baby))] for i in range(len(giant))]
    return P, keys, ct, diags, idx


FULL = lambda i, b: True  # noqa: E731
CASES = [
    ((1, 1, 1, 1), (3,), (0,), FULL, "random"),
    ((4, 2, 2, 3), (0, 1, 0, 3, 1), (0, 5, -7), lambda i, b: (i + b) % 2 == 0, "random"),
    ((6, 2, 3, 6), tuple(range(8)), (0, 8, 16, -8), FULL, "max"),
    ((6, 2, 3, 5), (0, 2, 9), (0, 1, 5, 64), lambda i, b: b == 0, "random"),   # only the identity has diagonals
    ((6, 2, 3, 4), (2, 9, 0), (0, 1, 5, 64), lambda i, b: i == 2, "random"),   # giant steps without any
    ((12, 3, 4, 11), tuple(range(-15, 17)), (0, 100, 200, 300), FULL, "max"),  # 32 baby steps, 4 digits
    ((6, 2, 3, 6), (0, 1, 2, 3), (0, 4, 8, 12, 16), FULL, "max"),              # five giant steps: two kernels
    ((7, 2, 4, 7), (0, 1), tuple(range(-8, 8)), FULL, "max"),                  # 16 giant steps
    ((5, 3, 2, 4), (0, 1, 2), (7, 0, 0, 7), FULL, "random"),                   # repeated and identity giant steps
    ((3, 1, 3, 3), (0, 0), (4, 9), FULL, "max"),                               # no rotating baby step
]


@pytest.mark.parametrize("shape,baby,giant,keep,fill", CASES)
def test_small_ring_oracle(fhe_lib, shape, baby, giant, keep, fill):
    from paper_2512_18345_gb300 import binding
    level = shape[3]
    P, keys, ct, diags, idx = setup(12, *shape, baby, giant, keep, fill)
    ctx = binding.Context.from_params(P)
    for r, k in keys.items():
        ctx.set_rot_key(r, binding.to_device(k))
    want = blt.lt_double_hoisted(oracle.OracleParams.from_params(P), ct, level, baby, giant, diags, idx, keys)
    got = ctx.linear_transform_dh(binding.to_device(ct), level, baby, giant, binding.to_device(diags), idx)
    assert np.array_equal(binding.to_numpy(got), want)
    ctx.close()


@pytest.mark.parametrize("shape,baby,giant,keep,fill", [
    ((5, 2, 3, 5), (0, 1, 2, 7), (0, 9), FULL, "max"),
    ((8, 2, 4, 7), (0, 3, 5), (0, -9, 1000, 77), lambda i, b: (i * 3 + b) % 4 != 1, "random"),
    ((12, 12, 1, 12), (4,), (0, 1), FULL, "random"),
])
def test_large_ring_two_kernel_form(fhe_lib, shape, baby, giant, keep, fill):
    from paper_2512_18345_gb300 import binding
    level = shape[3]
    P, keys, ct, diags, idx = setup(16, *shape, baby, giant, keep, fill)
    outs = []
    for staged in (1, 0):
        ctx = binding.Context.from_params(P)
        ctx.set_kernel_shape(ip_staged_gather=staged)
        for r, k in keys.items():
            ctx.set_rot_key(r, binding.to_device(k))
        got = ctx.linear_transform_dh(binding.to_device(ct), level, baby, giant, binding.to_device(diags), idx)
        outs.append(binding.to_numpy(got).copy())
        ctx.close()
    assert np.array_equal(outs[0], outs[1])
