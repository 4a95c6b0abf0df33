"""Launch lists at the edges of a by-value list: a transform call of more limbs than one list
holds is split, every limb reaching its own segment (the limb -> segment map).  Oracle: the
C transform, residue for residue."""
import numpy as np
import pytest

import oracle
from paper_2512_18345_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,run", [(97, 1), (1985, 6), (2049, 5), (2200, 6)])
def test_transform_of_many_limbs(fhe_lib, n, run):
    """n limbs in runs of `run` consecutive primes (run 1: every limb its own segment)."""
    from paper_2512_18345_gb300 import binding
    P = inputs.workload_params("hmult_relin_rescale_N4096_L4")
    idx = [(i % run) if run > 1 else (2 * i) % 6 for i in range(n)]
    primes = [P.primes[i] for i in idx]
    a = inputs.uniform_residues(inputs.rng(41 + n), primes, P.N)
    ctx = binding.Context.from_params(P)
    t = binding.to_device(a)
    ctx.ntt(t, idx)
    assert np.array_equal(binding.to_numpy(t), oracle.ntt(a, primes))
    ctx.intt(t, idx)
    assert np.array_equal(binding.to_numpy(t), a)


def test_context_after_a_refused_call(fhe_lib):
    """A probe of a device that is not there fails alone: a context is created after it and
    computes, its first launches included."""
    from paper_2512_18345_gb300 import binding
    P = inputs.workload_params("hmult_relin_rescale_N4096_L4")
    with pytest.raises(binding.FheError):
        binding.probe_int(63)
    ctx = binding.Context.from_params(P)
    a = inputs.uniform_residues(inputs.rng(3), P.primes[:2], P.N)
    t = binding.to_device(a)
    ctx.ntt(t, [0, 1])
    assert np.array_equal(binding.to_numpy(t), oracle.ntt(a, P.primes[:2]))
    assert np.array_equal(binding.to_numpy(ctx.add(t, t, 2, npoly=1))[0], (2 * oracle.ntt(a, P.primes[:2]).astype(np.uint64) %
                                                                         np.array(P.primes[:2], np.uint64)[:, None]))
