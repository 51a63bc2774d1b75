"""Entropies of vectors whose Schmidt blocks span more of FP64's exponents than
their squares can: a configuration beside amplitudes whose squared products
underflow (S = 0), and vectors of very small and very large norm, against the oracle."""
import numpy as np
import pytest

import oracle as O
from gpu_common import device_basis, lib, torch_dev

pytestmark = pytest.mark.gpu


def _entropies(V, L):
    torch, dev = torch_dev()
    pf = lib()
    dim, st = device_basis(pf, torch, dev, L)
    with pf.Ctx(0) as ctx:
        return pf.entanglement_entropy(ctx, L, st, torch.from_numpy(V).to(dev), dim, len(V), per_cut=True)


@pytest.mark.parametrize("L", [8, 14, 18])
def test_a_configuration_beside_tiny_amplitudes(L):
    states = O.basis(L)
    rng = np.random.default_rng(L)
    scales = [1e-38, 1e-74, 1e-77, 1e-78, 1e-79, 1e-80, 1e-81, 1e-120, 1e-155, 1e-162, 1e-310]
    V = np.zeros((2 * len(scales), len(states)))
    for i, a in enumerate(scales):
        V[2 * i] = a * rng.standard_normal(len(states))
        V[2 * i, len(states) // 3] = 1.0
        V[2 * i + 1, [1, len(states) // 2, len(states) - 2]] = a  # three of them
        V[2 * i + 1, 0] = 1.0
    got = _entropies(V, L)
    for v in range(len(V)):
        for x in (0, 1, L // 2 - 1):
            # the configuration alone has S = 0 and the rest changes it by less than 1e-37 (numpy's SVD of
            # the oracle is not finite for some of these); eigenvalues to 2^-53 of the trace, 2^(L/2) of them,
            # |ln| <= 42
            assert abs(got[v, x]) < 1e-11, (v, x, got[v, x])


@pytest.mark.parametrize("power", [-300, -130, 130, 255, 300])
def test_vectors_of_any_norm(power):
    L = 10
    states = O.basis(L)
    v = np.random.default_rng(3).standard_normal(len(states))
    v /= np.linalg.norm(v)
    got = _entropies(np.ldexp(v, power)[None, :], L)[0]
    for x in range(L // 2):
        # S of c psi = c^2 (S of psi - 2 ln c), c a power of two
        want = O.entanglement_entropy_cut(v, states, L, x) - 2 * power * np.log(2.0)
        assert abs(np.ldexp(got[x], -2 * power) - want) < 1e-11 * max(1.0, abs(want)), (x, got[x], want)
