"""Entropies through the library's own small-block eigenvalue kernels, at the edges
of their range: the smallest blocks (L = 4), the largest (L = 18, 126 rows), and
spectra with zeros and exact degeneracies (product, two-configuration and singlet
states), against the oracle's Schmidt decomposition."""
import numpy as np
import pytest

import oracle as O
from gpu_common import device_basis, lib, torch_dev

pytestmark = pytest.mark.gpu


def _vectors(kind, L, dim, states):
    rng = np.random.default_rng(L)
    if kind == "random":
        v = rng.standard_normal((2, dim))
    elif kind == "graded":  # weights over 16 decades: most Schmidt values are tiny
        v = rng.standard_normal((2, dim)) * 10.0 ** rng.uniform(-8, 0, (2, dim))
    elif kind == "product":
        v = np.zeros((2, dim))
        v[0, 0] = 1.0
        v[1, dim // 2] = -1.0
    else:  # two configurations of equal weight: S = ln 2 or 0 at every cut
        v = np.zeros((2, dim))
        v[0, [0, dim - 1]] = 1.0
        v[1, [1, dim // 3]] = 1.0
    return v / np.linalg.norm(v, axis=1, keepdims=True)


@pytest.mark.parametrize("L", [4, 6, 10, 16, 18])
@pytest.mark.parametrize("kind", ["random", "graded", "product", "pair"])
def test_entropy_small_blocks_vs_oracle(L, kind):
    torch, dev = torch_dev()
    pf = lib()
    dim, st = device_basis(pf, torch, dev, L)
    states = O.basis(L)
    V = _vectors(kind, L, dim, states)
    with pf.Ctx(0) as ctx:
        got = pf.entanglement_entropy(ctx, L, st, torch.from_numpy(V).to(dev), dim, 2, per_cut=True)
    cuts = range(L) if L <= 10 else (0, 1, L // 2 - 1)
    for v in range(2):
        for x in cuts:
            want = O.entanglement_entropy_cut(V[v], states, L, x)
            # eigenvalues to 2^-53 of the trace, 2^(L/2) of them, |ln| <= 42
            assert abs(got[v, x] - want) < 1e-11, (v, x, got[v, x], want)


def test_entropy_of_a_vector_that_is_not_finite_is_refused():
    torch, dev = torch_dev()
    pf = lib()
    dim, st = device_basis(pf, torch, dev, 10)
    V = torch.ones((1, dim), dtype=torch.float64, device=dev) / dim ** 0.5
    V[0, 3] = float("nan")
    with pf.Ctx(0) as ctx:
        with pytest.raises(pf.PolfedError) as e:
            pf.entanglement_entropy(ctx, 10, st, V, dim, 1)
        assert e.value.code == pf.POLFED_ECUDA
