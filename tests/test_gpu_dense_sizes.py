"""Block operations and the bounds recurrence at the edges of their sizes: every
block width (Gram chunks, Cholesky with its inverse in shared or global memory),
and single-vector Lanczos on sectors smaller than one check interval."""
import numpy as np
import pytest

import oracle as O
import polfed_inputs as I
from gpu_common import lib, models, torch_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [4, 6, 8, 10])
def test_spectral_bounds_of_small_sectors(L):
    torch_dev()
    pf = lib()
    for m in models(L):
        H, _ = O.dense_hamiltonian(m.L, m.J1, m.J2, m.Delta, m.h, m.periodic)
        w = np.linalg.eigvalsh(H)
        nrm = max(abs(w[0]), abs(w[-1]))
        with pf.Ctx(0) as ctx:
            lo, hi, err = pf.spectral_bounds(ctx, m)
        assert abs(lo - w[0]) <= 1e-10 * nrm and abs(hi - w[-1]) <= 1e-10 * nrm
        assert 0.0 <= err <= 1e-8 * nrm


def test_every_block_width_gives_the_same_eigenpairs():
    torch, dev = torch_dev()
    pf = lib()
    m = I.xxz(14, 3.0, 11, 0)
    ref = ref_res = None
    for n_b in (16, 32, 64, 128):
        with pf.Ctx(0) as ctx:
            ev, res, st, rc = pf.eigs(ctx, m, 0.5, 40, 0, n_b)
        nrm = max(abs(st["E_min"]), abs(st["E_max"]))
        assert rc == 0 and np.max(res) <= 1e-8 * nrm
        if ref is None:
            ref, ref_res = ev, res
        # both within their residual of the same level (spacing 1e-3)
        assert np.all(np.abs(ev - ref) <= res + ref_res + 1e-13 * nrm)
