"""Contexts with a bounded workspace: the bounds here are the least that each call
needs with one column slice's recurrence buffers at a time, and it runs within
them, with the results of a context without a bound."""
import numpy as np
import pytest

import polfed_inputs as I
from gpu_common import lib, torch_dev

pytestmark = pytest.mark.gpu

# bytes: the smallest accepted bound, found by bisection to 4096 bytes
EIGS = [(12, 20, 16, "F32", 6815640), (12, 20, 64, "F32", 18665187), (12, 20, 64, "F64", 23133855),
        (12, 20, 64, "DF64", 23133855), (14, 30, 64, "F32", 66780165), (14, 30, 64, "DF64", 74591117)]


@pytest.mark.parametrize("L,n_ev,n_b,prec,bound", EIGS)
def test_eigs_within_the_least_workspace(L, n_ev, n_b, prec, bound):
    torch_dev()
    pf = lib()
    o = pf.opts_default()
    o.precision = getattr(pf, prec)
    got = []
    for ws in (0, bound + 4096):
        with pf.Ctx(0, ws) as ctx:
            got.append(pf.eigs(ctx, I.xxz(L, 3.0, 1, 0), 0.5, n_ev, 0, n_b, o, allow_noconv=True))
    assert got[0][3] == got[1][3]
    # both resolve the same eigenvalues to tol_resid |H|
    assert np.max(np.abs(got[0][0] - got[1][0])) < 1e-8 * got[0][2]["E_max"]


def test_other_calls_within_the_least_workspace():
    torch_dev()
    pf = lib()
    m12, m14, m16 = (I.xxz(L, 3.0, 1, 0) for L in (12, 14, 16))
    o = pf.opts_default()
    o.precision, o.dos_rule = pf.DF64, pf.DOS_KPM
    for bound, call in ((36982219, lambda c: pf.eigs(c, m14, 0.5, 20, 0, 32, o, allow_noconv=True)),
                        (37223880, lambda c: pf.block_lanczos(c, m12, -40.0, 40.0, 0.0, 60, 64, 20, allow_noconv=True)),
                        (1470441, lambda c: pf.spectral_bounds(c, m14)),
                        (10182500, lambda c: pf.spectral_labels(c, m14, 0.5, 64, 64)),
                        (33598975, lambda c: pf.spectral_labels(c, m16, 0.5, 64, 64))):
        with pf.Ctx(0, bound + 4096) as ctx:
            call(ctx)
        with pf.Ctx(0, 65536) as ctx:
            with pytest.raises(pf.PolfedError) as e:
                call(ctx)
            assert e.value.code == pf.POLFED_ENOMEM
