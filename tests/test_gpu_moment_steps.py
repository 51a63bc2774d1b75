"""Chebyshev moments of several steps per launch: single columns and padded
widths, sectors smaller than a launch, more steps than one launch carries, and
more columns than are filtered together, against the recurrence written with
H applied in FP64."""
import numpy as np
import pytest

import polfed_inputs as I
from gpu_common import device_basis, lib, torch_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,which,R,n_mom", [
    (4, "xxz", 1, 40), (8, "j1j2", 3, 1001), (10, "obc", 17, 64), (12, "xxz", 1, 130),
    (14, "j1j2", 33, 62), (18, "xxz", 128, 20),
])
@pytest.mark.parametrize("dtype,tol", [("F64", 1e-11), ("DF64", 1e-10), ("F32", 1e-3)])
def test_moments_follow_the_recurrence(L, which, R, n_mom, dtype, tol):
    torch, dev = torch_dev()
    pf = lib()
    m = {"xxz": I.xxz(L, 3.0, 5, 0), "j1j2": I.j1j2(L, 4.0, 5, 1), "obc": I.xxz(L, 2.0, 5, 2, periodic=False)}[which]
    b = 0.25 * L * (abs(m.J1) * 3 + abs(m.J2) * 3) + 0.5 * float(np.sum(np.abs(m.h)))  # >= |H|
    dim, st = device_basis(pf, torch, dev, L)
    X = torch.randn(dim, R, dtype=torch.float64, device=dev, generator=torch.Generator(dev).manual_seed(L))
    if dtype == "F32":
        X = X.float()
    got = pf.kpm_moments(m, st, dim, -b, b, n_mom, X, R, getattr(pf, dtype))

    def apply(v):
        y = torch.empty_like(v)
        pf.h_apply(m, st, dim, -b, b, v, y, R, pf.F64)
        torch.cuda.synchronize()
        return y

    t0 = X.double()
    t1 = apply(t0)
    want = np.empty(n_mom)
    m0, m1 = float((t0 * t0).sum()), float((t0 * t1).sum())
    for k in range((n_mom + 1) // 2):
        want[2 * k] = m0 if k == 0 else 2 * float((t0 * t0).sum()) - m0
        if 2 * k + 1 < n_mom:
            want[2 * k + 1] = m1 if k == 0 else 2 * float((t1 * t0).sum()) - m1
        t0, t1 = t1, 2 * apply(t1) - t0
    want /= R
    assert np.max(np.abs(got - want)) <= tol * want[0]
