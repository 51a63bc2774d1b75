"""Calls of more than one launch whose grid barrier runs out (a lowered limit, set on
the host) return POLFED_ETIMEOUT, and the next call computes what it did before:
a filter of 1000 steps, per-column series, and moments, in the library's own
plans and in a context that keeps its buffers."""
import numpy as np
import pytest

import polfed_inputs as I
from gpu_common import device_basis, lib, torch_dev

pytestmark = pytest.mark.gpu


def _check(pf, call):
    want = call()
    try:
        pf.set_wait_limit(1)
        with pytest.raises(pf.PolfedError) as e:
            call()
        assert e.value.code == pf.POLFED_ETIMEOUT
    finally:
        pf.set_wait_limit(0)
    assert np.array_equal(call(), want)


def test_long_filters_and_moments_recover():
    torch, dev = torch_dev()
    pf = lib()
    L = 18
    dim, st = device_basis(pf, torch, dev, L)
    m = I.xxz(L, 3.0, 4, 0)
    X = torch.from_numpy(I.block(dim, 32, 5)).to(dev)
    X32 = X.float()
    C = np.random.default_rng(1).standard_normal((32, 1001)) / 1001

    def filt(dtype, x):
        y = torch.empty_like(x)
        pf.cheb_filter(m, st, dim, -60.0, 60.0, 0.0, 1000, x, y, 32, dtype)
        return y.cpu().numpy()

    def cols():
        y = torch.empty_like(X32)
        pf.cheb_filter_cols(m, st, dim, -60.0, 60.0, C, X32, y, 32)
        return y.cpu().numpy()

    _check(pf, lambda: filt(pf.F64, X))
    _check(pf, lambda: filt(pf.F32, X32))
    _check(pf, cols)
    for dtype, x in ((pf.F32, X32), (pf.F64, X), (pf.DF64, X)):
        _check(pf, lambda: pf.kpm_moments(m, st, dim, -60.0, 60.0, 2000, x, 32, dtype))


def test_a_context_recovers():
    torch_dev()
    pf = lib()
    m = I.xxz(16, 3.0, 4, 0)
    with pf.Ctx(0) as ctx:
        _check(pf, lambda: np.array(pf.spectral_labels(ctx, m, 0.5, 128, 16)))
