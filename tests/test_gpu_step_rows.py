"""The step kernel at the edges of its launch and data layout: numbers of steps
around what one launch carries (448), blocks of one column up to several slices,
blocks whose base or row pitch does not allow vector loads, and column slices
that run together or one after the other, against the spectral definition."""
import numpy as np
import pytest

import oracle as O
import polfed_inputs as I
from gpu_common import device_basis, lib, models, torch_dev

pytestmark = pytest.mark.gpu


def _tol(pf, dtype, K):
    # linear growth of the Clenshaw rounding error with K, as in test_gpu_kernels.py
    return {pf.F64: 1e-13 * (K + 1), pf.DF64: 1e-12 * (K + 1), pf.F32: 2e-7 * (K + 1) + 1e-6}[dtype]


@pytest.mark.parametrize("L,model", [(4, 0), (4, 1), (8, 0), (8, 3), (10, 1)])
@pytest.mark.parametrize("K,n_b,shift", [(1, 1, 0), (2, 3, 1), (447, 16, 0), (448, 37, 0), (449, 5, 1), (900, 128, 0)])
def test_filter_at_launch_and_layout_edges(L, model, K, n_b, shift):
    torch, dev = torch_dev()
    pf = lib()
    dim, st = device_basis(pf, torch, dev, L)
    m = models(L)[model]
    H, _ = O.dense_hamiltonian(m.L, m.J1, m.J2, m.Delta, m.h, m.periodic)
    w, V = np.linalg.eigh(H)
    lo, hi = w[0] - 0.05, w[-1] + 0.07
    lt = (2 * w - lo - hi) / (hi - lo)
    X = I.block(dim, n_b, K + L)
    want = O.filter_spectral(lt, V, X, 0.31, K)
    for dtype in (pf.F64, pf.DF64, pf.F32):
        tdt = torch.float32 if dtype == pf.F32 else torch.float64
        buf = torch.empty(2 * dim * n_b + 2, dtype=tdt, device=dev)
        Xd = buf[shift:shift + dim * n_b]  # shift 1: not aligned for vector access
        Yd = buf[dim * n_b + 1 + shift:][:dim * n_b]
        Xd.copy_(torch.from_numpy(X).to(dev, tdt).reshape(-1))
        pf.cheb_filter(m, st, dim, lo, hi, 0.31, K, Xd, Yd, n_b, dtype)
        err = np.abs(Yd.double().cpu().numpy().reshape(dim, n_b) - want).max() / np.abs(X).max()
        assert err < _tol(pf, dtype, K), (dtype, err)


@pytest.mark.parametrize("L,n_b", [(16, 100), (20, 70)])
def test_slices_together_and_in_turn_agree(L, n_b):
    """L = 16: all slices of the block in one launch; L = 20: groups of them.  Every
    column equals the filter of that column's own narrow block."""
    torch, dev = torch_dev()
    pf = lib()
    dim, st = device_basis(pf, torch, dev, L)
    m = I.j1j2(L, 3.0, 5, 1)
    b = 1.01 * (L * 2 * (0.5 + 0.55 / 4) + 0.5 * float(np.abs(m.h).sum()))
    X = torch.from_numpy(I.block(dim, n_b, 8)).to(dev)
    Y = torch.empty_like(X)
    pf.cheb_filter(m, st, dim, -b, b, 0.0, 20, X, Y, n_b, pf.F64)
    for c0, c1 in ((0, 1), (n_b - 3, n_b)):
        x = X[:, c0:c1].contiguous()
        y = torch.empty_like(x)
        pf.cheb_filter(m, st, dim, -b, b, 0.0, 20, x, y, c1 - c0, pf.F64)
        assert float((y - Y[:, c0:c1]).abs().max()) < 1e-13 * 21 * float(X.abs().max())
