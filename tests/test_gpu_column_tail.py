"""Blocks whose slices run one after the other: the columns beyond the last full
slice go through a narrower one.  Each column's arithmetic does not depend on its
slice, so the block equals its full slices and its tail computed by themselves,
bit for bit."""
import numpy as np
import pytest

import polfed_inputs as I
from gpu_common import device_basis, lib, torch_dev

pytestmark = pytest.mark.gpu
L = 20


@pytest.mark.parametrize("dtype,n_b,full", [("F32", 37, 32), ("F32", 33, 32), ("F32", 79, 64), ("F64", 21, 16),
                                            ("DF64", 17, 16), ("DF64", 37, 32)])
@pytest.mark.parametrize("what", ["apply", "filter", "filter0", "cols"])
def test_tail_columns_equal_a_block_of_their_own(dtype, n_b, full, what):
    torch, dev = torch_dev()
    if what == "cols" and dtype != "F32":
        pytest.skip("per-column coefficients are FP32")
    pf = lib()
    m = I.j1j2(L, 4.0, 3, 0)
    dim, st = device_basis(pf, torch, dev, L)
    td = torch.float32 if dtype == "F32" else torch.float64
    X = torch.randn(dim, n_b, dtype=td, device=dev, generator=torch.Generator(dev).manual_seed(n_b))
    c = np.random.default_rng(n_b).standard_normal((n_b, 7))

    def run(a, b):
        x = X[:, a:b].contiguous()
        y = torch.empty_like(x)
        k = getattr(pf, dtype)
        if what == "apply":
            pf.h_apply(m, st, dim, -80.0, 80.0, x, y, b - a, k)
        elif what == "cols":
            pf.cheb_filter_cols(m, st, dim, -80.0, 80.0, c[a:b], x, y, b - a)
        else:
            pf.cheb_filter(m, st, dim, -80.0, 80.0, 0.1, 0 if what == "filter0" else 6, x, y, b - a, k)
        torch.cuda.synchronize()
        return y

    assert torch.equal(run(0, n_b), torch.cat([run(0, full), run(full, n_b)], dim=1))


def test_moments_of_a_block_with_a_tail():
    torch, dev = torch_dev()
    pf = lib()
    m = I.xxz(L, 3.0, 3, 1)
    dim, st = device_basis(pf, torch, dev, L)
    X = torch.randn(dim, 21, dtype=torch.float64, device=dev, generator=torch.Generator(dev).manual_seed(1))
    mu = lambda x: x.shape[1] * pf.kpm_moments(m, st, dim, -60.0, 60.0, 12, x.contiguous(), x.shape[1], pf.DF64)
    got, want = mu(X), mu(X[:, :16]) + mu(X[:, 16:])
    assert np.max(np.abs(got - want)) <= 1e-13 * want[0]
