"""Sectors whose 128-byte slices exceed L2 are filtered in 64-byte rows (XXZ): the
block equals narrow blocks of its own columns, bit for bit."""
import pytest

import polfed_inputs as I
from gpu_common import device_basis, lib, torch_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,n_b", [("F32", 32), ("F32", 21), ("DF64", 16)])
def test_columns_do_not_depend_on_the_row_size(dtype, n_b):
    torch, dev = torch_dev()
    pf = lib()
    L, K = 24, 4
    m = I.xxz(L, 3.0, 3, 0)
    dim, st = device_basis(pf, torch, dev, L)
    X = torch.randn(dim, n_b, dtype=torch.float32 if dtype == "F32" else torch.float64, device=dev,
                    generator=torch.Generator(dev).manual_seed(n_b))

    def run(a, b):
        x = X[:, a:b].contiguous()
        y = torch.empty_like(x)
        pf.cheb_filter(m, st, dim, -80.0, 80.0, 0.1, K, x, y, b - a, getattr(pf, dtype))
        torch.cuda.synchronize()
        return y

    whole = run(0, n_b)
    for a, b in ((0, 1), (n_b // 2, n_b // 2 + 4), (n_b - 3, n_b)):
        assert torch.equal(whole[:, a:b], run(a, b))
