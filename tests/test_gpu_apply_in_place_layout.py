"""H~ on a block whose rows are whole slices of aligned 16-byte chunks is gathered
from the block itself; off that alignment it goes through slices.  Both do the same
arithmetic, so the same block at an odd offset gives the same bits."""
import pytest

from gpu_common import device_basis, lib, models, torch_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [4, 8, 14, 18])
@pytest.mark.parametrize("dtype,n_b", [("F32", 4), ("F32", 8), ("F32", 16), ("F32", 32), ("F32", 96), ("F64", 2), ("F64", 4),
                                       ("F64", 8), ("F64", 16), ("F64", 48), ("F64", 128), ("F64", 24), ("F32", 36)])
def test_direct_rows_equal_slices(L, dtype, n_b):
    torch, dev = torch_dev()
    pf = lib()
    dim, st = device_basis(pf, torch, dev, L)
    td = torch.float32 if dtype == "F32" else torch.float64
    X = torch.randn(dim * n_b, dtype=td, device=dev, generator=torch.Generator(dev).manual_seed(n_b))
    for m in models(L):
        out = []
        for shift in (0, 1):
            x = torch.empty(dim * n_b + 4, dtype=td, device=dev)[shift:shift + dim * n_b]
            guard = torch.full((dim * n_b + 8,), 7.0, dtype=td, device=dev)
            y = guard[4 + shift:4 + shift + dim * n_b]
            x.copy_(X)
            pf.h_apply(m, st, dim, -90.0, 90.0, x, y, n_b, getattr(pf, dtype))
            torch.cuda.synchronize()
            assert bool((guard[:4 + shift] == 7.0).all()) and bool((guard[4 + shift + dim * n_b:] == 7.0).all())
            out.append(y.clone())
        assert torch.equal(out[0], out[1])
