"""What the scratch pool holds after calls that need no context, of more scratch than
it may keep: at most 1/256 of the device's memory, which nothing else can use."""
import pytest

import polfed_inputs as I
from gpu_common import device_basis, lib, torch_dev

pytestmark = pytest.mark.gpu


def test_pool_holds_little_after_a_large_call():
    torch, dev = torch_dev()
    pf = lib()
    L = 26  # three slices of 1.3 GB
    total = torch.cuda.get_device_properties(0).total_memory
    dim, st = device_basis(pf, torch, dev, L)
    X = torch.ones(dim, 32, device=dev)
    Y = torch.empty_like(X)
    m = I.xxz(L, 3.0, 2, 0)
    pf.h_apply(m, st, dim, -80.0, 80.0, X, Y, 32, pf.F32)
    pf.Ctx(0).close()  # gives back what the pool holds
    torch.cuda.synchronize()
    base = torch.cuda.mem_get_info()[0]
    for _ in range(2):
        pf.cheb_filter(m, st, dim, -80.0, 80.0, 0.0, 4, X, Y, 32, pf.F32)
    torch.cuda.synchronize()
    assert base - torch.cuda.mem_get_info()[0] <= total // 256 + (64 << 20)
