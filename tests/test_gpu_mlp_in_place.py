"""Network outputs written over its inputs: polfed_mlp_forward reads all of d_x
before it writes where the two overlap, for the fused and the per-layer kernels."""
import pytest

from gpu_common import lib, torch_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_in,H,d_out", [(23, 128, 3), (3, 64, 40), (8, 16, 8), (600, 64, 5)])
@pytest.mark.parametrize("B", [5, 1000, 9001])
def test_forward_over_its_inputs(d_in, H, d_out, B):
    torch, dev = torch_dev()
    pf = lib()
    net = pf.MLP(d_in, H, d_out, 7)
    x = torch.randn(B * d_in, device=dev, generator=torch.Generator(dev).manual_seed(B))
    want = torch.empty(B * d_out, device=dev)
    net.forward(x, B, want)
    n = B * (d_in + d_out)
    for at in (0, 1, B * d_in // 2, B * d_in - 1):  # outputs from the at-th input on; after them nothing changes
        buf = torch.full((n,), 3.0, device=dev)
        buf[:B * d_in] = x
        rest = buf.clone()
        torch.cuda.synchronize()
        net.forward(buf, B, buf[at:at + B * d_out])
        assert torch.equal(buf[at:at + B * d_out], want)
        rest[at:at + B * d_out] = want
        assert torch.equal(buf, rest)
    # and inputs that begin inside the outputs
    buf = torch.zeros(n, device=dev)
    at = min(B * d_out - 1, B * d_out // 2)
    buf[at:at + B * d_in] = x
    torch.cuda.synchronize()
    net.forward(buf[at:at + B * d_in], B, buf[:B * d_out])
    assert torch.equal(buf[:B * d_out], want)
