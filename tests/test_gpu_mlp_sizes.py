"""The fused network kernels at the edges of their tiles, batch shares and range
(512 inputs and hidden units; wider networks run one kernel per layer), against
the oracle's gradient."""
import numpy as np
import pytest

from gpu_common import lib, torch_dev
from oracle import mlp_oracle as MO

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_in,H,d_out,B", [(1, 3, 3, 1), (33, 31, 5, 67), (23, 65, 3, 1030), (512, 512, 4, 40),
                                             (40, 513, 3, 9), (513, 64, 64, 33)])
def test_gradient_forward_and_loss_at_size_edges(d_in, H, d_out, B):
    torch, dev = torch_dev()
    pf = lib()
    rng = np.random.default_rng(d_in + H)
    p = MO.glorot_params(d_in, H, d_out, rng).astype(np.float32)
    net = pf.MLP(d_in, H, d_out)
    net.set_params(p)
    x = rng.normal(size=(B, d_in)).astype(np.float32)
    t = rng.normal(size=(B, d_out)).astype(np.float32)
    dx, dt = torch.from_numpy(x).to(dev), torch.from_numpy(t).to(dev)
    g = torch.full((net.num_params,), float("nan"), device=dev)
    loss = net.grad(dx, dt, B, g)
    p64, x64, t64 = p.astype(np.float64), x.astype(np.float64), t.astype(np.float64)
    wl, wg = MO.loss_and_grad(p64, x64, t64, d_in, H, d_out)
    assert loss == pytest.approx(wl, rel=1e-5)
    assert np.max(np.abs(g.cpu().numpy() - wg)) <= 2e-5 * np.max(np.abs(wg))
    dy = torch.empty((B, d_out), device=dev)
    net.forward(dx, B, dy)
    one = (np.zeros(d_in), np.ones(d_in), np.zeros(d_out), np.ones(d_out))
    want = MO.predict(p64, x64, d_in, H, d_out, one)
    assert np.max(np.abs(dy.cpu().numpy() - want)) <= 1e-5 * max(1.0, np.max(np.abs(want)))
    # the Adam step starts from the same gradient: first step lr * sign(g) where g is not tiny
    net.train_step(dx, dt, B, 1e-3)
    step = net.get_params().astype(np.float64) - p64
    big = np.abs(wg) > 1e-3 * np.max(np.abs(wg))
    assert np.max(np.abs(step + 1e-3 * np.sign(wg))[big]) <= 2e-5
