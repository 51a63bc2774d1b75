"""Networks of different sizes used by several threads at once: each call finds
the shared memory that its own size needs."""
import threading

import pytest

from gpu_common import lib, torch_dev

pytestmark = pytest.mark.gpu


def test_networks_of_two_sizes_on_eight_threads():
    torch, dev = torch_dev()
    pf = lib()
    # 8 batch rows x (inputs + 3 x hidden + 2 x outputs) floats: 65 and 55 KB
    nets = [pf.MLP(512, 512 if i % 2 else 400, 3, i) for i in range(8)]
    B = 1100
    X = torch.randn(B, 512, device=dev)
    want = []
    for n in nets:
        y = torch.empty(B, 3, device=dev)
        n.forward(X, B, y)
        want.append(y)
    torch.cuda.synchronize()
    errors = []

    def work(i):
        s = torch.cuda.Stream(dev)
        y = torch.zeros(B, 3, device=dev)
        s.wait_stream(torch.cuda.current_stream(dev))
        for _ in range(3000):
            try:
                nets[i].forward(X, B, y, stream=s.cuda_stream)
            except pf.PolfedError as e:
                errors.append(str(e))
        s.synchronize()
        if not torch.equal(y, want[i]):
            errors.append(f"network {i}: other outputs")

    ts = [threading.Thread(target=work, args=(i,)) for i in range(8)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not errors, (len(errors), errors[:3])
