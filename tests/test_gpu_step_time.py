"""The device time that the counters report is that of this thread's own step
launches: calls of several threads take turns on the device, so what the threads
report cannot add up to more than the time that passed."""
import threading
import time

import pytest

import polfed_inputs as I
from gpu_common import device_basis, lib, torch_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batched", [False, True])
def test_threads_report_their_own_device_time(batched):
    torch, dev = torch_dev()
    pf = lib()
    L, n_b, K, n_thr, reps = 14, 32, 400, 3, 20
    dim, st = device_basis(pf, torch, dev, L)
    m = I.xxz(L, 3.0, 1, 0)
    X = torch.randn(dim, n_b, device=dev)
    spent = [0.0] * n_thr
    start = threading.Barrier(n_thr + 1)

    def work(i):
        s = torch.cuda.Stream(dev)
        y = torch.empty_like(X)

        def call():
            if batched:
                pf.cheb_filter_batched([m], [-40.0], [40.0], [0.0], [K], [X], [y], n_b, pf.F32, stream=s.cuda_stream)
            else:
                pf.cheb_filter(m, st, dim, -40.0, 40.0, 0.0, K, X, y, n_b, pf.F32, stream=s.cuda_stream)

        call()
        a = pf.get_counters()["step_gpu_s"]
        start.wait()
        for _ in range(reps):
            call()
        spent[i] = pf.get_counters()["step_gpu_s"] - a

    torch.cuda.synchronize()
    ts = [threading.Thread(target=work, args=(i,)) for i in range(n_thr)]
    [t.start() for t in ts]
    start.wait()
    t0 = time.perf_counter()
    [t.join() for t in ts]
    wall = time.perf_counter() - t0
    assert min(spent) > 0.0
    assert sum(spent) <= 1.02 * wall
