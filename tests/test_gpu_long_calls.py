"""A long filter does not hold the device to its end: a short call of another
thread gets its turn between two launches of the long one."""
import threading
import time

import numpy as np
import pytest

import polfed_inputs as I
from gpu_common import device_basis, lib, torch_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["filter", "batched", "moments"])
def test_a_short_filter_runs_beside_a_long_call(kind):
    torch, dev = torch_dev()
    pf = lib()
    L = 18 if kind == "moments" else 14
    dim, st = device_basis(pf, torch, dev, L)
    m = I.xxz(L, 3.0, 1, 0)
    X = torch.randn(dim, 16, dtype=torch.float64, device=dev)
    Y = torch.empty_like(X)
    dim_s, st_s = device_basis(pf, torch, dev, 10)
    m_s = I.xxz(10, 3.0, 1, 1)
    X_s = torch.randn(dim_s, 4, dtype=torch.float64, device=dev)
    Y_s = torch.empty_like(X_s)
    s = torch.cuda.Stream(dev)

    def short():
        pf.cheb_filter(m_s, st_s, dim_s, -30.0, 30.0, 0.0, 20, X_s, Y_s, 4, pf.F64, stream=s.cuda_stream)

    short()
    want = Y_s.clone()
    torch.cuda.synchronize()
    ended = []

    def long_call():
        q = torch.cuda.Stream(dev)
        if kind == "filter":
            pf.cheb_filter(m, st, dim, -40.0, 40.0, 0.0, 400000, X, Y, 16, pf.F64, stream=q.cuda_stream)
        elif kind == "batched":
            pf.cheb_filter_batched([m], [-40.0], [40.0], [0.0], [400000], [X], [Y], 16, pf.DF64, stream=q.cuda_stream)
        else:
            pf.kpm_moments(m, st, dim, -60.0, 60.0, 65536, X, 16, pf.DF64, stream=q.cuda_stream)
        ended.append(time.perf_counter())

    t = threading.Thread(target=long_call)
    t.start()
    time.sleep(0.1)
    done = []
    for _ in range(3):
        Y_s.zero_()
        torch.cuda.synchronize()
        short()
        done.append(time.perf_counter())
    t.join()
    assert np.all(np.array(done) < ended[0]), (done, ended)
    assert torch.equal(Y_s, want)
