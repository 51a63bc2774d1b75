"""Scratch of the context-free calls comes from a pool that keeps a bounded amount
between calls: memory stays bounded, is given back with a context, and calls from
several threads on streams of their own give the results of one."""
import threading

import pytest

import polfed_inputs as I
from gpu_common import device_basis, lib, torch_dev

pytestmark = pytest.mark.gpu


def test_pool_is_bounded_and_given_back():
    torch, dev = torch_dev()
    pf = lib()
    total = torch.cuda.get_device_properties(0).total_memory
    m = I.xxz(18, 3.0, 2, 0)
    dim, st = device_basis(pf, torch, dev, 18)
    X = torch.randn(dim, 5, device=dev)
    Y = torch.empty_like(X)
    pf.h_apply(m, st, dim, -60.0, 60.0, X, Y, 5, pf.F32)
    pf.Ctx(0).close()
    torch.cuda.synchronize()
    base = torch.cuda.mem_get_info()[0]
    for n_b in (128, 5, 77, 128):
        x = torch.randn(dim, n_b, device=dev)
        pf.cheb_filter(m, st, dim, -60.0, 60.0, 0.0, 4, x, torch.empty_like(x), n_b, pf.F32)
    del x
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    assert base - torch.cuda.mem_get_info()[0] <= total // 64 + (64 << 20)
    pf.Ctx(0).close()
    assert base - torch.cuda.mem_get_info()[0] <= 64 << 20


def test_threads_and_streams_share_the_pool():
    torch, dev = torch_dev()
    pf = lib()
    L, K = 14, 20
    dim, st = device_basis(pf, torch, dev, L)
    ms = [I.xxz(L, 3.0, 2, i) for i in range(4)]
    Xs = [torch.randn(dim, 9 + i, dtype=torch.float64, device=dev, generator=torch.Generator(dev).manual_seed(i)) for i in range(4)]
    want, got = [], [[None] * 5 for _ in ms]

    def run(i, stream):
        y = torch.empty_like(Xs[i])
        pf.cheb_filter(ms[i], st, dim, -40.0, 40.0, 0.1, K, Xs[i], y, Xs[i].shape[1], pf.F64, stream=stream)
        return y

    for i in range(4):
        want.append(run(i, None))
    torch.cuda.synchronize()

    def work(i):
        s = torch.cuda.Stream(dev)
        with torch.cuda.stream(s):
            for r in range(5):
                got[i][r] = run(i, s.cuda_stream)
        s.synchronize()

    ts = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    torch.cuda.synchronize()
    for i in range(4):
        for r in range(5):
            assert torch.equal(got[i][r], want[i])
