"""FP32 moments keep the order of their sums: bond by bond (high, low, cross, or
low, cross, high for 128-byte rows of large groups), then the diagonal.  The
recurrence is repeated here in FP32 with that order, so that only the FP64 sums
over rows and columns are left to differ (1e-9, two orders below FP32 noise)."""
import numpy as np
import pytest

import polfed_inputs as I
from gpu_common import device_basis, lib, torch_dev

pytestmark = pytest.mark.gpu


def _tables(m, b, alpha, beta, st):
    """Diagonal in FP32 and, per class, [(indices of the antiparallel rows, their partners)] by part."""
    L = m.L
    bonds = [(min(i, (i + l) % L), max(i, (i + l) % L), l) for l, J in ((1, m.J1), (2, m.J2)) if J
             for i in range(L) if m.periodic or i + l < L]
    z = [((st >> i) & 1).astype(np.float64) - 0.5 for i in range(L)]
    part = {"low": [], "high": [], "cross": []}
    d = {"low": np.zeros(st.size), "high": np.zeros(st.size), "cross": np.zeros(st.size)}
    for i, j, l in bonds:
        k = "low" if j < b else ("high" if i >= b else "cross")
        d[k] += (m.J1 if l == 1 else m.J2) * m.Delta * z[i] * z[j]
        rows = np.nonzero(z[i] != z[j])[0]
        part[k].append((l, rows, np.searchsorted(st, st[rows] ^ ((1 << i) | (1 << j)))))
    for i in range(L):
        d["low" if i < b else "high"] += m.h[i] * z[i]
    f = lambda v: v.astype(np.float32)
    return f(alpha * d["low"]) + f(alpha * (d["high"] - beta)) + f(alpha * d["cross"]), part


@pytest.mark.parametrize("L,which,R,low_first", [(8, "j1j2", 3, False), (14, "xxz", 20, False), (18, "xxz", 17, True),
                                                 (18, "j1j2", 18, True), (18, "xxz", 9, False)])
def test_fp32_moments_in_bond_order(L, which, R, low_first):
    torch, dev = torch_dev()
    pf = lib()
    m = I.xxz(L, 3.0, 9, 0) if which == "xxz" else I.j1j2(L, 4.0, 9, 1)
    e_lo, e_hi = -1.1 * L - 1.0, 1.1 * L
    dim, dst = device_basis(pf, torch, dev, L)
    st = dst.cpu().numpy().astype(np.int64)
    alpha, beta = 2.0 / (e_hi - e_lo), 0.5 * (e_hi + e_lo)
    diag, part = _tables(m, max(2, L - 10), alpha, beta, st)
    o = {1: np.float32(alpha * 0.5 * m.J1), 2: np.float32(alpha * 0.5 * m.J2)}
    wide = lambda v: v.astype(np.float64)  # an FP32 product is exact in FP64: fma = one sum rounded to FP32

    def apply(t):
        s = {1: np.zeros_like(t), 2: np.zeros_like(t)}
        for k in ("low", "cross", "high") if low_first else ("high", "low", "cross"):
            for l, rows, nb in part[k]:
                s[l][rows] += t[nb]
        y = (wide(diag)[:, None] * wide(t) + wide(o[1] * s[1])).astype(np.float32)
        return (wide(y) + wide(s[2]) * float(o[2])).astype(np.float32) if m.J2 else y

    X = np.random.default_rng(L).standard_normal((dim, R)).astype(np.float32)
    n_mom = 16
    got = pf.kpm_moments(m, dst, dim, e_lo, e_hi, n_mom, torch.from_numpy(X).to(dev), R, pf.F32)
    raw, t0, t1 = np.zeros(n_mom), X, apply(X)
    for k in range(n_mom // 2):
        raw[2 * k], raw[2 * k + 1] = (wide(t0) ** 2).sum(), (wide(t0) * wide(t1)).sum()
        t0, t1 = t1, (2.0 * wide(apply(t1)) - wide(t0)).astype(np.float32)
    want = np.where(np.arange(n_mom) < 2, raw, 2.0 * raw - np.where(np.arange(n_mom) % 2, raw[1], raw[0])) / R
    assert np.max(np.abs(got - want)) <= 1e-9 * want[0]
