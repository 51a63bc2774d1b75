"""Workloads of the library as a user's program runs them, for timing and for comparing outputs.

Every case goes through the public entry points of ``paper_2005_09534_gb300``:
the H~ application, the Chebyshev filter (one coefficient set, or one per
column), the batched filter of many realizations, the KPM moments behind the
predictor's labels, the entanglement entropy of eigenvectors, a gradient of
the predictor's network, and a whole eigenpair run.  Sizes are those of the
repository's workloads (L = 12..24, the XXZ and J1-J2 points, n_b 1..128);
the filter orders are shorter than a production run's so that a pass stays
well under a second, which leaves the time per recurrence step unchanged.
"""
import math

import numpy as np
import torch

import paper_2005_09534_gb300 as pf

DEV = "cuda"
DTYPES = {"f64": pf.F64, "f32": pf.F32, "df64": pf.DF64}


# --------------------------------------------------------------------- cases
def listed():
    return [
        # one H application to one vector: the inner call of a Lanczos bound probe; latency only
        dict(name="apply_L12_f64_1", kind="apply", L=12, model="xxz", W=3.0, n_b=1, dtype="f64", scaled=False),
        # images H~ U of one 64-column panel in a Rayleigh-Ritz step of the L = 22 run
        dict(name="apply_L22_f64_64", kind="apply", L=22, model="xxz", W=3.0, n_b=64, dtype="f64", scaled=True),
        # plain FP64 filter of a 16-column block at L = 14, mid-spectrum target
        dict(name="filter_L14_f64_16", kind="filter", L=14, model="xxz", W=3.0, n_b=16, dtype="f64", K=200, sigma=0.0),
        # float-float filter of the L = 20 J1-J2 run's 32-column block
        dict(name="filter_L20_j1j2_df64_32", kind="filter", L=20, model="j1j2", W=4.0, n_b=32, dtype="df64", K=64,
             sigma=0.0),
        # FP32 filter of the L = 22 XXZ run's 64-column block: the headline run spends 98% of a step here
        dict(name="filter_L22_f32_64", kind="filter", L=22, model="xxz", W=3.0, n_b=64, dtype="f32", K=200, sigma=0.0),
        # FP32 filter of the L = 24 J1-J2 run's block: the largest workload
        dict(name="filter_L24_j1j2_f32_64", kind="filter", L=24, model="j1j2", W=5.0, n_b=64, dtype="f32", K=24,
             sigma=0.0),
        # a refinement sweep's per-column filter: a ragged number of columns is still converging
        dict(name="cols_L20_j1j2_f32_37", kind="cols", L=20, model="j1j2", W=4.0, n_b=37, K=48),
        # one round of the batched runner: L = 16 and 18 rings, orders of their own, FP32
        dict(name="batched16_L16_L18_f32_32", kind="batched", n=16, L=16, L2=18, W=3.0, n_b=32, dtype="f32", K=160),
        # density-of-states moments of one predictor label: 16 random vectors, 256 moments
        dict(name="moments_L18_df64_16", kind="moments", L=18, model="xxz", W=3.0, R=16, n_mom=256, dtype="df64"),
        # half-chain entropies of the 50 eigenvectors of an L = 14 run
        dict(name="entropy_L14_50", kind="entropy", L=14, n_vec=50),
        # one training gradient of the L = 22 predictor (23 inputs, 2 x 128 hidden, 3 outputs, batch 256)
        dict(name="mlp_grad_23_128_256", kind="mlp", d_in=23, hidden=128, B=256),
        # a whole run: 50 eigenpairs of an L = 14 ring, FP32 filter with refinement
        dict(name="eigs_L14_f32_50", kind="eigs", L=14, model="xxz", W=3.0, N_ev=50, n_b=16, dtype="f32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# column steps x bytes x bonds of the largest listed case
_COST = 2704156 * 64 * 24 * 4 * 2


def _cost(c, n_b, K, per):
    return math.comb(c["L"], c["L"] // 2) * n_b * K * per * (2 if c["model"] == "j1j2" else 1)


def draw(rng):
    kind = rng.choice(["apply", "filter", "filter", "filter", "cols", "batched", "moments", "entropy", "mlp", "eigs"])
    c = {"kind": kind}
    if kind in ("apply", "filter", "cols"):
        c["L"] = rng.choice([12, 14, 16, 18, 20, 22, 24])
        c["model"] = rng.choice(["xxz", "j1j2", "xxz_open"])
        c["W"] = round(rng.uniform(1.0, 8.0), 2)
        c["n_b"] = _log(rng, 1, 128)
        if kind != "cols":
            c["dtype"] = rng.choice(["f32", "df64", "f64"])
        per = {"f64": 32, "df64": 10, "f32": 4}[c.get("dtype", "f32")]  # FP64 arithmetic is the slow one
        if kind == "apply":
            c["scaled"] = rng.random() < 0.7
            while _cost(c, c["n_b"], 6, per) > _COST:
                c["n_b"] = max(1, c["n_b"] // 2)
        else:
            c["K"] = _log(rng, 8, 400)
            if kind == "filter":
                c["sigma"] = 0.0 if rng.random() < 0.5 else round(rng.uniform(-0.8, 0.8), 3)
            while _cost(c, max(c["n_b"], 4), c["K"] + 4, per) > _COST:
                if c["K"] > 16:
                    c["K"] = c["K"] // 2
                else:
                    c["n_b"] = c["n_b"] // 2
    elif kind == "batched":
        c.update(n=_log(rng, 2, 24), L=rng.choice([12, 14, 16]), L2=rng.choice([14, 16, 18]),
                 W=round(rng.uniform(1.0, 8.0), 2), n_b=rng.choice([8, 16, 32, 48, 64]),
                 dtype=rng.choice(["f32", "df64"]), K=_log(rng, 24, 240))
    elif kind == "moments":
        c.update(L=rng.choice([12, 14, 16, 18, 20]), model=rng.choice(["xxz", "j1j2"]), W=round(rng.uniform(1.0, 8.0), 2),
                 R=_log(rng, 4, 32), n_mom=_log(rng, 32, 256), dtype=rng.choice(["df64", "f64", "f32"]))
    elif kind == "entropy":
        c.update(L=rng.choice([10, 12, 14]), n_vec=_log(rng, 4, 100))
    elif kind == "mlp":
        c.update(d_in=rng.randint(13, 25), hidden=_log(rng, 32, 256), B=_log(rng, 32, 4224))
    else:
        c.update(L=rng.choice([12, 14]), model="xxz", W=round(rng.uniform(2.0, 6.0), 2), N_ev=rng.randint(20, 50),
                 n_b=rng.choice([8, 16]), dtype=rng.choice(["f32", "df64"]))
    return c


# ------------------------------------------------------------------- inputs
class _Chain:
    """Parameters of Eq. (1) in the form the library's calls take."""

    def __init__(self, L, model, W, seed):
        self.L = L
        self.J1 = 1.0
        self.J2, self.Delta = (1.0, 0.55) if model == "j1j2" else (0.0, 1.0)
        self.periodic = not model.endswith("_open")
        self.h = np.random.default_rng(seed).uniform(-W, W, L)
        # an interval that holds the spectrum: every bond term lies in [-|J| (1/2 + Delta/4), |J| Delta/4 or (1/2 - Delta/4)]
        nb1, nb2 = (L, L) if self.periodic else (L - 1, L - 2)
        J = nb1 * abs(self.J1) + nb2 * abs(self.J2)
        f = 0.5 * float(np.abs(self.h).sum())
        self.e_lo = -J * (0.5 + self.Delta / 4) - f
        self.e_hi = J * max(self.Delta / 4, 0.5 - self.Delta / 4) + f

    def bonds(self):
        out = []
        for l, J in ((1, self.J1), (2, self.J2)):
            if J != 0.0:
                out += [(i, (i + l) % self.L, J) for i in range(self.L) if i + l < self.L or self.periodic]
        return out


def _dim(L):
    return math.comb(L, L // 2)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _block(dim, n, seed, dtype):
    """Columns of unit length on average, as the columns of a Lanczos block are."""
    t = torch.float32 if dtype == "f32" else torch.float64
    return torch.randn((dim, n), generator=_gen(seed), device=DEV, dtype=t) / math.sqrt(dim)


def _basis(L):
    dim = pf.basis_build(L, L // 2)
    st = torch.empty(dim, dtype=torch.int32, device=DEV)
    pf.basis_build(L, L // 2, st)
    return dim, st


def _col_coeffs(n_b, K, seed):
    """Jackson-damped order-K transforms, each centred at its column's own value of H~."""
    x = np.random.default_rng(seed).uniform(-0.3, 0.3, n_b)
    n = np.arange(K + 1)
    q = math.pi / (K + 2)
    g = ((K + 2 - n) * np.cos(q * n) + np.sin(q * n) / math.tan(q)) / (K + 2)
    c = np.cos(np.outer(np.arccos(x), n)) * g
    c[:, 1:] *= 2.0
    return c / K


def _orders(c, n):
    return [max(1, c["K"] - 7 * (i % 5)) for i in range(n)]


def _rings(c, seed):
    return [_Chain(c["L"] if i % 2 == 0 else c["L2"], "xxz", c["W"], [seed, i]) for i in range(c["n"])]


def _net_params(c, seed):
    r = np.random.default_rng(seed)
    d, H, o = c["d_in"], c["hidden"], 3
    w = [(H, d), (H,), (H, H), (H,), (o, H), (o,)]
    return np.concatenate([(r.uniform(-1, 1, s) * math.sqrt(6.0 / sum(s)) if len(s) == 2 else r.uniform(-0.1, 0.1, s))
                           .astype(np.float32).ravel() for s in w])


def _net_data(c, seed):
    g = _gen(seed)
    x = torch.randn((c["B"], c["d_in"]), generator=g, device=DEV)
    t = torch.randn((c["B"], 3), generator=g, device=DEV)
    return x, t


def _unit_vectors(c, seed):
    """n_vec normalized sector vectors, one per row (column-major dim x n_vec), with the spread of localized states."""
    g = _gen(seed)
    v = torch.randn((c["n_vec"], _dim(c["L"])), generator=g, device=DEV, dtype=torch.float64)
    v = v * torch.exp(2.0 * torch.randn(v.shape, generator=g, device=DEV, dtype=torch.float64))
    return v / v.norm(dim=1, keepdim=True)


def prepare(case, seed):
    c = dict(case)
    s = {"c": c}
    k = c["kind"]
    if k in ("apply", "filter", "cols", "moments"):
        ch = _Chain(c["L"], c["model"], c["W"], seed)
        s["e"] = (ch.e_lo, ch.e_hi) if c.get("scaled", True) else (0.0, 0.0)
        s["m"] = pf.Model.of(ch)
        s["dim"], s["st"] = _basis(c["L"])
        s["X"] = _block(s["dim"], c.get("n_b") or c["R"], seed, c.get("dtype", "f32"))
        if k == "moments":
            s["X"] = s["X"] * math.sqrt(s["dim"])  # unit-variance entries
        else:
            s["Y"] = torch.empty_like(s["X"])
        if k == "cols":
            s["coef"] = _col_coeffs(c["n_b"], c["K"], seed)
    elif k == "batched":
        rings = _rings(c, seed)
        s["m"] = [pf.Model.of(r) for r in rings]
        s["lo"], s["hi"] = [r.e_lo for r in rings], [r.e_hi for r in rings]
        s["X"] = [_block(_dim(r.L), c["n_b"], seed * 100 + i, c["dtype"]) for i, r in enumerate(rings)]
        s["Y"] = [torch.empty_like(x) for x in s["X"]]
        s["K"] = _orders(c, c["n"])
    elif k == "entropy":
        s["ctx"] = pf.Ctx(0)
        s["dim"], s["st"] = _basis(c["L"])
        s["V"] = _unit_vectors(c, seed)
    elif k == "mlp":
        s["net"] = pf.MLP(c["d_in"], c["hidden"], 3)
        s["net"].set_params(_net_params(c, seed))
        s["x"], s["t"] = _net_data(c, seed)
        s["g"] = torch.empty(s["net"].num_params, dtype=torch.float32, device=DEV)
    else:
        s["ctx"] = pf.Ctx(0)
        s["m"] = pf.Model.of(_Chain(c["L"], c["model"], c["W"], seed))
        s["o"] = pf.opts_default()
        s["o"].precision = DTYPES[c["dtype"]]
    torch.cuda.synchronize()
    return s


# --------------------------------------------------------------------- pass
def run(s):
    c = s["c"]
    k = c["kind"]
    if k == "apply":
        pf.h_apply(s["m"], s["st"], s["dim"], s["e"][0], s["e"][1], s["X"], s["Y"], c["n_b"], DTYPES[c["dtype"]])
        return s["Y"]
    if k == "filter":
        pf.cheb_filter(s["m"], s["st"], s["dim"], s["e"][0], s["e"][1], c["sigma"], c["K"], s["X"], s["Y"], c["n_b"],
                       DTYPES[c["dtype"]])
        return s["Y"]
    if k == "cols":
        pf.cheb_filter_cols(s["m"], s["st"], s["dim"], s["e"][0], s["e"][1], s["coef"], s["X"], s["Y"], c["n_b"])
        return s["Y"]
    if k == "batched":
        pf.cheb_filter_batched(s["m"], s["lo"], s["hi"], [0.0] * c["n"], s["K"], s["X"], s["Y"], c["n_b"],
                               DTYPES[c["dtype"]])
        return s["Y"]
    if k == "moments":
        return pf.kpm_moments(s["m"], s["st"], s["dim"], s["e"][0], s["e"][1], c["n_mom"], s["X"], c["R"],
                              DTYPES[c["dtype"]])
    if k == "entropy":
        return pf.entanglement_entropy(s["ctx"], c["L"], s["st"], s["V"], s["dim"], c["n_vec"], per_cut=True)
    if k == "mlp":
        loss = s["net"].grad(s["x"], s["t"], c["B"], s["g"])
        return {"loss": np.float32(loss), "grad": s["g"]}
    # the eigenvectors are converged to a residual of 1e-8 ||H|| and their signs are arbitrary: the
    # eigenvalues are what two correct runs agree on
    ev, _, _, _ = pf.eigs(s["ctx"], s["m"], 0.5, c["N_ev"], 0, c["n_b"], s["o"])
    return ev


# --------------------------------------------------------------------- work
def _apply_flops(L, model, n):
    nb = {"xxz": L, "j1j2": 2 * L, "xxz_open": L - 1}[model]
    return _dim(L) * n * (nb * L / (2.0 * (L - 1)) + 3.0)  # antiparallel bonds, diagonal, scaling


def work(case):
    c = case
    k = c["kind"]
    if k in ("apply", "filter", "cols"):
        es = 4 if c.get("dtype", "f32") == "f32" else 8
        io = 2.0 * _dim(c["L"]) * c["n_b"] * es
        return {"bytes": io, "flops": _apply_flops(c["L"], c["model"], c["n_b"]) * c.get("K", 1)}
    if k == "batched":
        es = 4 if c["dtype"] == "f32" else 8
        Ls = [c["L"] if i % 2 == 0 else c["L2"] for i in range(c["n"])]
        return {"bytes": sum(2.0 * _dim(L) * c["n_b"] * es for L in Ls),
                "flops": sum(_apply_flops(L, "xxz", c["n_b"]) * K for L, K in zip(Ls, _orders(c, c["n"])))}
    if k == "moments":
        es = 4 if c["dtype"] == "f32" else 8
        ap = (c["n_mom"] + 1) // 2
        n = _dim(c["L"]) * c["R"]
        return {"bytes": float(n * es + 8 * c["n_mom"]), "flops": ap * (_apply_flops(c["L"], c["model"], c["R"]) + 6.0 * n)}
    if k == "entropy":
        h = c["L"] // 2
        fl = sum(2.0 * math.comb(h, q) ** 3 + 4.0 / 3.0 * math.comb(h, q) ** 3 for q in range(h + 1))
        return {"bytes": 8.0 * c["n_vec"] * (_dim(c["L"]) + c["L"]), "flops": fl * h * c["n_vec"]}
    if k == "mlp":
        p = c["hidden"] * (c["d_in"] + c["hidden"] + 3)
        return {"bytes": 4.0 * (2 * (p + 2 * c["hidden"] + 3) + c["B"] * (c["d_in"] + 3)), "flops": 6.0 * p * c["B"]}
    # a run needs at least 2 N_ev Lanczos columns through a filter of order about N / N_ev
    n = _dim(c["L"])
    return {"bytes": 8.0 * n * c["N_ev"], "flops": _apply_flops(c["L"], c["model"], 2 * c["N_ev"]) * (n / c["N_ev"])}


# -------------------------------------------------------------------- exact
def _states(L):
    s = torch.arange(1 << L, device=DEV, dtype=torch.int64)
    p = torch.zeros_like(s)
    for i in range(L):
        p += (s >> i) & 1
    return s[p == L // 2]


def _matrix(ch, scaled):
    """Sparse FP64 matrix of H, or of H~ = [2 H - (e_lo + e_hi)] / (e_hi - e_lo), in the S^z = 0 sector."""
    st = _states(ch.L)
    n = st.numel()
    z = [((st >> i) & 1).double() - 0.5 for i in range(ch.L)]
    d = torch.zeros(n, device=DEV, dtype=torch.float64)
    for i in range(ch.L):
        d += float(ch.h[i]) * z[i]
    rows, cols, vals = [], [], []
    ids = torch.arange(n, device=DEV)
    for i, j, J in ch.bonds():
        d += J * ch.Delta * z[i] * z[j]
        r = ids[z[i] != z[j]]
        rows.append(r)
        cols.append(torch.searchsorted(st, st[r] ^ ((1 << i) | (1 << j))))
        vals.append(torch.full((r.numel(),), 0.5 * J, device=DEV, dtype=torch.float64))
    a, b = (2.0 / (ch.e_hi - ch.e_lo), 0.5 * (ch.e_hi + ch.e_lo)) if scaled else (1.0, 0.0)
    rows, cols, vals = torch.cat(rows + [ids]), torch.cat(cols + [ids]), torch.cat(vals + [d - b]) * a
    order = torch.argsort(rows, stable=True)
    crow = torch.zeros(n + 1, device=DEV, dtype=torch.int64)
    crow[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return torch.sparse_csr_tensor(crow.int(), cols[order].int(), vals[order], (n, n))


def _series(H, X, C):
    """sum_n C[:, n] T_n(H) X column by column (C: columns x (K + 1)), by the three-term recurrence."""
    C = torch.as_tensor(C, device=DEV, dtype=torch.float64)
    t0, t1 = X, H @ X
    Y = t0 * C[:, 0] + t1 * C[:, 1]
    for n in range(2, C.shape[1]):
        t0, t1 = t1, 2.0 * (H @ t1) - t0
        if bool((C[:, n] != 0).any()):
            Y = Y + t1 * C[:, n]
    return Y


def _transform(sigma, K):
    """Eq. (2): c_n / D with c_n = sqrt(4 - 3 delta_0n) cos(n arccos sigma), D = sum_n c_n T_n(sigma)."""
    t = np.cos(np.arange(K + 1) * math.acos(sigma))
    if sigma == 0.0:
        t = np.array([(1.0, 0.0, -1.0, 0.0)[n % 4] for n in range(K + 1)])
    c = 2.0 * t
    c[0] = t[0]
    return c / float((c * t).sum())


def exact(case, seed):
    c = dict(case)
    k = c["kind"]
    if k in ("apply", "filter", "cols", "moments"):
        ch = _Chain(c["L"], c["model"], c["W"], seed)
        H = _matrix(ch, c.get("scaled", True))
        n_b = c.get("n_b") or c["R"]
        X = _block(_dim(c["L"]), n_b, seed, c.get("dtype", "f32"))
        if k == "moments":
            X = (X * math.sqrt(_dim(c["L"]))).double()
            mu = np.zeros(c["n_mom"])
            t0, t1 = X, H @ X
            m0, m1 = float((t0 * t0).sum()), float((t0 * t1).sum())
            mu[0], mu[1] = m0, m1
            for j in range(1, (c["n_mom"] + 1) // 2):
                t0, t1 = t1, 2.0 * (H @ t1) - t0
                mu[2 * j] = 2.0 * float((t0 * t0).sum()) - m0
                if 2 * j + 1 < c["n_mom"]:
                    mu[2 * j + 1] = 2.0 * float((t0 * t1).sum()) - m1
            return mu / c["R"]
        X = X.double()
        if k == "apply":
            return H @ X
        C = _col_coeffs(n_b, c["K"], seed) if k == "cols" else np.tile(_transform(c["sigma"], c["K"]), (n_b, 1))
        return _series(H, X, C)
    if k == "batched":
        out = []
        for i, (r, K) in enumerate(zip(_rings(c, seed), _orders(c, c["n"]))):
            X = _block(_dim(r.L), c["n_b"], seed * 100 + i, c["dtype"]).double()
            out.append(_series(_matrix(r, True), X, np.tile(_transform(0.0, K), (c["n_b"], 1))))
        return out
    if k == "entropy":
        L, h = c["L"], c["L"] // 2
        st, V = _states(L), _unit_vectors(c, seed)
        S = np.zeros((c["n_vec"], L))
        for x in range(h):
            rot = ((st >> x) | (st << (L - x))) & ((1 << L) - 1)
            psi = torch.zeros((c["n_vec"], 1 << L), device=DEV, dtype=torch.float64)
            psi[:, rot] = V
            lam = torch.linalg.svdvals(psi.reshape(c["n_vec"], 1 << h, 1 << h).cpu()) ** 2
            e = torch.special.entr(lam).sum(dim=1).numpy()
            S[:, x] = e
            S[:, x + h] = e
        return S
    if k == "mlp":
        p = torch.from_numpy(_net_params(c, seed)).to(DEV).double().requires_grad_(True)
        x, t = (v.double() for v in _net_data(c, seed))
        d, H = c["d_in"], c["hidden"]
        W1, b1, W2, b2, W3, b3 = torch.split(p, [H * d, H, H * H, H, 3 * H, 3])
        a = torch.tanh(x @ W1.view(H, d).T + b1)
        a = torch.tanh(a @ W2.view(H, H).T + b2)
        loss = 0.5 / c["B"] * ((a @ W3.view(3, H).T + b3 - t) ** 2).sum()
        loss.backward()
        return {"loss": float(loss.detach()), "grad": p.grad}
    ch = _Chain(c["L"], c["model"], c["W"], seed)
    w = torch.linalg.eigvalsh(_matrix(ch, False).to_dense())
    target = 0.5 * (w[0] + w[-1])
    near = torch.argsort((w - target).abs())[: c["N_ev"]]
    return torch.sort(w[near]).values.cpu().numpy()
