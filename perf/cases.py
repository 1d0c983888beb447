"""What the performance of this package is measured on: calls of its public entry points over
the sizes, precisions and options that its users run them with.

listed() names the cases, draw() gives more of the same ranges, prepare() makes what a program
has in hand before the call (device arrays, a loaded network), run() is one call, work() the
bytes and operations the call cannot do without, and exact() the same result in plain FP64
torch.  Inputs follow the recipes of paper_1808_06992_gb300/synth.py, drawn on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1808_06992_gb300 import native

DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # The smallest call: one exploratory fit of a table with a few hundred rows, in the
        # library's default precision (FP64).  Launches, allocations and waits are what counts.
        dict(name="lasso_small_fp64", kind="lasso", n=200, p=50, nnz=10, rho=0.0, precision="fp64",
             warm="path", B1=20, B2=10, q=16),
        # An ordinary fit with every parameter left at its default (FP64, path start, 20/20/16).
        dict(name="lasso_mid_fp64", kind="lasso", n=5000, p=400, nnz=20, rho=0.5, precision="fp64",
             warm="path", B1=20, B2=20, q=16),
        # The same call on a large table: the FP64 form's moments, inverse and streamed solves.
        dict(name="lasso_large_fp64", kind="lasso", n=20000, p=1000, nnz=50, rho=0.5, precision="fp64",
             warm="path", B1=20, B2=20, q=16),
        # An ordinary fit in the mixed form at odd sizes, default start: few chains, many short steps.
        dict(name="lasso_mid_mixed", kind="lasso", n=4999, p=301, nnz=15, rho=0.0, precision="mixed",
             warm="path", B1=24, B2=24, q=32),
        # The headline workload: 48 x 48 x 48 on 50000 x 2000, mixed form, all lambdas at once.
        dict(name="lasso_large_mixed", kind="lasso", n=50000, p=2000, nnz=100, rho=0.5, precision="mixed",
             warm="none", B1=48, B2=48, q=48),
        # Many uneven problems in one call (grouped solves), sizes of the batched workload.
        dict(name="batch_mixed", kind="batch", count=24, n_lo=500, n_hi=20000, p_lo=100, p_hi=1500,
             B1=24, B2=24, q=32, sizes=4),
        # A small macro-economic VAR: two lags, an intercept, blocks of rows, FP64.
        dict(name="var_small_fp64", kind="var", p=30, T=1000, order=2, intercept=1, density=0.1, radius=0.8,
             precision="fp64", B1=20, B2=20, q=16, block=20),
        # The 192-channel recording of the paper's real-data section, VAR(1), mixed form.
        dict(name="var_192_mixed", kind="var", p=192, T=5000, order=1, intercept=0, density=0.03, radius=0.9,
             precision="mixed", B1=30, B2=30, q=32, block=100),
        # The same recording with two lags and an intercept (384 regressors per equation).
        dict(name="var2_192_mixed", kind="var", p=192, T=5000, order=2, intercept=1, density=0.02, radius=0.9,
             precision="mixed", B1=20, B2=20, q=16, block=100),
        # A wide VAR with few bootstraps: 500 equations sharing one design of 500 regressors.
        dict(name="var_500_mixed", kind="var", p=500, T=10000, order=1, intercept=0, density=0.01, radius=0.9,
             precision="mixed", B1=8, B2=8, q=16, block=100),
        # The selection solver alone on a caller's weights, several responses, FP64 (the default).
        dict(name="admm_fp64", kind="admm", n=2000, p=150, r=8, nnz=12, B=16, q=16, warm="path"),
        # One gradient of the warm-start network on host rows (its training loop's unit, forward
        # and backward).
        dict(name="warmstart_grad", kind="ws", rows=65536),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lasso64", "lasso32", "lasso32", "batch", "var64", "var32", "var32", "admm", "ws"])
    if kind == "lasso64":
        n, p = _log_int(rng, 200, 20000), _log_int(rng, 40, 1000)
        return dict(kind="lasso", n=n, p=p, nnz=max(3, p // rng.choice([10, 20])), rho=rng.choice([0.0, 0.5]),
                    precision="fp64", warm=rng.choice(["path", "path", "none"]), B1=20, B2=rng.choice([10, 20]), q=16)
    if kind == "lasso32":
        n, p = _log_int(rng, 500, 50000), _log_int(rng, 60, 2000)
        B = rng.choice([20, 24, 48])
        # from a path start a wide problem iterates one chain per bootstrap: such fits stay moderate
        warm = "none" if p > 700 else rng.choice(["path", "none"])
        return dict(kind="lasso", n=n, p=p, nnz=max(3, p // 20), rho=rng.choice([0.0, 0.5]), precision="mixed",
                    warm=warm, B1=B, B2=B, q=rng.choice([16, 32, 48]))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 24), n_lo=1000, n_hi=_log_int(rng, 2000, 20000), p_lo=100,
                    p_hi=_log_int(rng, 250, 1500), B1=24, B2=24, q=32, sizes=rng.randint(0, 1 << 20))
    if kind == "var64":
        return dict(kind="var", p=_log_int(rng, 5, 48), T=_log_int(rng, 300, 4000), order=rng.randint(1, 3),
                    intercept=rng.randint(0, 1), density=0.1, radius=0.8, precision="fp64", B1=20, B2=20, q=16,
                    block=rng.choice([5, 20, 50]))
    if kind == "var32":
        order = rng.choice([1, 1, 2])
        p = _log_int(rng, 40, 400 // order)
        return dict(kind="var", p=p, T=_log_int(rng, 2500, 12000), order=order, intercept=rng.randint(0, 1),
                    density=max(0.01, min(0.1, 6.0 / p)), radius=0.9, precision="mixed", B1=20, B2=20,
                    q=rng.choice([16, 24]), block=100)
    if kind == "admm":
        p = _log_int(rng, 20, 320)
        return dict(kind="admm", n=_log_int(rng, 400, 6000), p=p, r=rng.randint(1, 24), nnz=max(3, p // 12),
                    B=rng.randint(1, 20), q=16, warm=rng.choice(["path", "none"]))
    return dict(kind="ws", rows=_log_int(rng, 2000, 131072))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _lasso_data(n, p, nnz, rho, seed, sigma=None, mag=(0.5, 3.0)):
    """y = X beta + noise, rows N(0, Sigma) with Sigma_ij = rho^|i-j|; signal-to-noise 5 unless sigma is given."""
    g = _gen(seed)
    E = torch.randn((p, n), generator=g, device=DEV, dtype=torch.float64)
    if rho:
        c = math.sqrt(1.0 - rho * rho)
        for j in range(1, p):
            E[j].mul_(c).add_(E[j - 1], alpha=rho)
    X = E.t().contiguous()
    beta = torch.zeros(p, device=DEV, dtype=torch.float64)
    idx = torch.randperm(p, generator=g, device=DEV)[:nnz]
    size = mag[0] + (mag[1] - mag[0]) * torch.rand(nnz, generator=g, device=DEV, dtype=torch.float64)
    sign = torch.randint(0, 2, (nnz,), generator=g, device=DEV).double() * 2 - 1
    beta[idx] = size * sign
    signal = torch.mv(X, beta)
    noise = torch.randn(n, generator=g, device=DEV, dtype=torch.float64)
    y = signal + (signal.std() / math.sqrt(5.0) if sigma is None else sigma) * noise
    return X, y


def _var_data(p, T, order, intercept, density, radius, seed):
    """A stable VAR(order) series, N(0, I) innovations, mean shifted with an intercept."""
    r = np.random.RandomState(seed % (1 << 31))
    nnz = max(1, int(round(density * p * p)))
    A = np.zeros((order, p * p))
    for j in range(order):
        A[j, r.choice(p * p, size=nnz, replace=False)] = r.standard_normal(nnz)
    A = A.reshape(order, p, p)
    comp = np.zeros((order * p, order * p))
    comp[:p] = np.concatenate(list(A), axis=1)
    comp[p:, :-p] = np.eye((order - 1) * p)
    # spectral radius by squarings (the norm of a high power), then lags scaled by c^j
    C = torch.from_numpy(comp).to(DEV)
    log_rad, share = 0.0, 1.0
    for _ in range(8):
        nrm = float(torch.linalg.matrix_norm(C))
        if nrm == 0.0:
            break
        log_rad += share * math.log(nrm)
        share *= 0.5
        C = C / nrm
        C = C @ C
    rad = math.exp(log_rad)
    c = radius / rad
    A *= (c ** np.arange(1, order + 1))[:, None, None]
    comp[:p] = np.concatenate(list(A), axis=1)
    burn = 300
    g = _gen(seed + 1)
    W = torch.zeros((T + burn, order * p), device=DEV, dtype=torch.float64)
    W[:, :p] = torch.randn((T + burn, p), generator=g, device=DEV, dtype=torch.float64)
    # state_t = sum_k C^k w_{t-k}, by doubling
    P = torch.from_numpy(comp).to(DEV)
    k = 1
    while k < T + burn and radius ** k > 1e-12:
        W[k:] += W[:-k] @ P.t()
        P = P @ P
        k *= 2
    S = W[burn:, :p].contiguous()
    if intercept:
        S += torch.randn(p, generator=g, device=DEV, dtype=torch.float64)
    return S


def _batch_sizes(case):
    r = np.random.RandomState(int(case["sizes"]) + 17)
    ns = r.randint(case["n_lo"], case["n_hi"] + 1, size=case["count"])
    ps = r.randint(case["p_lo"], case["p_hi"] + 1, size=case["count"])
    sp = r.uniform(0.02, 0.10, size=case["count"])
    return [(int(n), int(p), max(1, int(round(s * p)))) for n, p, s in zip(ns, ps, sp)]


def _admm_data(case, seed):
    n, p, r, B = case["n"], case["p"], case["r"], case["B"]
    g = _gen(seed)
    X = torch.randn((n, p), generator=g, device=DEV, dtype=torch.float64)
    coef = torch.zeros((p, r), device=DEV, dtype=torch.float64)
    for e in range(r):
        idx = torch.randperm(p, generator=g, device=DEV)[:case["nnz"]]
        coef[idx, e] = torch.randn(case["nnz"], generator=g, device=DEV, dtype=torch.float64) * 2.0
    Y = X @ coef + torch.randn((n, r), generator=g, device=DEV, dtype=torch.float64)
    draws = torch.randint(0, n, (B, n), generator=g, device=DEV)
    w = torch.zeros((B, n), device=DEV, dtype=torch.int32)
    w.scatter_add_(1, draws, torch.ones((B, n), device=DEV, dtype=torch.int32))
    lmax = float((X.t() @ Y).abs().max()) / n
    lam = lmax * 1e-3 ** (torch.arange(case["q"], device=DEV, dtype=torch.float64) / (case["q"] - 1))
    return X, Y, w, lam


WS_SHAPES = [(512, 8), (512,), (512, 512), (512,), (512, 512), (512,), (3, 512), (3,)]


def _ws_data(rows, seed):
    """Feature and target rows with the ranges the warm start meets, and a network's weights."""
    r = np.random.RandomState(seed % (1 << 31))
    pos = r.randint(0, 32, rows) / 31.0
    corr = r.standard_normal(rows)
    diag = r.uniform(0.7, 1.4, rows)
    step = 1e-3 ** (1.0 / 31.0)
    lam = 1e-3 ** pos
    c = np.clip(corr * 0.05 / lam, -50, 50)
    a = np.clip(corr * 0.04 * diag / lam, -50, 50)
    X = np.stack([lam, pos, c, diag, a, np.abs(a), c * step, a * step], axis=1).astype(np.float32)
    active = (np.abs(c) > 1.0).astype(np.float64)
    T = np.stack([np.clip(a * active * 0.5, -4, 4), np.clip(c, -1, 1), active], axis=1).astype(np.float32)
    flat = []
    for sh in WS_SHAPES:
        bound = 1.0 / math.sqrt(sh[-1] if len(sh) > 1 else 512)
        flat.append(r.uniform(-bound, bound, int(np.prod(sh))).astype(np.float32))
    return X, T, np.concatenate(flat)


_PREC = {"fp64": native.PREC_FP64, "mixed": native.PREC_MIXED}
_WARM = {"path": native.WARM_PATH, "none": native.WARM_NONE}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lasso":
        X, y = _lasso_data(case["n"], case["p"], case["nnz"], case["rho"], seed)
        kw = dict(B1=case["B1"], B2=case["B2"], q=case["q"], precision=_PREC[case["precision"]],
                  warm_start=_WARM[case["warm"]])
        return dict(kind=kind, X=X, y=y, kw=kw, family=case["precision"] == "fp64")
    if kind == "batch":
        data = [_lasso_data(n, p, nnz, 0.0, seed * 1000 + i, sigma=1.0, mag=(1.0, 3.0))
                for i, (n, p, nnz) in enumerate(_batch_sizes(case))]
        kw = dict(B1=case["B1"], B2=case["B2"], q=case["q"], precision=native.PREC_MIXED,
                  warm_start=native.WARM_NONE)
        return dict(kind=kind, X=[d[0] for d in data], y=[d[1] for d in data], kw=kw)
    if kind == "var":
        S = _var_data(case["p"], case["T"], case["order"], case["intercept"], case["density"], case["radius"], seed)
        kw = dict(B1=case["B1"], B2=case["B2"], q=case["q"], precision=_PREC[case["precision"]],
                  block_len=case["block"], intercept=case["intercept"])
        return dict(kind=kind, S=S, order=case["order"], kw=kw)
    if kind == "admm":
        X, Y, w, lam = _admm_data(case, seed)
        return dict(kind=kind, X=X, Y=Y, w=w, lam=lam, warm=_WARM[case["warm"]])
    X, T, flat = _ws_data(case["rows"], seed)
    model = native.WarmStartModel(seed=1)
    model.set_params(flat)
    return dict(kind=kind, X=X, T=T, model=model)


def run(state):
    kind = state["kind"]
    if kind == "lasso":
        out = native.uoi_lasso_fit(state["X"], state["y"], family=state["family"], **state["kw"])
        return [out["beta"], out["family"]] if state["family"] else [out["beta"]]
    if kind == "batch":
        return [o["beta"] for o in native.uoi_lasso_fit_batch(state["X"], state["y"], **state["kw"])]
    if kind == "var":
        out = native.uoi_var_fit(state["S"], order=state["order"], **state["kw"])
        return [out["A"], out["mu"]]
    if kind == "admm":
        out = native.lasso_admm_batch(state["X"], state["Y"], state["w"], state["lam"], warm_start=state["warm"])
        return [out["beta"], out["iters"], out["conv"]]
    loss, grad = state["model"].loss_grad(state["X"], state["T"])
    return [loss, grad]


# ---------------------------------------------------------------------------
# what a call cannot do without
# ---------------------------------------------------------------------------
def _fit_flops(m, p, r, B1, B2, q, iters):
    """Moments over the rows a bootstrap touches (about 63 % of them in the selection, half of them
    for training and a fifth for evaluation, on a tenth of the features), one inverse per
    bootstrap, iters x-updates per column, and the support-restricted solves."""
    s = max(1.0, 0.1 * p)
    moments = 2.0 * m * (0.632 * B1 * (p * (p + 1) / 2 + p * r) + 0.7 * B2 * (s * s / 2 + s * r))
    inverse = 1.0 * B1 * float(p) ** 3
    solves = 2.0 * B1 * q * r * iters * float(p) ** 2
    ols = B2 * q * r * s ** 3 / 3
    return moments + inverse + solves + ols


def work(case):
    kind = case["kind"]
    if kind == "lasso":
        n, p = case["n"], case["p"]
        return dict(bytes=8.0 * (n * p + n + p), flops=_fit_flops(n, p, 1, case["B1"], case["B2"], case["q"], 35))
    if kind == "batch":
        total = dict(bytes=0.0, flops=0.0)
        for n, p, _ in _batch_sizes(case):
            total["bytes"] += 8.0 * (n * p + n + p)
            total["flops"] += _fit_flops(n, p, 1, case["B1"], case["B2"], case["q"], 35)
        return total
    if kind == "var":
        m, p, P = case["T"] - case["order"], case["p"], case["p"] * case["order"]
        return dict(bytes=8.0 * (case["T"] * p + p * P + p),
                    flops=_fit_flops(m, P, p, case["B1"], case["B2"], case["q"], 100))
    if kind == "admm":
        n, p, r, B, q = (case[k] for k in ("n", "p", "r", "B", "q"))
        return dict(bytes=8.0 * (n * p + n * r + q) + 4.0 * B * n + 8.0 * B * q * r * p + 5.0 * B * q * r,
                    flops=2.0 * 0.632 * n * B * (p * (p + 1) / 2 + p * r) + 1.0 * B * p ** 3 +
                    2.0 * B * q * r * 30 * p * p)
    N, params = case["rows"], sum(int(np.prod(s)) for s in WS_SHAPES)
    return dict(bytes=4.0 * (11 * N + 2 * params), flops=6.0 * N * (8 * 512 + 2 * 512 * 512 + 3 * 512))


# ---------------------------------------------------------------------------
# the same results in plain FP64
# ---------------------------------------------------------------------------
_U64 = np.uint64


def _mulhi(a, b):
    """High 64 bits of a * b (uint64 arrays or scalars)."""
    m32 = _U64(0xFFFFFFFF)
    a0, a1, b0, b1 = a & m32, a >> _U64(32), b & m32, b >> _U64(32)
    mid = a1 * b0 + ((a0 * b0) >> _U64(32))
    mid2 = a0 * b1 + (mid & m32)
    return a1 * b1 + (mid >> _U64(32)) + (mid2 >> _U64(32))


def _philox(count, k, tag):
    """The first `count` draws of stream (k, tag) of Philox4x64-10 with a zero key."""
    old = np.seterr(over="ignore")
    blocks = (count + 3) // 4
    c = [np.arange(blocks, dtype=_U64), np.full(blocks, k, _U64), np.full(blocks, tag, _U64), np.zeros(blocks, _U64)]
    k0, k1 = _U64(0), _U64(0)
    M0, M1 = _U64(0xD2E7470EE14C6C93), _U64(0xCA5A826395121157)
    for i in range(10):
        if i:
            k0, k1 = k0 + _U64(0x9E3779B97F4A7C15), k1 + _U64(0xBB67AE8584CAA73B)
        h0, l0, h1, l1 = _mulhi(M0, c[0]), M0 * c[0], _mulhi(M1, c[2]), M1 * c[2]
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    np.seterr(**old)
    return np.stack(c, axis=1).reshape(-1)[:count]


def _rows_of(counts, m, L):
    return np.repeat(counts, L)[:m]


def _selection_weights(m, L, k):
    units = -(-m // L)
    pick = _mulhi(_philox(units, k, 1), _U64(units)).astype(np.int64)
    return _rows_of(np.bincount(pick, minlength=units), m, L)


def _estimation_weights(m, L, k, frac=0.8):
    units = -(-m // L)
    pool = int(math.floor(frac * units))
    perm = np.argsort(_philox(units, k, 2), kind="stable")
    train = np.bincount(perm[_mulhi(_philox(pool, k, 3), _U64(pool)).astype(np.int64)], minlength=units)
    held = np.zeros(units, dtype=np.int64)
    held[perm[pool:]] = 1
    return _rows_of(train, m, L), _rows_of(held, m, L)


def _cuda64(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).to(DEV)


def _admm_columns(G, b, nk, lam, warm, rho=1.0, tol=1e-6, cap=1000):
    """Scaled-form ADMM of every (bootstrap, lambda, response): G (B, p, p), b (B, p, r) -> z (B, q, r, p)."""
    B, p, _ = G.shape
    r, q = b.shape[2], lam.numel()
    M = torch.linalg.inv(G / nk[:, None, None] + rho * torch.eye(p, device=DEV, dtype=torch.float64))
    c = torch.bmm(M, b / nk[:, None, None])
    root = math.sqrt(p) * tol

    def solve(z, u, kappa, c):
        live = torch.ones((B, 1, z.shape[2]), device=DEV, dtype=torch.bool)
        for it in range(cap):
            x = c + rho * torch.bmm(M, z - u)
            v = x + u
            zn = torch.sign(v) * torch.clamp(v.abs() - kappa, min=0.0)
            un = v - zn
            pri, dual = (x - zn).norm(dim=1, keepdim=True), rho * (zn - z).norm(dim=1, keepdim=True)
            done = (pri <= root + tol * torch.maximum(x.norm(dim=1, keepdim=True), zn.norm(dim=1, keepdim=True))) & \
                   (dual <= root + tol * rho * un.norm(dim=1, keepdim=True))
            z, u = torch.where(live, zn, z), torch.where(live, un, u)
            live = live & ~done
            if it % 8 == 7 and not bool(live.any()):
                break
        return z, u

    if warm == "none":
        zero = torch.zeros((B, p, q * r), device=DEV, dtype=torch.float64)
        kappa = (lam / rho).repeat_interleave(r)[None, None, :]
        z, _ = solve(zero, zero, kappa, c.repeat(1, 1, q))
        return z.reshape(B, p, q, r).permute(0, 2, 3, 1).contiguous()
    z = u = torch.zeros((B, p, r), device=DEV, dtype=torch.float64)
    out = []
    for j in range(q):
        z, u = solve(z, u, lam[j] / rho, c)
        out.append(z.transpose(1, 2))
    return torch.stack(out, dim=1)


def _moments(X, Y, w):
    wx = X * w[:, None]
    return wx.t() @ X, wx.t() @ Y


def _exact_fit(X, Y, case, L, intercept):
    """Alg. 1 / Alg. 2 of the paper: the bagged coefficients, r x pe (the intercept last)."""
    m, p = X.shape
    r, B1, B2, q, warm = Y.shape[1], case["B1"], case["B2"], case["q"], case.get("warm", "path")
    xbar, ybar = torch.zeros(p, device=DEV, dtype=torch.float64), torch.zeros(r, device=DEV, dtype=torch.float64)
    if intercept:
        xbar, ybar = X.mean(0), Y.mean(0)
        X, Y = X - xbar, Y - ybar
    lmax = (X.t() @ Y).abs().max() / m
    lam = lmax * 1e-3 ** (torch.arange(q, device=DEV, dtype=torch.float64) / max(q - 1, 1))
    G = torch.empty((B1, p, p), device=DEV, dtype=torch.float64)
    b = torch.empty((B1, p, r), device=DEV, dtype=torch.float64)
    nk = torch.empty(B1, device=DEV, dtype=torch.float64)
    for k in range(B1):
        w = _cuda64(_selection_weights(m, L, k))
        Xk, Yk = X, Y
        if intercept:
            Xk, Yk = X - (w @ X) / w.sum(), Y - (w @ Y) / w.sum()
        G[k], b[k] = _moments(Xk, Yk, w)
        nk[k] = w.sum()
    S = (_admm_columns(G, b, nk, lam, warm) != 0).all(dim=0)                   # q x r x p
    if intercept:
        X = torch.cat([X, torch.ones((m, 1), device=DEV, dtype=torch.float64)], dim=1)
        Se = torch.cat([S, torch.ones((q, r, 1), device=DEV, dtype=torch.bool)], dim=2)
    else:
        Se = S
    pe = X.shape[1]
    U = torch.nonzero(Se.reshape(-1, pe).any(dim=0)).reshape(-1)
    chosen = torch.zeros((B2, r, pe), device=DEV, dtype=torch.float64)
    if U.numel():
        Xu, mask = X[:, U], Se[:, :, U].double()
        eye = torch.eye(U.numel(), device=DEV, dtype=torch.float64)
        for k in range(B2):
            wt, we = (_cuda64(v) for v in _estimation_weights(m, L, k))
            Gt, bt = _moments(Xu, Y, wt)
            A = Gt * mask[..., :, None] * mask[..., None, :] + eye * (1 - mask)[..., None]
            sol = torch.linalg.solve(A, (bt.t()[None] * mask)[..., None])[..., 0]    # q x r x U
            held = torch.nonzero(we).reshape(-1)
            res = Y[held].t()[None] - torch.matmul(sol, Xu[held].t())
            j = int(np.argmin(res.square().sum(dim=(1, 2)).cpu().numpy()))
            chosen[k][:, U] = sol[j]
    if intercept:
        chosen[:, :, p] += ybar - chosen[:, :, :p] @ xbar
    v = torch.sort(chosen, dim=0).values
    beta = v[B2 // 2] if B2 % 2 else 0.5 * (v[B2 // 2 - 1] + v[B2 // 2])
    return beta


def _exact_ws(case, seed):
    X, T, flat = _ws_data(case["rows"], seed)
    at, ps = 0, []
    for sh in WS_SHAPES:
        k = int(np.prod(sh))
        ps.append(_cuda64(flat[at:at + k].reshape(sh)).requires_grad_(True))
        at += k
    h, t = _cuda64(X), _cuda64(T)
    for i in range(0, 6, 2):
        h = torch.nn.functional.gelu(torch.nn.functional.linear(h, ps[i], ps[i + 1]))
    o = torch.nn.functional.linear(h, ps[6], ps[7])
    loss = ((o[:, 0] - t[:, 0]) ** 2 + (o[:, 1] - t[:, 1]) ** 2 + torch.nn.functional.softplus(o[:, 2]) -
            t[:, 2] * o[:, 2]).mean()
    loss.backward()
    return [float(loss), torch.cat([v.grad.reshape(-1) for v in ps])]


def exact(case, seed):
    kind = case["kind"]
    if kind == "ws":
        return _exact_ws(case, seed)
    if kind == "admm":
        X, Y, w, lam = _admm_data(case, seed)
        wd = w.double()
        G, b = zip(*(_moments(X, Y, wd[k]) for k in range(case["B"])))
        return [_admm_columns(torch.stack(G), torch.stack(b), wd.sum(1), lam, case["warm"]), None, None]
    if kind == "lasso":
        n, p, B1, B2, q = (case[k] for k in ("n", "p", "B1", "B2", "q"))
        # plain FP64 products at about a teraflop a second, and hundreds of dependent steps
        cost = 2.0 * n * p * p * (B1 + B2) + 16.0 * B1 * p ** 3 + 60.0 * q * 2 * B1 * p * p * (q if case["warm"] == "none" else 1)
        if cost > 4e12:
            return None
        X, y = _lasso_data(n, p, case["nnz"], case["rho"], seed)
        beta = _exact_fit(X, y.reshape(-1, 1), case, 1, 0)
        return [beta[0], None] if case["precision"] == "fp64" else [beta[0]]
    if kind == "var" and case["p"] * case["order"] <= 144 and case["precision"] == "fp64":
        S = _var_data(case["p"], case["T"], case["order"], case["intercept"], case["density"], case["radius"], seed)
        d, p = case["order"], case["p"]
        N = S.shape[0]
        X = torch.cat([S[d - j:N - j] for j in range(1, d + 1)], dim=1)
        beta = _exact_fit(X, S[d:], case, case["block"], case["intercept"])
        A = beta[:, :d * p].reshape(p, d, p).permute(1, 0, 2).contiguous()
        return [A, beta[:, d * p] if case["intercept"] else torch.zeros(p, device=DEV, dtype=torch.float64)]
    return None
