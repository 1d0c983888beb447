"""FP64 ADMM iterates on designs whose columns differ in scale by up to 2^30, against 80-bit
arithmetic over several steps: every layout of the chain schedule (M in shared memory and streamed, one
CTA and clusters, one and four chains) and the schedule past it.  Integer data times powers of two and
a power of two of rows: the moments are exact."""
import numpy as np
import pytest

from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

STEPS, RHO = 6, 1e-2


def cholesky_ld(A):
    L = np.zeros_like(A)
    for c in range(len(A)):
        L[c, c] = np.sqrt(A[c, c] - L[c, :c] @ L[c, :c])
        L[c + 1:, c] = (A[c + 1:, c] - L[c + 1:, :c] @ L[c, :c]) / L[c, c]
    return L


def solve_factored(L, b):
    x = b.copy()
    for i in range(len(b)):
        x[i] = (x[i] - L[i, :i] @ x[:i]) / L[i, i]
    for i in range(len(b) - 1, -1, -1):
        x[i] = (x[i] - L[i + 1:, i] @ x[i + 1:]) / L[i, i]
    return x


def problem(p, r, spread, seed):
    g = np.random.default_rng(seed)
    n = 64
    while n < 2 * p:
        n *= 2
    e = g.integers(-spread, spread + 1, p)
    H = g.integers(-9, 10, (n, p)).astype(np.float64)
    Y = np.rint(H @ g.uniform(-1.0, 1.0, (p, r))) + g.integers(-20, 21, (n, r))
    return np.ldexp(H, e), Y, n


# M in shared memory: one row, one CTA, a cluster; streamed: four chains, one chain in a cluster
LAYOUTS = [(1, 1, 1), (24, 2, 2), (63, 1, 200), (160, 2, 100), (209, 6, 30), (400, 1, 6), (500, 1, 3)]


@pytest.mark.parametrize("spread", [0, 3, 15])
@pytest.mark.parametrize("p,r,B", LAYOUTS)
def test_every_feature_keeps_its_bits(p, r, B, spread):
    """In the scaling that makes the diagonal of A = G / n + rho I one, M is off by p 2^-53, and
    each step by a rounding of (p + 4) 2^-53 of the largest term, both times the condition number;
    the steps' errors add up (x = c + rho M (z - u) with 0 <= rho M <= I, then two projections)."""
    X, Y, n = problem(p, r, spread, p + spread)
    lam = np.array([2.0 ** -12, 2.0 ** -40])
    w = torch.ones((B, n), dtype=torch.int32).cuda()
    out = native.lasso_admm_batch(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(), w, torch.from_numpy(lam).cuda(),
                                  rho=RHO, abs_tol=0.0, rel_tol=0.0, max_iter=STEPS)
    beta = out["beta"].cpu().numpy()
    assert (out["iters"].cpu().numpy() == STEPS).all()
    A = (X.T @ X / n).astype(np.longdouble) + np.longdouble(RHO) * np.eye(p, dtype=np.longdouble)
    L = cholesky_ld(A)
    d = np.sqrt(np.diag(A))
    cond = float(np.linalg.cond((A / d[:, None] / d[None, :]).astype(float)))
    for e in {0, r - 1}:
        b = (X.T @ Y[:, e] / n).astype(np.longdouble)
        z = u = np.zeros(p, dtype=np.longdouble)
        for j, lm in enumerate(lam):
            kappa = np.longdouble(lm) / np.longdouble(RHO)
            big = np.longdouble(0)
            for _ in range(STEPS):
                x = solve_factored(L, b + np.longdouble(RHO) * (z - u))
                v = x + u
                z = np.sign(v) * np.maximum(np.abs(v) - kappa, 0)
                u = v - z
                big = max(big, np.abs(x * d).max(), np.abs((z - u) * RHO / d).max())
            tol = (j + 1) * STEPS * 2 * (p + 4) * 2.0 ** -53 * cond * float(big) * np.sqrt(p)
            for k in {0, B - 1}:
                assert np.linalg.norm(((beta[k, j, e] - z) * d).astype(float)) <= tol
