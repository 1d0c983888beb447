"""The FP64 inverse of G/n + rho I by Newton steps from an FP32 inverse (p >= 64), seen through
the first ADMM step at a vanishing lambda, z = M b / n, against 80-bit arithmetic: tile and
chunk edges, columns of very different scales, and systems it must leave to the factor."""
import numpy as np
import pytest

from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def first_step(X, y, w, rho):
    out = native.lasso_admm_batch(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(),
                                  torch.from_numpy(w.astype(np.int32)).cuda(),
                                  torch.tensor([1e-280], dtype=torch.float64).cuda(), rho=rho, max_iter=1)
    z = out[0] if isinstance(out, tuple) else out["beta"]
    return z.cpu().numpy().reshape(len(w), -1)


def solve_ld(A, b):
    L = np.zeros_like(A)
    for c in range(len(b)):
        L[c, c] = np.sqrt(A[c, c] - L[c, :c] @ L[c, :c])
        L[c + 1:, c] = (A[c + 1:, c] - L[c + 1:, :c] @ L[c, :c]) / L[c, c]
    x = b.copy()
    for i in range(len(b)):
        x[i] = (x[i] - L[i, :i] @ x[:i]) / L[i, i]
    for i in range(len(b) - 1, -1, -1):
        x[i] = (x[i] - L[i + 1:, i] @ x[i + 1:]) / L[i, i]
    return x


@pytest.mark.parametrize("spread,rho", [(0, 1.0), (0, 1e-4), (15, 1e-2)])
@pytest.mark.parametrize("p", [63, 64, 65, 127, 129, 193, 256, 300])
def test_first_step(p, spread, rho):
    """In the scaling that makes the diagonal 1 the moments are off by n 2^-53, a factor by
    p 2^-53, and the solution by their sum times the condition number (2-norm)."""
    g = np.random.default_rng(p)
    n = 2 * p + 50
    X = g.standard_normal((n, p)) * 2.0 ** g.integers(-spread, spread + 1, p)
    y = (X / np.abs(X).max(axis=0)) @ g.uniform(1.0, 2.0, p) + 0.1 * g.standard_normal(n)
    w = g.multinomial(n, np.full(n, 1.0 / n), size=3).astype(np.uint32)
    z = first_step(X, y, w, rho)
    for k in (0, 2):
        Xl, wl = X.astype(np.longdouble), w[k].astype(np.longdouble)[:, None]
        A = (Xl * wl).T @ Xl / n + np.longdouble(rho) * np.eye(p, dtype=np.longdouble)
        ref = solve_ld(A, (Xl * wl).T @ y.astype(np.longdouble) / n)
        d = np.sqrt(np.diag(A))
        cond = float(np.linalg.cond((A / d[:, None] / d[None, :]).astype(float)))
        err = np.linalg.norm(((z[k] - ref) * d).astype(float)) / np.linalg.norm((ref * d).astype(float))
        assert err <= (n + p) * 2.0 ** -53 * cond


def test_near_singular_systems_take_the_factor():
    """Every column twice and rho = 1e-9: no FP32 inverse.  On integer data both forms of the
    moments are exact, so the factor must give the bits of the no-allocation entry point,
    which has no other path."""
    g = np.random.default_rng(5)
    n, p = 400, 128
    H = g.integers(-9, 10, (n, p // 2)).astype(np.float64)
    X = np.concatenate([H, H], axis=1)
    y = g.integers(-9, 10, n).astype(np.float64)
    args = [torch.from_numpy(a).cuda() for a in (X, y.reshape(-1, 1), np.ones((1, n), dtype=np.int32),
                                                 np.array([1e-280]))]
    plain = native.lasso_admm_batch_noalloc(*args, rho=1e-9, max_iter=1)
    plain = plain[0] if isinstance(plain, tuple) else plain["beta"]
    z = first_step(X, y, np.ones((1, n), dtype=np.uint32), 1e-9)[0]
    np.testing.assert_array_equal(z, plain.cpu().numpy().reshape(-1))
