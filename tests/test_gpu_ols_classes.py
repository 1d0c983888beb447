"""Support-restricted OLS of the estimation stage at the edges of its size classes (a warp up
to 32 columns, register tiles up to 64 and 128, a blocked factor above), against least
squares in extended precision on the traced samples; the chosen lambda and the median over
the bootstraps against their definitions."""
import numpy as np
import pytest

from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def solve_ld(A, b):
    """Cholesky solution in 80-bit arithmetic."""
    A, b = A.astype(np.longdouble), b.astype(np.longdouble)
    s = len(b)
    L = np.zeros_like(A)
    for c in range(s):
        L[c, c] = np.sqrt(A[c, c] - L[c, :c] @ L[c, :c])
        L[c + 1:, c] = (A[c + 1:, c] - L[c + 1:, :c] @ L[c, :c]) / L[c, c]
    y = np.zeros_like(b)
    for i in range(s):
        y[i] = (b[i] - L[i, :i] @ y[:i]) / L[i, i]
    for i in range(s - 1, -1, -1):
        y[i] = (y[i] - L[i + 1:, i] @ y[i + 1:]) / L[i, i]
    return y


@pytest.mark.parametrize("B2", [1, 4, 33])
@pytest.mark.parametrize("p", [1, 31, 32, 33, 64, 65, 128, 129])
def test_supports_of_every_class(p, B2):
    """One tiny lambda keeps all p columns, one of 10 keeps none.  Columns scaled by 1 to 4:
    the moments' condition number stays below 200, so FP64 moments with errors of n 2^-53
    leave the solution within 200 * 600 * 2^-53 < 1.4e-11 relative."""
    g = np.random.default_rng(p)
    n = 600
    X = g.standard_normal((n, p)) * 2.0 ** g.integers(0, 3, p)
    y = X @ g.uniform(1.0, 2.0, p) + 0.1 * g.standard_normal(n)
    out = native.uoi_fit_traced(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), B1=1, B2=B2, q=2,
                                lambdas=torch.tensor([1e6, 1e-7], dtype=torch.float64).cuda(), seed=p)
    a = {k: (v.cpu().numpy() if hasattr(v, "cpu") else v) for k, v in out.items()}
    fam = np.unpackbits(a["family"].reshape(2, -1).view(np.uint8), axis=1, bitorder="little")[:, :p].astype(bool)
    assert not fam[0].any() and fam[1].all()
    assert (a["est_singular"] == 0).all()
    beta = a["est_beta"].reshape(B2, p)
    for k in {0, B2 - 1}:
        w, ev = a["est_weights"][k].astype(np.int64), a["est_eval"][k].astype(bool)
        assert a["est_jstar"][k] == 1
        ref = solve_ld((X * w[:, None]).T @ X, (X * w[:, None]).T @ y)
        assert np.abs(beta[k] - ref).max() <= 1.4e-11 * np.abs(ref).max()
        loss = float(((y[ev] - X[ev] @ ref.astype(float)) ** 2).sum())
        yy = float((y[ev] ** 2).sum())
        assert abs(a["est_loss"][k, 1, 0] - loss) <= 1e-12 * 600 * yy   # a difference of sums of yy's size
        assert abs(a["est_loss"][k, 0, 0] - yy) <= 600 * 2.0 ** -52 * yy
    np.testing.assert_array_equal(a["beta"].reshape(p), np.median(beta, axis=0))
