"""Support-restricted OLS of up to 128 columns on designs whose columns differ in scale, against
80-bit arithmetic.  Integer data times powers of two: the moments are exact, so all of the error is
the solve's."""
import numpy as np
import pytest

from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def solve_ld(A, b):
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


def exponent(d):
    return (np.frexp(d)[1] + 1) >> 1


@pytest.mark.parametrize("yscale", [0, -300, 300])
@pytest.mark.parametrize("s", [24, 32, 33, 64, 100, 128])
def test_small_columns_keep_their_bits(s, yscale):
    """Half of the columns are 2^-4 as large (pivots 2^-8 of the largest: still the FP32 inverse and
    its refinement), the response 2^yscale.  In the scaling that brings G's diagonal to
    [1/4, 1), the residual's integers of `bits` bits carry independent roundings of G's entries
    and of x (uniform, 2^-bits wide).  1.5 times their 2-norm, through the inverse, is the bound;
    beside it the rounding of x."""
    g = np.random.default_rng(s)
    n = 600
    X = np.ldexp(g.integers(-9, 10, (n, s)).astype(np.float64), -4 * g.integers(0, 2, s))
    y = np.ldexp(g.integers(-50, 51, n) + np.rint(X @ g.uniform(1.0, 2.0, s)), yscale)
    lam = np.ldexp(np.array([1e6, 1e-7]), yscale)
    out = native.uoi_fit_traced(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), B1=1, B2=3, q=2,
                                lambdas=torch.from_numpy(lam).cuda(), seed=s)
    a = {k: (v.cpu().numpy() if hasattr(v, "cpu") else v) for k, v in out.items()}
    fam = np.unpackbits(a["family"].reshape(2, -1).view(np.uint8), axis=1, bitorder="little")[:, :s].astype(bool)
    assert fam[1].all() and (a["est_singular"] == 0).all() and (a["est_jstar"] == 1).all()
    bits = 57 if s <= 32 else 58 if s <= 64 else 56
    for k in range(3):
        w = a["est_weights"][k].astype(np.int64)
        G, b = (X * w[:, None]).T @ X, (X * w[:, None]).T @ y
        ref = solve_ld(G, np.ldexp(b, -yscale))                # over 2^yscale
        e = exponent(np.diag(G))
        Gh = np.ldexp(G, -(e[:, None] + e[None, :]))
        xh = np.ldexp(ref, e)
        err = np.ldexp(np.ldexp(a["est_beta"][k].reshape(s), -yscale) - ref, e)
        rnd = 2.0 ** -bits / np.sqrt(12.0)
        row = np.sqrt(s + 1) * rnd
        bound = 1.5 * np.sqrt(s) * row * np.abs(xh).max() / np.linalg.eigvalsh(Gh)[0] + 2.0 ** -53 * np.linalg.norm(xh.astype(float))
        assert float(np.linalg.norm(err.astype(float))) <= bound
