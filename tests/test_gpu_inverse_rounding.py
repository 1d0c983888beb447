"""The triangular inverse behind the FP64 factor divides: on 2 x 2 systems with an integer factor
every operation is known, and the inverse's entry below the diagonal has the bits of
(b (1 / a)) / c (1 / c)."""
import numpy as np
import pytest

from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# L = [[a, 0], [b, c]] where the product with 1 / c rounds otherwise than the division by c
@pytest.mark.parametrize("a,b,c", [(5, 3, 3), (8, 7, 3)])
def test_division_by_the_diagonal(a, b, c):
    # G / n + I = L L^T from rows 8 e1, 8 e2, 8 (e1 + e2) and zeros, n = 2^12
    n, A = 1 << 12, np.array([[a * a, a * b], [a * b, b * b + c * c]]) - np.eye(2, dtype=int)
    w = [n // 64 * (A[0, 0] - A[0, 1]), n // 64 * (A[1, 1] - A[0, 1]), n // 64 * A[0, 1]]
    w.append(n - sum(w))
    assert min(w) >= 0 and w[1] & (w[1] - 1) == 0
    X = 8.0 * np.array([[1, 0], [0, 1], [1, 1], [0, 0]])
    y = np.array([[0.0], [1.0], [0.0], [0.0]])          # X^T W y = (0, 8 w_1)
    out = native.lasso_admm_batch(*(torch.from_numpy(v).cuda() for v in (X, y, np.array([w], dtype=np.int32),
                                                                         np.array([1e-280]))), max_iter=1)
    z = out["beta"].cpu().numpy().reshape(2)
    below = -((b * (1.0 / a)) / c)
    assert z[0] == below * (1.0 / c) * (8.0 * w[1] / n)
