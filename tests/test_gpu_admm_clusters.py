"""The chain schedule's clusters at their start.  Rank 0 of a cluster hands the first chain to the
other CTAs by stores into their shared memory, which those must have reached by then."""
import numpy as np
import pytest

from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# clusters of 2, 6 and 8 CTAs; M in shared memory and streamed (there rank 0 is quickest)
@pytest.mark.parametrize("p,B", [(70, 2), (400, 20), (700, 8)])
def test_every_launch_gives_the_first_ones_columns(p, B):
    g = np.random.default_rng(50 + p)
    n = 2 * p
    X = g.standard_normal((n, p))
    y = X[:, :5] @ g.uniform(0.5, 2.0, 5) + g.standard_normal(n)
    w = g.multinomial(n, np.full(n, 1.0 / n), size=B).astype(np.int32)
    lam = np.abs(X.T @ y).max() / n * np.array([1.0, 0.1])
    X, y, w, lam = (torch.from_numpy(a).cuda() for a in (X, y.reshape(-1, 1), w, lam))
    first = native.lasso_admm_batch(X, y, w, lam, max_iter=3)
    for _ in range(50):
        again = native.lasso_admm_batch(X, y.clone(), w, lam, max_iter=3)
        assert torch.equal(first["beta"], again["beta"]) and torch.equal(first["iters"], again["iters"])
