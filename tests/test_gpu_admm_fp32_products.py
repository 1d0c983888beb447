"""FP32 chains with many responses: M's diagonal meets V in FP32, whichever kernel runs.  On the columns of
a Hadamard matrix M is 1/2 on the diagonal and zero beside it, exactly, so the iterates are those of
plain FP32 arithmetic, bit for bit (a split of V into two 11-bit pieces would not give them)."""
import numpy as np
import pytest

from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

F = np.float32


def iterates(c, kappa, steps, resident):
    """Path start over the thresholds; c: r x p."""
    z, u, out = np.zeros_like(c), np.zeros_like(c), []
    for k in kappa:
        for _ in range(steps):
            x = c + F(0.5) * (z - u)
            v = x + u
            if resident:                                 # z by the soft threshold, u what is left
                z = np.where(v > k, v - k, np.where(v < -k, v + k, F(0)))
                u = v - z
            else:                                        # u by the clamp
                u = np.minimum(np.maximum(v, -k), k)
                z = v - u
        out.append(z)
    return np.stack(out)


@pytest.mark.parametrize("p,r", [(1, 40), (33, 40), (64, 40), (65, 9), (96, 130), (128, 40), (161, 40), (192, 130)])
def test_iterates_are_those_of_fp32_arithmetic(p, r):
    n, steps = 256, 7
    H = np.ones((1, 1))
    while len(H) < n:
        H = np.block([[H, H], [H, -H]])
    g = np.random.default_rng(p)
    X = np.ascontiguousarray(H[:, g.permutation(n)[:p]])
    Y = g.integers(-40, 41, (n, r)).astype(np.float64)
    lam = np.array([1.3, 0.7, 0.05])
    w = torch.ones((3, n), dtype=torch.int32).cuda()
    out = native.lasso_admm_batch(*(torch.from_numpy(a).cuda() for a in (X, Y)), w, torch.from_numpy(lam).cuda(),
                                  precision=native.PREC_MIXED, max_iter=steps, abs_tol=0.0, rel_tol=0.0)
    assert (out["iters"].cpu().numpy() == steps).all()
    c = (0.5 * (X.T @ Y).T / n).astype(F)                  # exact
    want = iterates(c, lam.astype(F), steps, p <= 64)
    got = out["beta"].cpu().numpy()
    for k in range(3):
        np.testing.assert_array_equal(got[k], want.astype(np.float64))
