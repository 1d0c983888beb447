"""ADMM calls at the rarer ends of the schedules' ranges: more thresholds than shared memory keeps, a
response that is zero, and many FP64 chains past the size where four of them share a read of M."""
import numpy as np
import pytest

import mixed_check
import oracle
from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def problem(n, p, r, B, seed):
    g = np.random.default_rng(seed)
    X = g.standard_normal((n, p))
    k = min(p, 5)
    Y = X[:, :k] @ g.uniform(0.5, 2.0, (k, r)) + g.standard_normal((n, r))
    w = g.multinomial(n, np.full(n, 1.0 / n), size=B).astype(np.uint32)
    return X, Y, w, np.abs(X.T @ Y).max() / n


@pytest.mark.parametrize("p,r,warm", [(20, 6, 1), (70, 2, 1), (70, 6, 0), (96, 6, 1)])
def test_three_hundred_thresholds(p, r, warm):
    X, Y, w, top = problem(300, p, r, 2, p)
    lam = top * 1e-2 ** (np.arange(300) / 299)
    gpu = native.lasso_admm_batch(X, Y, w, lam, warm_start=warm)
    ref = oracle.lasso_admm_batch(X, Y, w, lam, warm_start=warm)
    np.testing.assert_array_equal(gpu["iters"], ref["iters"])
    assert np.linalg.norm(gpu["beta"] - ref["beta"], axis=-1).max() <= 1e-6 * np.linalg.norm(ref["beta"], axis=-1).max()
    mixed = native.lasso_admm_batch(X, Y, w, lam, warm_start=warm, precision=native.PREC_MIXED)
    assert mixed["conv"].all()
    mixed_check.check_residuals(X, Y, w, lam, mixed["beta"], mixed_check.ETA_MIXED)


@pytest.mark.parametrize("prec", [native.PREC_FP64, native.PREC_MIXED])
@pytest.mark.parametrize("p,r", [(40, 1), (40, 9), (130, 9)])
def test_a_zero_response_stays_zero(p, r, prec):
    X, Y, w, top = problem(400, p, r, 3, p + r)
    Y[:, r // 2] = 0.0
    lam = top * np.array([1.0, 0.1])
    out = native.lasso_admm_batch(X, Y, w, lam, precision=prec)
    assert (out["beta"][:, :, r // 2] == 0).all() and out["conv"].all() and np.isfinite(out["beta"]).all()
    assert (out["iters"][:, :, r // 2] == 1).all()


def test_many_chains_of_a_wide_fp64_problem():
    X, Y, w, top = problem(1700, 1600, 5, 1, 7)
    lam = top * np.array([0.5, 0.1])
    gpu = native.lasso_admm_batch(X, Y, w, lam, max_iter=8, abs_tol=0.0, rel_tol=0.0)
    ref = oracle.lasso_admm_batch(X, Y, w, lam, max_iter=8, abs_tol=0.0, rel_tol=0.0, eq_list=[0, 4])
    z = gpu["beta"][:, :, [0, 4]]
    assert np.linalg.norm(z - ref["beta"], axis=-1).max() <= 1e-9 * np.linalg.norm(ref["beta"], axis=-1).max()
