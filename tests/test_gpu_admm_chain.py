"""The chain schedule of the ADMM (one cluster per chain) against the oracle, at the sizes
where its layout changes: rows that end inside a 16-row block, M in shared memory and
streamed, one CTA and clusters, one and four chains per cluster."""
import numpy as np
import pytest

import mixed_check
import oracle
from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def problem(n, p, r, B, q, seed):
    g = np.random.default_rng(seed)
    X = g.standard_normal((n, p))
    coef = np.zeros((p, r))
    for e in range(r):
        coef[g.choice(p, size=min(p, 6), replace=False), e] = g.uniform(0.5, 2.0, size=min(p, 6))
    Y = X @ coef + g.standard_normal((n, r))
    w = np.stack([np.bincount(g.integers(0, n, n), minlength=n) for _ in range(B)]).astype(np.uint32)
    lam = np.abs(X.T @ Y).max() / n * 1e-2 ** (np.arange(q) / max(q - 1, 1))
    return X, Y, w, lam


# (p, r, B, warm): one row; block edges; the largest M in shared memory and the first
# streamed one; clusters of 2 to 6; four chains per cluster with fewer chains than slots at the end
FP64 = [(1, 1, 1, 1), (16, 1, 3, 1), (17, 2, 2, 0), (63, 3, 4, 1), (97, 1, 20, 1), (129, 8, 20, 1),
        (160, 2, 2, 0), (176, 8, 20, 1), (209, 6, 30, 1), (257, 1, 9, 1), (400, 1, 20, 1)]


@pytest.mark.parametrize("p,r,B,warm", FP64)
def test_fp64_chain_follows_the_oracle(p, r, B, warm):
    X, Y, w, lam = problem(max(60, 2 * p), p, r, B, 3, 100 + p)
    gpu = native.lasso_admm_batch(X, Y, w, lam, warm_start=warm)
    ks = sorted({0, B // 2, B - 1})
    es = sorted({0, r - 1})
    ref = oracle.lasso_admm_batch(X, Y, w[ks], lam, warm_start=warm, eq_list=es)
    np.testing.assert_array_equal(gpu["iters"][ks][:, :, es], ref["iters"])
    np.testing.assert_array_equal(gpu["conv"][ks][:, :, es].astype(bool), ref["conv"])
    z, zr = gpu["beta"][ks][:, :, es], ref["beta"]
    edge = np.abs(np.abs(ref["v"]) - lam[None, :, None, None]) <= 1e-6
    assert not (((z != 0) != (zr != 0)) & ~edge).any()
    # the bar of the other FP64 parity tests (relative l2 per column)
    assert np.linalg.norm(z - zr, axis=-1).max() <= 1e-6 * np.linalg.norm(zr, axis=-1).max()


@pytest.mark.parametrize("max_iter", [1, 5])
def test_fp64_chain_iteration_cap(max_iter):
    X, Y, w, lam = problem(200, 70, 2, 4, 3, 9)
    gpu = native.lasso_admm_batch(X, Y, w, lam, max_iter=max_iter)
    ref = oracle.lasso_admm_batch(X, Y, w, lam, max_iter=max_iter)
    np.testing.assert_array_equal(gpu["iters"], ref["iters"])
    np.testing.assert_array_equal(gpu["conv"].astype(bool), ref["conv"])
    assert np.abs(gpu["beta"] - ref["beta"]).max() <= 1e-12


# FP32: one CTA, a cluster whose last CTA is short, the largest cluster, and past it
@pytest.mark.parametrize("p,r,B", [(33, 1, 3), (193, 1, 8), (301, 2, 8), (500, 4, 3), (641, 1, 3)])
def test_fp32_chain_meets_the_stopping_bound(p, r, B):
    X, Y, w, lam = problem(3 * p, p, r, B, 3, 300 + p)
    gpu = native.lasso_admm_batch(X, Y, w, lam, precision=native.PREC_MIXED)
    assert gpu["conv"].all()
    mixed_check.check_residuals(X, Y, w, lam, gpu["beta"], mixed_check.ETA_MIXED)
