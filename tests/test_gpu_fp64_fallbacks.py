"""The FP64 forms that few calls reach, at the edges of their tiles: the ADMM schedule of p past 5000
(one launch per iteration) against the oracle, and the CUDA-core moments (inputs that the slicing does
not take, devices without memory for it) against 80-bit sums."""
import numpy as np
import pytest

import oracle
from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture
def streaming():
    native.selftest_admm_streaming(True)
    yield
    native.selftest_admm_streaming(False)


# rows per warp group (8) and per tile (128), chains per tile (64), few chains (4) and more
@pytest.mark.parametrize("p,r,B,warm", [(1, 1, 2, 1), (7, 1, 3, 1), (9, 4, 2, 0), (33, 2, 2, 1), (127, 5, 2, 1), (128, 3, 1, 0),
                                        (129, 65, 1, 1), (200, 22, 2, 0)])
def test_streaming_schedule_follows_the_oracle(p, r, B, warm, streaming):
    g = np.random.default_rng(900 + p)
    n = max(60, 2 * p)
    X = g.standard_normal((n, p))
    Y = X[:, : min(p, 5)] @ g.uniform(0.5, 2.0, (min(p, 5), r)) + g.standard_normal((n, r))
    w = g.multinomial(n, np.full(n, 1.0 / n), size=B).astype(np.uint32)
    lam = np.abs(X.T @ Y).max() / n * np.array([1.0, 0.1, 0.01])
    gpu = native.lasso_admm_batch(X, Y, w, lam, warm_start=warm)
    ref = oracle.lasso_admm_batch(X, Y, w, lam, warm_start=warm)
    np.testing.assert_array_equal(gpu["iters"], ref["iters"])
    np.testing.assert_array_equal(gpu["conv"].astype(bool), ref["conv"])
    z, zr = gpu["beta"], ref["beta"]
    edge = np.abs(np.abs(ref["v"]) - lam[None, :, None, None]) <= 1e-6
    assert not (((z != 0) != (zr != 0)) & ~edge).any()
    # the bar of the other FP64 parity tests (relative l2 per column)
    assert np.linalg.norm(z - zr, axis=-1).max() <= 1e-6 * np.linalg.norm(zr, axis=-1).max()


@pytest.mark.parametrize("n,p,r,B", [(1, 1, 1, 1), (7, 63, 1, 2), (65, 64, 3, 1), (200, 65, 64, 2), (300, 129, 65, 2)])
def test_plain_moments(n, p, r, B):
    g = np.random.default_rng(n + p)
    X, Y = g.standard_normal((n, p)), g.standard_normal((n, r))
    w = g.integers(0, 4, (B, n))
    args = [torch.from_numpy(a).cuda() for a in (X, Y, w.astype(np.int32))]
    native.selftest_alloc_limit(8)                       # nothing for the slicing
    try:
        G, Bm = (a.cpu().numpy() for a in native.weighted_moments(*args))
    finally:
        native.selftest_alloc_limit(0)
    Z = np.concatenate([X, Y], axis=1).astype(np.longdouble)
    for k in range(B):
        wz = Z * w[k].astype(np.longdouble)[:, None]
        got = np.concatenate([G[k], Bm[k]], axis=1)
        # sums of n products in FP64: n 2^-53 of the sum of their magnitudes (and one for the weight)
        assert (np.abs(got - (wz.T @ Z)[:p]) <= (n + 1) * 2.0 ** -53 * (np.abs(wz).T @ np.abs(Z))[:p]).all()
