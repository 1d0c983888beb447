"""The one-launch tensor-core ADMM (many FP32 chains, p <= 512) against what the stopping
rule guarantees (mixed_check), at the sizes where its layout changes: one to four 128-k
accumulators, clusters of one to eight, a last k block and a last 128-chain tile that are
not full, more chains than the device holds at once, cold and path starts."""
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


SIZES = [(9, 6, 1, 3, 1), (32, 5, 2, 4, 0), (33, 129, 2, 2, 1), (97, 16, 1, 9, 0), (128, 40, 3, 2, 1),
         (193, 7, 2, 3, 1), (257, 130, 2, 2, 1), (385, 20, 1, 2, 0), (512, 8, 1, 2, 1), (513, 8, 1, 2, 1)]


@pytest.mark.parametrize("p,r,B,q,warm", SIZES)
def test_columns_meet_the_stopping_bound(p, r, B, q, warm):
    X, Y, w, lam = problem(3 * p + 40, p, r, B, q, 700 + p)
    gpu = native.lasso_admm_batch(X, Y, w, lam, precision=native.PREC_MIXED, warm_start=warm)
    assert gpu["conv"].all()
    some = list(range(r)) if r <= 6 else [0, 1, r // 2, r - 1]
    z = np.ascontiguousarray(gpu["beta"][:, :, some])
    mixed_check.check_residuals(X, np.ascontiguousarray(Y[:, some]), w, lam, z, mixed_check.ETA_MIXED)
    # the iterates are the oracle's up to FP32 rounding: so are their counts, but for a step
    # at a stop that rounding decides
    ref = oracle.lasso_admm_batch(X, Y, w[:1], lam, warm_start=warm, eq_list=some)
    assert np.abs(gpu["iters"][:1][:, :, some] - ref["iters"]).max() <= 2


def test_more_chains_than_fit_the_device():
    """Chains past a cluster's 128 lanes are taken over by lanes whose chain has ended:
    every column must come out, and as in a call with that response alone."""
    X, Y, w, lam = problem(500, 140, 300, 60, 2, 5)
    X, Y, lam = (torch.from_numpy(v).cuda() for v in (X, Y, lam))
    w = torch.from_numpy(w.astype(np.int32)).cuda()
    full = native.lasso_admm_batch(X, Y, w, lam, precision=native.PREC_MIXED)
    assert bool(full["conv"].all())
    part = native.lasso_admm_batch(X, Y[:, 290:300].contiguous(), w, lam, precision=native.PREC_MIXED)
    # same products and sums whatever the lane: only c = M b (a product over responses) may round apart
    assert float((full["beta"][:, :, 290:300] - part["beta"]).abs().max()) <= 1e-5


def test_iteration_cap_and_family_of_a_fit():
    X, Y, w, lam = problem(300, 100, 12, 2, 3, 8)
    gpu = native.lasso_admm_batch(X, Y, w, lam, precision=native.PREC_MIXED, max_iter=3)
    assert (gpu["iters"] == 3).all() and not gpu["conv"].any() and gpu["status"] == native.OK_WITH_WARNINGS
    out = native.uoi_fit_traced(X, Y, B1=4, B2=3, q=5, precision=native.PREC_MIXED)
    keep = (out["sel_beta"] != 0).all(axis=0)                     # q x r x p
    bits = np.zeros_like(keep)
    for i in range(100):
        bits[..., i] = (out["family"][..., i // 64] >> np.uint64(i % 64)) & np.uint64(1)
    np.testing.assert_array_equal(bits, keep)
