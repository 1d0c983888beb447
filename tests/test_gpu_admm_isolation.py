"""Responses that are not finite stay alone: chains that take over a lane, a slot or a cluster from
one that held NaN or Inf come out as in a call without it.  Every chain of a call runs to the cap of
iterations, so that the poisoned chain's place is taken over by others."""
import numpy as np
import pytest

from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# FP32: more chains than the clusters' lanes, cold and path start, the resident sizes and past them;
# FP64: one chain per cluster and four
@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e200])
@pytest.mark.parametrize("p,r,B,warm,prec", [(140, 300, 60, 1, native.PREC_MIXED), (140, 150, 60, 0, native.PREC_MIXED),
                                             (400, 300, 20, 1, native.PREC_MIXED), (90, 40, 20, 1, native.PREC_FP64),
                                             (300, 40, 60, 0, native.PREC_FP64)])
def test_other_responses_are_untouched(p, r, B, warm, prec, bad):
    if bad == 1e200 and prec == native.PREC_FP64:
        pytest.skip("an ordinary value in FP64")
    g = np.random.default_rng(p + r)
    n = 500
    X = g.standard_normal((n, p))
    Y = X[:, :6] @ g.uniform(0.5, 2.0, (6, r)) + g.standard_normal((n, r))
    w = g.multinomial(n, np.full(n, 1.0 / n), size=B).astype(np.int32)
    lam = np.abs(X.T @ Y).max() / n * np.array([0.5, 0.05])
    others = np.setdiff1d(np.arange(r), [3])
    X, w, lam, Yd = (torch.from_numpy(a).cuda() for a in (X, w, lam, Y))
    kw = dict(warm_start=warm, precision=prec, max_iter=6, abs_tol=0.0, rel_tol=0.0)
    want = native.lasso_admm_batch(X, Yd, w, lam, **kw)
    Yd = Yd.clone()
    Yd[n // 2, 3] = bad
    got = native.lasso_admm_batch(X, Yd, w, lam, **kw)
    assert torch.isfinite(want["beta"]).all()
    assert bool((got["iters"] == 6).all())
    a, b = (v["beta"][:, :, others].cpu().numpy() for v in (got, want))
    # moments that hold a value that is not finite may be summed by another kernel: rounding apart
    assert np.isfinite(a).all()
    tol = 1e-12 if prec == native.PREC_FP64 else 1e-4
    assert np.abs(a - b).max() <= tol * np.abs(b).max()
