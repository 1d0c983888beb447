"""Calls from threads that come and go: each has a second stream of its own, given back when it ends,
and gets the results of the main thread."""
import threading

import numpy as np
import pytest

from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_gradients_and_fits_from_short_lived_threads():
    g = np.random.default_rng(3)
    X = (g.standard_normal((700, 8))).astype(np.float32)
    T = np.column_stack([g.standard_normal(700), g.uniform(-1, 1, 700), g.integers(0, 2, 700)]).astype(np.float32)
    m = native.WarmStartModel(seed=1)
    A = torch.from_numpy(g.standard_normal((900, 40))).cuda()
    y = A[:, :4].sum(dim=1) + torch.randn(900, dtype=torch.float64, device="cuda")
    kw = dict(B1=8, B2=6, q=6, precision=native.PREC_MIXED)
    want, fit = m.loss_grad(X, T), native.uoi_lasso_fit(A, y, **kw)["beta"]
    got = []

    def call():
        got.append((m.loss_grad(X, T), native.uoi_lasso_fit(A, y, **kw)["beta"]))

    for _ in range(12):
        t = threading.Thread(target=call)
        t.start()
        t.join()
    assert len(got) == 12
    native.lib().uoi_shutdown()                          # the ended threads' stream goes; calls go on
    call()
    for (loss, grad), beta in got:
        assert loss == want[0] and np.array_equal(grad, want[1]) and torch.equal(beta, fit)
