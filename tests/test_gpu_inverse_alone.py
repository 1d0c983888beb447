"""The inverse of one system does not depend on the systems beside it: not on one that needs another
Newton step, not on one that has to take the factor, and not on the run."""
import numpy as np
import pytest

from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def first_step(X, y, w, rho, prec):
    out = native.lasso_admm_batch(X, y, torch.from_numpy(np.stack(w).astype(np.int32)).cuda(),
                                  torch.tensor([1e-280 if prec == native.PREC_FP64 else 1e-30], dtype=torch.float64).cuda(),
                                  rho=rho, max_iter=1, precision=prec)
    return out["beta"].cpu().numpy().reshape(len(w), -1)


# rho = 1e-3: rows few enough to leave G singular need steps more; 1e-9: no FP32 inverse, the factor
# (in the mixed form an error)
@pytest.mark.parametrize("p,prec,rho", [(64, native.PREC_FP64, 1e-3), (64, native.PREC_FP64, 1e-9),
                                        (129, native.PREC_FP64, 1e-3), (129, native.PREC_FP64, 1e-9),
                                        (300, native.PREC_FP64, 1e-3), (300, native.PREC_FP64, 1e-9),
                                        (100, native.PREC_MIXED, 1e-3), (192, native.PREC_MIXED, 1e-3)])
def test_neighbours_change_no_bit(p, prec, rho):
    g = np.random.default_rng(p)
    n = 4 * p
    X = torch.from_numpy(g.integers(-9, 10, (n, p)).astype(np.float64)).cuda()
    y = torch.from_numpy(g.integers(-9, 10, (n, 1)).astype(np.float64)).cuda()
    good = [g.multinomial(n, np.full(n, 1.0 / n)) for _ in range(5)]
    poor = np.zeros(n, dtype=np.int64)
    poor[: p // 2] = n // (p // 2)                       # G of rank p / 2
    want = first_step(X, y, good, rho, prec)
    assert np.isfinite(want).all()
    for places in ((0,), (4,), (1, 2), (0, 2, 4)):
        w = [poor if k in places else good[k] for k in range(5)]
        for _ in range(2):
            got = first_step(X, y, w, rho, prec)
            assert np.isfinite(got).all()
            for k in range(5):
                if k not in places:
                    np.testing.assert_array_equal(got[k], want[k])


def test_a_system_without_an_inverse_is_named():
    """Both columns of a pair equal and rho 2^-60 of the diagonal: no factor either."""
    g = np.random.default_rng(1)
    n, p = 400, 96
    X = g.integers(-9, 10, (n, p)).astype(np.float64)
    w = np.ones((3, n), dtype=np.int32)
    w[1] = 0
    w[1, :2] = n // 2                                    # rank 2
    args = [torch.from_numpy(a).cuda() for a in (X, X[:, :1].copy(), w, np.array([0.1]))]
    with pytest.raises(Exception, match="item 1"):
        native.lasso_admm_batch(*args, rho=1e-17)
