"""The FP64 moments from exact integer products on the tensor cores (weighted_moments in
the plain form): integer data must come back exactly, real data within the bound of
the slicing, and inputs the slicing does not take must give the plain sums."""
import numpy as np
import pytest

from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def moments(X, Y, w):
    Xd, Yd = torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda()
    G, B = native.weighted_moments(Xd, Yd, torch.from_numpy(w.astype(np.int32)).cuda())
    return G.cpu().numpy(), B.cpu().numpy()


# tile edges (64 columns, 128 rows of Z), chunk edges (128 listed rows), one row, many responses
SIZES = [(1, 1, 1, 1), (127, 63, 1, 2), (128, 64, 64, 1), (129, 65, 3, 3), (300, 127, 1, 5), (1000, 130, 2, 2),
         (257, 5, 200, 2), (20000, 3, 1, 1)]


@pytest.mark.parametrize("n,p,r,B", SIZES)
def test_integer_data_is_exact(n, p, r, B):
    g = np.random.default_rng(n + p)
    X = g.integers(-3000, 3001, (n, p)).astype(np.float64)
    Y = g.integers(-50, 51, (n, r)).astype(np.float64)
    X[:, p // 2] = 0.0
    w = g.integers(0, 4, (B, n)).astype(np.uint32)
    w[0, n // 2] = 70001                                 # many bits; the sums stay below 2^53
    G, Bm = moments(X, Y, w)
    Xi, Yi = X.astype(np.int64), Y.astype(np.int64)
    for k in range(B):
        wx = Xi * w[k].astype(np.int64)[:, None]
        np.testing.assert_array_equal(G[k], (wx.T @ Xi).astype(np.float64))
        np.testing.assert_array_equal(Bm[k], (wx.T @ Yi).astype(np.float64))


@pytest.mark.parametrize("n,p,spread", [(200, 50, 0), (5000, 40, 0), (700, 33, 30)])
def test_real_data_within_the_slicing_bound(n, p, spread):
    """spread: columns scaled by powers of two over +-spread.  Rounding of a column to 56
    bits: 2^-55 of its largest value; products of orders 7..12: 6.1 2^-54 of the product
    of the largest values; one final rounding (2^-52 to spare the two-step sum)."""
    g = np.random.default_rng(7 * n + p)
    X = g.standard_normal((n, p)) * 2.0 ** g.integers(-spread, spread + 1, p)
    y = g.standard_normal((n, 1))
    w = g.multinomial(n, np.full(n, 1.0 / n), size=2).astype(np.uint32)
    G, Bm = moments(X, y, w)
    for k in range(2):
        Z = np.concatenate([X, y], axis=1).astype(np.longdouble)
        ref = (Z * w[k].astype(np.longdouble)[:, None]).T @ Z
        big = np.abs(Z[w[k] > 0]).max(axis=0)
        tol = float(w[k].sum()) * np.outer(big, big) * (2.0 ** -54 + 6.1 * 2.0 ** -54) + 2.0 ** -52 * np.abs(ref)
        assert (np.abs(G[k] - ref[:p, :p]) <= tol[:p, :p]).all()
        assert (np.abs(Bm[k] - ref[:p, p:]) <= tol[:p, p:]).all()
        # no worse than a plain FP64 product on the same data
        Zd = Z.astype(np.float64)
        plain = np.zeros((p, p))
        for t in np.nonzero(w[k])[0]:
            plain += w[k][t] * np.outer(Zd[t, :p], Zd[t, :p])
        scale = np.sqrt(np.outer(np.diag(ref[:p, :p]), np.diag(ref[:p, :p])))
        err = np.sqrt(np.mean(((G[k] - ref[:p, :p]) / scale).astype(np.float64) ** 2))
        assert err <= np.sqrt(np.mean(((plain - ref[:p, :p]) / scale).astype(np.float64) ** 2))


def test_scale_follows_the_rows_in_use():
    """A huge value in a row of weight zero costs the others nothing."""
    g = np.random.default_rng(3)
    X = g.standard_normal((300, 20))
    y = g.standard_normal((300, 1))
    w = np.ones((1, 300), dtype=np.uint32)
    w[0, 10] = 0
    G0, _ = moments(X, y, w)
    X2 = X.copy()
    X2[10] = 1e200
    G1, _ = moments(X2, y, w)
    np.testing.assert_array_equal(G0, G1)


@pytest.mark.parametrize("what", ["nan", "inf", "heavy"])
def test_inputs_past_the_slicing_take_the_plain_sums(what):
    g = np.random.default_rng(4)
    X = g.integers(-9, 10, (200, 10)).astype(np.float64)
    y = np.ones((200, 1))
    w = np.ones((1, 200), dtype=np.uint32)
    if what == "heavy":
        w[0, 3] = 1 << 25
    else:
        X[5, 2] = np.nan if what == "nan" else np.inf
    G, _ = moments(X, y, w)
    ref = (X * w[0][:, None]).T @ X
    np.testing.assert_array_equal(np.isnan(G[0]), np.isnan(ref))
    np.testing.assert_array_equal(G[0][np.isfinite(ref)], ref[np.isfinite(ref)])
