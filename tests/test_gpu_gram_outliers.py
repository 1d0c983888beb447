"""FP64 moments of columns with entries far above their others: where the other column is zero in
those rows, entries of G must come from the ordinary values with all their bits."""
import numpy as np
import pytest

from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def moments(X, Y, w):
    G, B = native.weighted_moments(*(torch.from_numpy(a).cuda() for a in (X, Y, w.astype(np.int32))))
    return G.cpu().numpy(), B.cpu().numpy()


# huge entries: none, one, some, more than the share that is summed apart (plain sums); in X, in y
@pytest.mark.parametrize("far", [0, 1, 3, 60])
@pytest.mark.parametrize("n,p,B", [(7, 3, 1), (200, 20, 3), (400, 130, 2), (3000, 65, 2)])
def test_ordinary_entries_keep_their_bits(n, p, B, far):
    g = np.random.default_rng(n + far)
    X = g.integers(-9, 10, (n, p)).astype(np.float64)
    Y = g.integers(-9, 10, (n, 2)).astype(np.float64)
    w = g.integers(0, 3, (B, n))
    rows = g.permutation(n)[: min(far, n // 2)]
    for i, t in enumerate(rows):
        X[t] = 0.0
        Y[t] = 0.0
        if i % 3 == 2:
            Y[t, 1] = 2.0 ** 60
        else:
            X[t, i % p] = -(2.0 ** 62)
        w[:, t] = 1 + i % 2
    G, Bm = moments(X, Y, w)
    Z = np.concatenate([X, Y], axis=1)
    for k in range(B):
        small = np.where(np.abs(Z) < 10, Z, 0.0).astype(np.int64)
        ref = ((small * w[k][:, None]).T @ small).astype(np.float64)
        big = np.where(np.abs(Z) < 10, 0.0, Z)
        ref += (big * w[k][:, None]).T @ big                 # on the diagonal alone: one rounding
        got = np.concatenate([G[k], Bm[k]], axis=1)
        off = ~np.eye(p, p + 2, dtype=bool)
        np.testing.assert_array_equal(got[off], ref[:p][off])
        assert (np.abs(np.diag(got[:, :p]) - np.diag(ref)[:p]) <= 2.0 ** -51 * np.diag(ref)[:p]).all()
        np.testing.assert_array_equal(G[k], G[k].T)


def test_heavy_tails_stay_near_the_exact_sums():
    """Log-normal columns (largest entries 2^13 to 2^20 times the typical one): every entry within
    what FP64 sums of n products may be off by, n 2^-53 of the sum of their magnitudes."""
    g = np.random.default_rng(7)
    n, p = 2000, 12
    X = np.exp(3.0 * g.standard_normal((n, p))) * g.choice([-1.0, 1.0], (n, p))
    X[:, 5] *= np.abs(X[:, 0]) < 1.0                         # zero where the first column is large
    y = g.standard_normal((n, 1))
    w = g.multinomial(n, np.full(n, 1.0 / n), size=2)
    G, Bm = moments(X, y, w)
    for k in range(2):
        Z = np.concatenate([X, y], axis=1).astype(np.longdouble)
        wz = Z * w[k].astype(np.longdouble)[:, None]
        got = np.concatenate([G[k], Bm[k]], axis=1)
        assert (np.abs(got - (wz.T @ Z)[:p]) <= n * 2.0 ** -53 * (np.abs(wz).T @ np.abs(Z))[:p]).all()
