"""Scratch memory of the FP64 form: the moments' digit slices stay within their budget however many
rows a call has, and a device with less memory gets the same bits from smaller pieces, or from the
forms that need none."""
import numpy as np
import pytest

from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture
def limit():
    yield native.selftest_alloc_limit
    native.selftest_alloc_limit(0)


# whole; in ranges of rows (several items at a time, one); the plain sums
@pytest.mark.parametrize("nbytes", [0, 300 << 20, 100 << 20, 20 << 20, 7 << 20, 1 << 20])
@pytest.mark.parametrize("n,p,r,B", [(20000, 400, 1, 4), (20001, 130, 150, 3)])
def test_moments_with_less_memory_are_the_same(n, p, r, B, nbytes, limit):
    g = np.random.default_rng(n + p)
    X = g.integers(-300, 301, (n, p)).astype(np.float64)
    Y = g.integers(-50, 51, (n, r)).astype(np.float64)
    w = g.multinomial(n, np.full(n, 1.0 / n), size=B).astype(np.int32)
    w[0, : n // 3] = 0                                   # items of different lengths
    Xd, Yd, wd = (torch.from_numpy(a).cuda() for a in (X, Y, w))
    limit(nbytes)
    G, Bm = native.weighted_moments(Xd, Yd, wd)
    for k in range(B):
        wx = Xd * wd[k][:, None].double()
        assert torch.equal(G[k], wx.T @ Xd) and torch.equal(Bm[k], wx.T @ Yd)    # integers below 2^53


def test_rows_past_the_budget_are_taken_in_ranges():
    """1.5e6 x 1000 (12 GB): all slices at once would be 21.5 GB.  The call may take the budget of
    16 GB, and its lists and sums (far below 1 GB)."""
    n, p = 1_500_000, 1000
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.empty((n, p), dtype=torch.float64, device="cuda")
    for i in range(0, n, 100_000):
        X[i:i + 100_000] = torch.randint(-9, 10, (100_000, p), generator=g, device="cuda").double()
    y = torch.randint(-9, 10, (n, 1), generator=g, device="cuda").double()
    w = torch.ones((1, n), dtype=torch.int32, device="cuda")
    G = torch.empty(0)
    native.weighted_moments(X[:256, :8].contiguous(), y[:256], w[:, :256].contiguous())
    torch.cuda.empty_cache()
    free0 = torch.cuda.mem_get_info()[0]
    G, Bm = native.weighted_moments(X, y, w)
    torch.cuda.synchronize()
    used = free0 - torch.cuda.mem_get_info()[0]
    assert used <= 17 * 2 ** 30
    for c in (0, 448, 936):
        assert torch.equal(G[0, c:c + 64, :64], X[:, c:c + 64].T @ X[:, :64])
    assert torch.equal(Bm[0], X.T @ y)


@pytest.mark.parametrize("nbytes", [40 << 20, 6 << 20, 3 << 20])
def test_a_solve_with_less_memory_gives_the_same_columns(nbytes, limit):
    """Below the inverse's scratch the systems take the factor: rounding apart."""
    g = np.random.default_rng(2)
    X = g.standard_normal((3000, 200))
    y = X[:, :5] @ g.uniform(0.5, 2.0, 5) + g.standard_normal(3000)
    w = g.multinomial(3000, np.full(3000, 1.0 / 3000), size=4).astype(np.int32)
    lam = np.abs(X.T @ y).max() / 3000 * np.array([0.5, 0.05])
    args = [torch.from_numpy(a).cuda() for a in (X, y, w, lam)]
    want = native.lasso_admm_batch(*args)
    limit(nbytes)
    got = native.lasso_admm_batch(*args)
    assert torch.equal(got["iters"], want["iters"])
    assert float((got["beta"] - want["beta"]).abs().max()) <= 1e-12 * float(want["beta"].abs().max())


def test_a_call_that_cannot_do_with_less_says_so(limit):
    X = torch.randn((2000, 64), dtype=torch.float64, device="cuda")
    w = torch.ones((1, 2000), dtype=torch.int32, device="cuda")
    lam = torch.tensor([0.1], dtype=torch.float64, device="cuda")
    limit(1 << 10)
    with pytest.raises(Exception, match="(?i)memory|limit"):
        native.lasso_admm_batch(X, X[:, 0].contiguous(), w, lam)
    limit(0)
    assert native.lasso_admm_batch(X, X[:, 0].contiguous(), w, lam)["status"] >= 0
