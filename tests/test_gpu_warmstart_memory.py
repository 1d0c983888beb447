"""Device memory of a warm-start gradient per row of its batch."""
import numpy as np
import pytest

from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_gradient_takes_fifteen_activations_per_row():
    """512 features: three FP32 pre-activations, three BF16 activations and their transposes, one
    BF16 gradient and two transposes; beside them inputs and outputs (below 200 bytes a row) and
    what does not grow with the rows (slices of weight gradients, 33 MB; granules of the pool)."""
    n = 600_000
    g = np.random.default_rng(0)
    X = g.standard_normal((n, 8)).astype(np.float32)
    T = np.column_stack([g.standard_normal(n), g.uniform(-1, 1, n), g.integers(0, 2, n)]).astype(np.float32)
    m = native.WarmStartModel(seed=0)
    m.loss_grad(X[:64], T[:64])
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    m.loss_grad(X, T)
    torch.cuda.synchronize()
    used = free0 - torch.cuda.mem_get_info()[0]
    assert used <= n * (512 * (3 * 4 + 9 * 2) + 200) + (512 << 20)
