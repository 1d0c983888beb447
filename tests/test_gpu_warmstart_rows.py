"""Gradient of the warm-start network at batch sizes around its row slices (256), tiles (64
rows) and vector pairs, against the FP64 reference, with the bound of test_gpu_warmstart.py."""
import numpy as np
import pytest

from oracle import mlp
from paper_1808_06992_gb300 import native

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 63, 65, 255, 256, 257, 513])
def test_gradient_at_row_edges(n):
    g = np.random.Generator(np.random.PCG64(n))
    X = (g.standard_normal((n, 8)) * 1.5).astype(np.float32)
    T = np.column_stack([g.standard_normal(n), g.uniform(-1, 1, n), g.integers(0, 2, n)]).astype(np.float32)
    m = native.WarmStartModel(seed=n)
    params = mlp.bf16_round(m.get_params()).astype(np.float32)
    m.set_params(params)
    P = mlp.unflatten(params.astype(np.float64))
    L, grad = m.loss_grad(X, T)
    Lr, gr = mlp.loss_and_grad(P, X.astype(np.float64), T.astype(np.float64), round_act=mlp.bf16_round)
    assert abs(L - Lr) <= 5e-5 * abs(Lr)
    at = 0
    for sh, want in zip(mlp.shapes(), gr):
        k = int(np.prod(sh))
        got = grad[at:at + k].astype(np.float64).reshape(sh)
        at += k
        # a BF16 rounding that FP32 and FP64 values decide differently moves one of n 512 terms by
        # 2^-8: the whole gradient's bound, with that one term beside it for small batches
        assert np.linalg.norm(got - want) <= (5e-4 + 2.0 ** -8 / np.sqrt(n)) * np.linalg.norm(want)
