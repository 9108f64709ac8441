"""Gradients of one minibatch, computed again: the weight and bias gradients of the two hidden layers are the
same bits where no more than two partial sums meet (below 3072 and up to 1024 rows)."""
import numpy as np
import pytest

from paper_2410_19993_gb300 import xbar

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

H = 256


@pytest.mark.parametrize("rows", [1, 128, 300, 513, 1024, 1025, 2047, 2944])
def test_same_bits(rows):
    M = 40
    s = xbar.Surrogate(M, M, (1.0, 2.5, 2.5, 10.0), passes=2, g_scale=1e-4, v_scale=0.5, seed=0)
    rng = np.random.default_rng(rows)
    X = rng.random((rows, 3 * M)).astype(np.float32)
    y = rng.normal(0.0, 1.0, rows).astype(np.float32)
    Fp = (3 * M + 127) // 128 * 128
    W1, b1, W2, b2 = slice(0, H * Fp), slice(H * Fp, H * Fp + H), slice(H * Fp + H, H * Fp + H + H * H), \
        slice(H * Fp + H + H * H, H * Fp + 2 * H + H * H)
    first = np.array(s.grad(X, y)[1])
    for _ in range(20):
        g = np.array(s.grad(X, y)[1])
        for part in (W1, W2) + ((b1, b2) if rows <= 1024 else ()):
            assert np.array_equal(first[part], g[part])
