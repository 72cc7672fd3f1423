"""The forward pass alone changes kernels above 5120 samples: predictions have the same bits
on both sides (the same operations in the same order) and losses are the mean of their
squared errors, whose FP32 parts of 4 or 128 squares err by at most 8 * 2^-24 = 5e-7."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_1402_7285_gb300 as tb
from paper_1402_7285_gb300 import scheduler


@pytest.mark.parametrize("n", [1, 4, 5119, 5120, 5121, 20000, 100001])
def test_predictions_have_the_same_bits_in_any_batch(n):
    X = np.random.default_rng(n).standard_normal((n, 32)).astype(np.float32)
    p = scheduler.init_params(3)
    with tb.Context() as ctx:
        all_ = tb.mlp_predict(ctx, p, X)
        parts = np.concatenate([tb.mlp_predict(ctx, p, X[s:s + 4999]) for s in range(0, n, 4999)])
        dev = tb.mlp_predict(ctx, p, torch.as_tensor(X, device="cuda")).cpu().numpy()
    assert np.array_equal(all_, parts) and np.array_equal(all_, dev)


@pytest.mark.parametrize("n", [5120, 5121, 30001])
def test_loss_is_the_mean_squared_error(n):
    rng = np.random.default_rng(n)
    X, y = rng.standard_normal((n, 32)).astype(np.float32), rng.standard_normal(n).astype(np.float32)
    with tb.Context() as ctx:
        p, hist = tb.mlp_train(ctx, X, y, epochs=2, batch=4096, lr=1e-3, params=scheduler.init_params(3))
        pred = tb.mlp_predict(ctx, p, X)
    assert np.isclose(hist[-1], np.mean((pred.astype(np.float64) - y) ** 2), rtol=1e-6)
