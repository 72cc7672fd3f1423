"""mlp_grad where its kernels divide the samples: one sample, a CTA's four and five,
the largest batch that is added in order and the first that is split over groups
of threads, against the FP64 oracle at the FP16-rounded weights.

Bound: a gradient entry is a sum of n FP32 products, off by at most n 2^-24 of the sum
of magnitudes when added in order, and by about sqrt(n) 2^-24 in the 2-norm over
the entries; sqrt(5000) 2^-24 = 4e-6, and five times that, 2e-5, covers the forward
pass and tanh.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_1402_7285_gb300 as tb
from oracle import mlp


@pytest.mark.parametrize("n", [1, 4, 5, 1024, 1025, 5000])
def test_gradient_at_batch_edges(n):
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 32)).astype(np.float32)
    y = rng.standard_normal(n).astype(np.float32)
    p = mlp.init_params(11)
    flat = np.concatenate([np.asarray(p[k], np.float64).ravel() for k in mlp.PARAM_NAMES]).astype(np.float32)
    ph, off = {}, 0
    for k in mlp.PARAM_NAMES:
        v = np.asarray(p[k])
        ph[k] = flat[off:off + v.size].astype(np.float16).astype(np.float64).reshape(v.shape)
        off += v.size
    with tb.Context() as ctx:
        g, loss = tb.mlp_grad(ctx, flat, X, y)
        again, _ = tb.mlp_grad(ctx, flat, X, y)
    ref = mlp.backward(ph, X.astype(np.float64), y.astype(np.float64))
    ref = np.concatenate([np.asarray(ref[k]).ravel() for k in mlp.PARAM_NAMES])
    assert np.linalg.norm(g - ref) <= 2e-5 * np.linalg.norm(ref)
    assert abs(loss - mlp.loss(ph, X.astype(np.float64), y.astype(np.float64))) <= 2e-5 * loss
    assert np.array_equal(g, again)
