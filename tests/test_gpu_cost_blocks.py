"""Cost-model training with one block, a cluster, a cooperative grid, many
chunks to a block, and ragged last chunks, against the float64 reference."""
import numpy as np
import pytest

from oracle import cost_mlp
from tests.gpu_util import torch_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 32, 33, 80, 256, 257, 300, 2048, 2080, 4096, 5000, 20001])
def test_gradient_steps_and_prediction(n):
    torch_dev()
    from paper_1411_3212_gb300 import mqr
    rng = np.random.default_rng(n)
    X = rng.uniform(-1, 1, size=(n, 5)).astype(np.float32).astype(np.float64)
    y = (0.5 * X[:, 0] - X[:, 1] ** 2 + 0.3 * X[:, 2] * X[:, 3] + 0.1).astype(np.float32).astype(np.float64)
    p0 = cost_mlp.init(5).astype(np.float32)
    p64 = p0.astype(np.float64)
    m = mqr.CostModel(p0)
    g, loss = m.gradient(X, y)
    want = cost_mlp.grad(p64, X, y)
    # fp32 sums of n terms: each entry to n-independent 2^-24 steps of the largest partial sums
    np.testing.assert_allclose(g, want, rtol=1e-3, atol=1e-5 * np.abs(want).max())
    assert loss == pytest.approx(cost_mlp.loss(p64, X, y), rel=1e-4)
    np.testing.assert_array_equal(m.params(), p0)                  # a gradient changes nothing
    np.testing.assert_allclose(m.predict(X), cost_mlp.forward(p64, X)[0], rtol=1e-4, atol=1e-4)
    m.train(X, y, epochs=2, lr=1e-3)
    m.train(X, y, epochs=1, lr=1e-3)                               # the moments and the step count carry over
    ref = cost_mlp.adam(p64, X, y, epochs=3, lr=1e-3)[0]
    moved = np.abs(ref - p64) > 1e-4                               # entries whose gradient is not rounding noise
    assert moved.any()
    np.testing.assert_allclose(m.params()[moved], ref[moved], atol=3e-4)
    m.close()
