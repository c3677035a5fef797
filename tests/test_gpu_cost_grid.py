"""Training whose grid cannot run: its wait runs out, its launch is refused, or
an allocation before it fails.  The model is trained all the same, or as it was."""
import numpy as np
import pytest

from tests.gpu_util import torch_dev

pytestmark = pytest.mark.gpu


@pytest.fixture
def hooks():
    yield
    from paper_1411_3212_gb300 import mqr
    mqr.mqr_debug_cost_grid(0)
    mqr.mqr_debug_fail_allocation(-1)


def samples(n):
    rng = np.random.default_rng(n)
    X = rng.uniform(-1, 1, size=(n, 5)).astype(np.float32)
    return X, (0.5 * X[:, 0] - X[:, 1] ** 2 + 0.3 * X[:, 2] * X[:, 3]).astype(np.float32)


@pytest.mark.parametrize("n", [257, 300, 4096, 20001])
@pytest.mark.parametrize("mode", [1, 2])
def test_training_without_a_grid_is_the_same(n, mode, hooks):
    torch_dev()
    from paper_1411_3212_gb300 import mqr
    from paper_1411_3212_gb300.costmodel import he_uniform_params
    X, y = samples(n)
    models = [mqr.CostModel(he_uniform_params(4)) for _ in range(2)]
    got = []
    for k, m in enumerate(models):
        got.append([])
        for epochs in (3, 2):                                  # moments and step count carry over
            mqr.mqr_debug_cost_grid(mode if k else 0)
            loss = m.train(X, y, epochs=epochs, lr=3e-3)
            got[k] += [np.float32(loss), m.params()]
        mqr.mqr_debug_cost_grid(mode if k else 0)
        g, loss = m.gradient(X, y)
        got[k] += [np.float32(loss), g, m.params(), m.predict(X)]
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
    for m in models:
        m.close()


def test_a_failed_training_changes_nothing(hooks):
    torch_dev()
    from paper_1411_3212_gb300 import mqr
    from paper_1411_3212_gb300.costmodel import he_uniform_params
    X, y = samples(300)
    p0 = he_uniform_params(4)
    want = mqr.CostModel(p0)
    want.train(X, y, epochs=3, lr=3e-3)
    failed = 0
    for after in range(12):
        m = mqr.CostModel(p0)
        mqr.mqr_debug_fail_allocation(after)
        try:
            m.train(X, y, epochs=3, lr=3e-3)
        except mqr.MqrError as e:
            assert e.status == mqr.MQR_ERR_OOM
            failed += 1
            np.testing.assert_array_equal(m.params(), p0)
            mqr.mqr_debug_fail_allocation(-1)
            m.train(X, y, epochs=3, lr=3e-3)
        mqr.mqr_debug_fail_allocation(-1)
        np.testing.assert_array_equal(m.params(), want.params())
        m.close()
    assert failed >= 4
    want.close()
