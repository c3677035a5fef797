"""Models trained in several threads at once, with launches of different sizes:
each as if it were alone."""
import threading

import numpy as np
import pytest

from tests.gpu_util import torch_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(300, 4096), (4096, 4096), (80, 300, 2080, 9000)])
def test_concurrent_trainings(sizes):
    torch_dev()
    from paper_1411_3212_gb300 import mqr
    from paper_1411_3212_gb300.costmodel import he_uniform_params
    p0 = he_uniform_params(4)

    def train(n, repeats):
        rng = np.random.default_rng(n)
        X = rng.uniform(-1, 1, size=(n, 5)).astype(np.float32)
        y = (0.5 * X[:, 0] - X[:, 1] ** 2).astype(np.float32)
        m = mqr.CostModel(p0)
        for _ in range(repeats):
            m.set_params(p0)
            m.train(X, y, epochs=3, lr=3e-3)
        p = m.params()
        m.close()
        return p

    want = [train(n, 1) for n in sizes]
    got = [None] * len(sizes)

    def work(i):
        try:
            got[i] = train(sizes[i], 150)
        except Exception as e:                      # reported below, in the test's own thread
            got[i] = e

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for g, w in zip(got, want):
        assert not isinstance(g, Exception), g
        np.testing.assert_array_equal(g, w)
