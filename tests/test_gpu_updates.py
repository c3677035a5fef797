"""Update calls at the edges of the update kernels' items."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import to_dev, torch_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 255, 256, 257, 1023, 1024, 1025, 5000])
def test_update_calls_of_every_size(n):
    torch, dev = torch_dev()
    from paper_1411_3212_gb300 import mqr
    rng = np.random.default_rng(n)
    nmax = 3000
    idx = mqr.Index(leaf_cap=32, max_objects=nmax)
    st = oracle.State(nmax)
    for k in range(3):                                   # repeated ids within a call, later calls win
        ids = rng.integers(0, nmax, n).astype(np.uint32)
        xy = rng.random((n, 2)).astype(np.float32)
        idx.apply_updates(to_dev(ids, dev), to_dev(xy, dev))
        st.apply_updates(ids, xy)
    rects = np.array([[0.0, 0.0, 1.0, 1.0], [0.2, 0.3, 0.5, 0.9]], np.float32)
    off, got = oracle.join_grid(st, rects, cell_side=0.1)
    res, offs = idx.tick(to_dev(rects, dev), kind="csr_sorted")
    np.testing.assert_array_equal(offs.cpu().numpy(), off.astype(np.int64))
    np.testing.assert_array_equal(res.cpu().numpy().view(np.uint32), got)
    idx.close()
