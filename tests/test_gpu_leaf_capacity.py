"""Quadtree leaves at the largest capacity of the shared-memory tables, one
below it, and in the global tables above it, against Alg. 1 level by level."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import to_dev, torch_dev
from tests.test_gpu_leaves import skewed

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [40_000, 70_001])
def test_leaves_at_the_largest_capacities(n):
    torch, dev = torch_dev()
    from paper_1411_3212_gb300 import mqr
    xy = skewed(n, n)
    ids = np.arange(n, dtype=np.uint32)
    st = oracle.State(n)
    st.apply_updates(ids, xy)
    keys = np.sort(oracle.keys(st))
    rects = to_dev(np.zeros((0, 4), np.float32), dev)
    for cap in [16376, 16383, 16384, 16385, 30_000, n - 1, n]:
        idx = mqr.Index(leaf_cap=cap, max_objects=n)
        idx.apply_updates(to_dev(ids, dev), to_dev(xy, dev))
        idx.tick(rects, kind="count")
        want = oracle.quadtree(keys, cap, 15)
        want = want[want["begin"] != want["end"]]
        np.testing.assert_array_equal(idx.leaves(), np.stack([want["level"], want["z"], want["begin"], want["end"]], 1),
                                      err_msg=str(cap))
        idx.close()
