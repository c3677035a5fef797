"""Quadtree leaves at capacities around the leaf builder's blocks of eight
positions, at populations around its tiles, against Alg. 1 level by level."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import to_dev, torch_dev

pytestmark = pytest.mark.gpu


def skewed(n, seed):
    rng = np.random.default_rng(seed)
    xy = rng.random((n, 2)).astype(np.float32)
    xy[::3] = (0.7 + 0.002 * rng.normal(size=(len(xy[::3]), 2))).astype(np.float32)
    xy[: n // 10] = xy[0]                                # a pile deeper than any capacity below n / 10
    return xy


@pytest.mark.parametrize("n", [9, 2047, 2048, 2049, 4097, 12345])
def test_leaves_at_block_edges(n):
    torch, dev = torch_dev()
    from paper_1411_3212_gb300 import mqr
    xy = skewed(n, n)
    ids = np.arange(n, dtype=np.uint32)
    st = oracle.State(n)
    st.apply_updates(ids, xy)
    keys = np.sort(oracle.keys(st))
    idx = mqr.Index(leaf_cap=1, max_objects=n)
    idx.apply_updates(to_dev(ids, dev), to_dev(xy, dev))
    rects = to_dev(np.zeros((0, 4), np.float32), dev)
    for cap in [1, 2, 3, 6, 7, 8, 9, 11, 15, 16, 17, 20, 23, 24, 25, 31, 33, 63, 64, 65, 71, 100, 127, 128, 129, 136,
                200, 255, 256, 257, 511, 1000, 2040, 2047, 2048, 2049, 4096, 9000, 12344, 16384]:
        idx.set_index(0, leaf_cap=cap)
        idx.tick(rects, kind="count")
        want = oracle.quadtree(keys, cap, 15)
        want = want[want["begin"] != want["end"]]
        np.testing.assert_array_equal(idx.leaves(), np.stack([want["level"], want["z"], want["begin"], want["end"]], 1),
                                      err_msg=str(cap))
    idx.close()
