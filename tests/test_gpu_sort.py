"""The object sort at the edges of its paths: the one-launch cluster sort (up
to 65,536 objects; one, two or four keys a thread), the tile passes, and their
digit starts added per tile (up to 32 groups of 32 tiles) or scanned first."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import to_dev, torch_dev

pytestmark = pytest.mark.gpu


def points(n, seed):
    """Skewed positions with ties: half in one small square, some repeated."""
    rng = np.random.default_rng(seed)
    xy = rng.random((n, 2)).astype(np.float32)
    xy[::2] = (0.3 + 0.01 * xy[::2]).astype(np.float32)
    xy[n // 2: n // 2 + n // 8] = xy[0]
    return xy


def keys_of(n, ids, xy):
    st = oracle.State(n)
    st.apply_updates(ids, xy)
    return oracle.keys(st)


@pytest.mark.parametrize("n", [1, 33, 1024, 1025, 16384, 16385, 32769, 65535, 65536, 65537, 131072, 131073, 135169])
def test_noalloc_sort_sizes(n):
    torch, dev = torch_dev()
    from paper_1411_3212_gb300 import mqr
    xy = points(n, n)
    k = torch.zeros(n + 1, dtype=torch.int32, device=dev)
    i = torch.zeros(n + 1, dtype=torch.int32, device=dev)
    mqr.mqr_sort_objects_noalloc((0.0, 0.0, 1.0, 1.0), to_dev(xy, dev), n, k, i)
    want = keys_of(n, np.arange(n, dtype=np.uint32), xy)
    order = np.argsort(want, kind="stable")
    np.testing.assert_array_equal(k.cpu().numpy().view(np.uint32)[:n], want[order])
    np.testing.assert_array_equal(i.cpu().numpy().view(np.uint32)[:n], order)
    assert int(k[n]) == 0 and int(i[n]) == 0            # nothing past the end


@pytest.mark.parametrize("n", [1, 1025, 16385, 40001, 65536, 65537, 131073, 4194304, 4194305])
def test_index_sort_sizes_with_absent_slots(n):
    torch, dev = torch_dev()
    from paper_1411_3212_gb300 import mqr
    xy = points(n, n)
    ids = np.arange(n, dtype=np.uint32)
    ids = ids[ids % 7 != 3] if n > 1 else ids           # absent slots throughout
    idx = mqr.Index(leaf_cap=64, max_objects=n)
    idx.apply_updates(to_dev(ids, dev), to_dev(xy[ids], dev))
    rects = to_dev(np.array([[0.0, 0.0, 1.0, 1.0]], np.float32), dev)
    res, _ = idx.tick(rects, kind="csr_sorted")         # every position through the filter or a run
    assert res.shape[0] == ids.shape[0]
    k, i = idx.sorted_objects()
    idx.close()
    want = keys_of(n, ids, xy[ids])[ids]
    order = np.argsort(want, kind="stable")
    np.testing.assert_array_equal(k, want[order])
    np.testing.assert_array_equal(i, ids[order])


def test_small_sort_of_batched_worlds():
    torch, dev = torch_dev()
    from paper_1411_3212_gb300 import mqr
    base = np.array([0, 10, 10, 2000, 9001, 20000], np.uint32)
    n = int(base[-1])
    xy = points(n, 5)
    idx = mqr.Index(leaf_cap=64, max_objects=n)
    idx.apply_updates(to_dev(np.arange(n, dtype=np.uint32), dev), to_dev(xy, dev))
    idx.set_worlds(base)
    q = np.array([0, 1, 2, 3, 4, 5], np.uint32)
    idx.set_query_worlds(q)
    rects = to_dev(np.tile(np.array([[0.0, 0.0, 1.0, 1.0]], np.float32), (5, 1)), dev)
    res, offs = idx.tick(rects, kind="csr_sorted")
    idx.close()
    np.testing.assert_array_equal(offs.cpu().numpy(), base)
    np.testing.assert_array_equal(res.cpu().numpy(), np.arange(n))
