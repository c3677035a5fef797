"""Filter items one, two and four to a ticket: numbers of items on both sides of
one and of four to a warp of the grid (made small by the launch shapes)."""
import numpy as np
import pytest

import oracle
from paper_1411_3212_gb300 import workloads
from tests.gpu_util import oracle_state, to_dev, torch_dev

pytestmark = pytest.mark.gpu


def test_items_per_ticket():
    torch, dev = torch_dev()
    from paper_1411_3212_gb300 import mqr
    warps = 8 * torch.cuda.get_device_properties(0).multi_processor_count
    seen = set()
    for n in [1, 2000, 4 * warps - 40, 4 * warps + 40, 5 * warps, 16 * warps - 80, 16 * warps + 80, 20 * warps]:
        # n objects on a grid, four to a leaf: about n / 4 items when every leaf is cut
        rng = np.random.default_rng(n)
        k = int(np.ceil(np.sqrt(n)))
        at = np.stack(np.meshgrid(np.arange(k), np.arange(k)), -1).reshape(-1, 2)[:n]
        xy = ((at + 0.5) / k + rng.uniform(-0.1, 0.1, (n, 2)) / k).astype(np.float32)
        ids = np.arange(n, dtype=np.uint32)
        rects = workloads.squares_around(xy[rng.permutation(n)], 1.2 / k)
        want, _ = oracle.join_grid(oracle_state(n, [(ids, xy)]), rects, cell_side=4.0 / k)
        idx = mqr.Index(leaf_cap=4, max_objects=n, covering=False)
        idx.apply_updates(to_dev(ids, dev), to_dev(xy, dev))
        for blocks in (1, 2, 8):
            idx.set_launch_config(filter=blocks)
            _, offs = idx.tick(to_dev(rects, dev), kind="count")
            np.testing.assert_array_equal(offs.cpu().numpy().view(np.uint64), want)
            s, w = idx.stats(), blocks * warps
            items, words = s["n_filter_items"], s["n_bitmap_words"]
            seen.add(1 if items <= w else 4 if items >= 4 * w and words < 16 * items else 2)
        idx.close()
    assert seen == {1, 2, 4}
