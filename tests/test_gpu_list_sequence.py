"""Sorted output kinds over ticks whose lists change: what a tick keeps for the
next (the list buffer, whether it had long lists) never shows in the results."""
import numpy as np
import pytest

from tests.gpu_util import to_dev, torch_dev
from tests.test_gpu_list_sort import strips

pytestmark = pytest.mark.gpu

N = 60_000
SHORT, LONG = [3, 0, 200, 1000, 64], [5000, 7, 4097, 16384, 0, 4096]
LONGER, NONE = [16385, 12, 60_000, 300], []
MANY = [900] * 70


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("kind", ["csr_sorted", "pairs_sorted"])
@pytest.mark.parametrize("order", [
    [SHORT, LONG, LONG, NONE, LONG, LONGER, SHORT, LONGER, LONG, MANY, NONE, SHORT],
    [LONG, LONG, NONE, NONE, SHORT, NONE, LONGER, NONE, LONG, SHORT, LONG],
    [NONE, LONGER, MANY, LONG, SHORT, MANY],
])
def test_lists_that_change(order, kind, graph):
    torch, dev = torch_dev()
    from paper_1411_3212_gb300 import mqr
    idx = mqr.Index(leaf_cap=64, max_objects=N)
    idx.set_graph(graph)
    xy = strips([], N, 11)[0]                      # the same positions for every set of lists of this seed
    idx.apply_updates(to_dev(np.arange(N, dtype=np.uint32), dev), to_dev(xy, dev))
    for lengths in order:
        xy2, rects, want = strips(lengths, N, 11)
        np.testing.assert_array_equal(xy, xy2)
        flat = np.concatenate(want) if want else np.zeros(0, np.uint32)
        res, offs = idx.tick(to_dev(rects.reshape(-1, 4), dev), kind=kind)
        np.testing.assert_array_equal(offs.cpu().numpy(), np.concatenate([[0], np.cumsum([len(w) for w in want])]))
        got = res.cpu().numpy().view(np.uint32)
        if kind == "pairs_sorted":
            np.testing.assert_array_equal(got[:, 0], np.repeat(np.arange(len(want)), [len(w) for w in want]))
            got = got[:, 1]
        np.testing.assert_array_equal(got, flat)
    idx.close()
