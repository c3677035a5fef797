"""Sorted output kinds at the edges of the per-query list sort: lists that end
at, below and above a warp's and a block's networks, the longest list a block
takes and one more (the radix sort), both layouts, with and without offsets,
first ticks (no list buffer yet) and later ones."""
import numpy as np
import pytest

from tests.gpu_util import to_dev, torch_dev

pytestmark = pytest.mark.gpu


def strips(lengths, n, seed):
    """Objects on a line in random id order and queries over given numbers of them."""
    rng = np.random.default_rng(seed)
    x = ((np.arange(n) + 0.5) / n).astype(np.float32)
    order = rng.permutation(n)
    xy = np.empty((n, 2), np.float32)
    xy[order, 0] = x                                    # object order[k] is the k-th along the line
    xy[:, 1] = 0.5
    rects, want = [], []
    for m in lengths:
        if m == 0:
            rects.append((2.0, 0.0, 3.0, 1.0))
            want.append(np.zeros(0, np.uint32))
            continue
        a = int(rng.integers(0, n - m + 1))
        rects.append((x[a], 0.0, x[a + m - 1], 1.0))
        want.append(np.sort(order[a:a + m]).astype(np.uint32))
    return xy, np.array(rects, np.float32), want


@pytest.mark.parametrize("lengths,n", [
    ([0, 1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 0, 0, 1023, 1024, 1], 40000),
    ([1025, 0, 2047, 2048, 2049, 5, 4096, 4097, 8191, 8192, 8193, 16383, 16384, 40, 12000], 40000),
    ([16384, 16385, 3, 40000, 0, 77], 40000),
    ([4096, 1500, 4095, 9, 3000], 20000),
    ([4096, 1500, 4095, 9, 3000], 20000),
    ([7], 7),
    ([0], 100),
])
@pytest.mark.parametrize("kind", ["csr_sorted", "pairs_sorted"])
def test_lists_of_every_length(lengths, n, kind):
    torch, dev = torch_dev()
    from paper_1411_3212_gb300 import mqr
    xy, rects, want = strips(lengths, n, len(lengths))
    idx = mqr.Index(leaf_cap=64, max_objects=n)
    idx.apply_updates(to_dev(np.arange(n, dtype=np.uint32), dev), to_dev(xy, dev))
    rd = to_dev(rects, dev)
    flat = np.concatenate(want)
    offs_want = np.concatenate([[0], np.cumsum([len(w) for w in want])])
    pairs = np.stack([np.repeat(np.arange(len(want)), [len(w) for w in want]), flat], 1)
    for graph in (False, False, True, True):            # the first tick finds no list buffer
        idx.set_graph(graph)
        res, offs = idx.tick(rd, kind=kind)
        np.testing.assert_array_equal(offs.cpu().numpy(), offs_want)
        np.testing.assert_array_equal(res.cpu().numpy(), pairs if kind == "pairs_sorted" else flat)
    if kind == "pairs_sorted":                          # no offsets asked for, and a buffer one pair too small
        out = torch.full((len(flat) + 1, 2), -1, dtype=torch.int32, device=dev)
        st, cnt = mqr.mqr_tick(idx.ctx, rd, len(want), mqr.MQR_OUT_PAIRS_SORTED, out, 8 * len(flat), None)
        assert st == mqr.MQR_OK and cnt == len(flat)
        np.testing.assert_array_equal(out[:-1].cpu().numpy(), pairs)
        assert int(out[-1].sum()) == -2                 # nothing past the end
        if len(flat) > 1:
            st, cnt = mqr.mqr_tick(idx.ctx, rd, len(want), mqr.MQR_OUT_PAIRS_SORTED, out, 8 * len(flat) - 8, None)
            assert st == mqr.MQR_ERR_CAPACITY and cnt == len(flat)
    idx.close()
