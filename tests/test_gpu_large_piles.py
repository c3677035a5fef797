"""Ticks whose bitmap words pass 2^30 (exact) and 2^32 (refused before the
filter runs): piles of objects in one cell cut by many queries."""
import numpy as np
import pytest

from tests.gpu_util import to_dev, torch_dev

pytestmark = pytest.mark.gpu

PILE, REST = 4_000_000, 20_000


def inside(xy, r):
    return int(np.count_nonzero((xy[:, 0] >= r[0]) & (xy[:, 0] <= r[2]) & (xy[:, 1] >= r[1]) & (xy[:, 1] <= r[3])))


def test_words_beyond_30_and_32_bits():
    torch, dev = torch_dev()
    from paper_1411_3212_gb300 import mqr
    rng = np.random.default_rng(3)
    rest = rng.random((REST, 2)).astype(np.float32)
    p = np.float32(0.0010)                                # early in Morton order: most leaves follow the pile's
    xy = torch.full((PILE + REST, 2), float(p), dtype=torch.float32, device=dev)
    xy[PILE:] = to_dev(rest, dev)
    idx = mqr.Index(leaf_cap=16, max_objects=PILE + REST, covering=False)
    idx.apply_updates(torch.arange(PILE + REST, dtype=torch.int32, device=dev), xy)
    eps = np.float32(1e-6)                                # far less than a cell (3e-5): both kinds meet the pile's leaf
    kinds = np.array([[p, p, 0.4, 0.3], [p + eps, p, 0.3, 0.4], [p, p, p, p]], np.float32)
    others = rng.random((500, 2)).astype(np.float32) * np.float32(0.9)
    others = np.concatenate([others, others + np.float32(0.05)], 1).astype(np.float32)

    def tick(q):
        rects = np.concatenate([kinds[np.arange(q) % 3], others])
        offs = torch.full((len(rects) + 1,), -1, dtype=torch.int64, device=dev)
        st, n = mqr.mqr_tick(idx.ctx, to_dev(rects, dev), len(rects), mqr.MQR_OUT_COUNT, None, 0, offs)
        return rects, st, n, offs.cpu().numpy()

    pile_point = np.array([[p, p]], np.float32)
    counts = [inside(rest, r) + PILE * inside(pile_point, r) for r in np.concatenate([kinds, others])]
    assert counts[0] > PILE and 0 < counts[1] < REST and counts[2] == PILE

    def check(q):
        _, st, n, offs = tick(q)
        want = np.array([counts[k % 3] for k in range(q)] + counts[3:], np.int64)
        assert st == mqr.MQR_OK and n == want.sum()
        np.testing.assert_array_equal(np.diff(offs), want)
        return idx.stats()["n_bitmap_words"]

    assert check(300) < 2 ** 30
    words = check(9000)
    assert 2 ** 30 < words < 2 ** 32
    with pytest.raises(mqr.MqrError, match="2\\^32"):
        rects = np.concatenate([kinds[np.arange(36_000) % 3], others])
        idx.tick(to_dev(rects, dev), kind="csr")
    assert idx.stats()["n_bitmap_words"] > 2 ** 32
    _, st, _, _ = tick(36_000)
    assert st == mqr.MQR_ERR_CAPACITY
    with pytest.raises(mqr.MqrError):
        idx.footprint()
    check(300)                                            # the context answers on
    idx.close()
