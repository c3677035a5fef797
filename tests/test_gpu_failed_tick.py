"""What a context does after a tick that failed: its records are not there to be
read, whichever allocation of the growth failed, and the next tick is exact."""
import numpy as np
import pytest

import oracle
from paper_1411_3212_gb300 import workloads
from tests.gpu_util import assert_same_csr, gpu_csr_sorted, oracle_state, to_dev, torch_dev

pytestmark = pytest.mark.gpu


@pytest.fixture
def hooks():
    yield
    from paper_1411_3212_gb300 import mqr
    mqr.mqr_debug_fail_allocation(-1)
    mqr.mqr_debug_stall_scan(False)


def world(n, q, side, seed):
    rng = np.random.default_rng(seed)
    xy = rng.random((n, 2)).astype(np.float32)
    ids = np.arange(n, dtype=np.uint32)
    rects = workloads.squares_around(rng.random((q, 2)).astype(np.float32), side)
    return ids, xy, rects, oracle.join_grid(oracle_state(n, [(ids, xy)]), rects, cell_side=0.02)


def index(mqr, ids, xy, dev):
    idx = mqr.Index(leaf_cap=32, max_objects=len(ids))
    idx.apply_updates(to_dev(ids, dev), to_dev(xy, dev))
    return idx


def test_records_of_a_timed_out_tick_are_not_read(hooks):
    torch, dev = torch_dev()
    from paper_1411_3212_gb300 import mqr
    ids, xy, rects, want = world(20_000, 8_000, 0.02, 2)
    idx = index(mqr, ids, xy, dev)
    rd = to_dev(rects, dev)
    assert_same_csr(gpu_csr_sorted(idx, rects, dev), want)
    assert idx.footprint()["tested_leaves"] > 0
    out = torch.empty(2 * int(want[0][-1]) + 2048, dtype=torch.int32, device=dev)
    mqr.mqr_debug_stall_scan(True)
    status, _ = mqr.mqr_tick(idx.ctx, rd, len(rects), mqr.MQR_OUT_PAIRS, out, out.numel() * 4, check=False)
    assert status == mqr.MQR_ERR_TIMEOUT
    for read in (idx.footprint, lambda: idx.region_work(rd, 2)):
        with pytest.raises(mqr.MqrError) as exc:
            read()
        assert exc.value.status == mqr.MQR_ERR_INVALID_ARG
    assert_same_csr(gpu_csr_sorted(idx, rects, dev), want)
    assert idx.footprint()["tested_leaves"] > 0
    idx.close()


def test_every_allocation_of_a_growing_tick_may_fail(hooks):
    """The n-th allocation after a small tick fails, for every n: the tick reports it, and the next one is exact."""
    torch, dev = torch_dev()
    from paper_1411_3212_gb300 import mqr
    ids, xy, rects, want = world(20_000, 30_000, 0.05, 2)
    failed = 0
    for first in (False, True):                     # the context's first tick, and one whose buffers grow
        for after in range(40):
            idx = index(mqr, ids, xy, dev)
            if not first:
                idx.tick(to_dev(rects[:100], dev), kind="count")
            mqr.mqr_debug_fail_allocation(after)
            try:
                idx.tick(to_dev(rects, dev), kind="count")
                done = True
            except mqr.MqrError as e:
                assert e.status == mqr.MQR_ERR_OOM
                done = False
            mqr.mqr_debug_fail_allocation(-1)
            if not done:
                failed += 1
                if not first:                       # nothing of the failed tick is read
                    try:
                        idx.footprint()
                    except mqr.MqrError as e:
                        assert e.status == mqr.MQR_ERR_INVALID_ARG
            _, offs = idx.tick(to_dev(rects, dev), kind="count")
            np.testing.assert_array_equal(offs.cpu().numpy().view(np.uint64), want[0])
            idx.close()
            if done:
                break
    assert failed > 20
