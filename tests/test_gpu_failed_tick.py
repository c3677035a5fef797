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
    from paper_1411_3212_gb300 import mqr
    torch, dev = torch_dev()
    rng = np.random.default_rng(seed)
    xy = rng.random((n, 2)).astype(np.float32)
    ids = np.arange(n, dtype=np.uint32)
    idx = mqr.Index(leaf_cap=32, max_objects=n)
    idx.apply_updates(to_dev(ids, dev), to_dev(xy, dev))
    rects = workloads.squares_around(rng.random((q, 2)).astype(np.float32), side)
    return mqr, torch, dev, idx, rects, oracle.join_grid(oracle_state(n, [(ids, xy)]), rects, cell_side=0.02)


def test_records_of_a_timed_out_tick_are_not_read(hooks):
    mqr, torch, dev, idx, rects, want = world(20_000, 8_000, 0.02, 2)
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
