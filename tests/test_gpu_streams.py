"""Inputs that torch's stream has yet to write when a call takes them: the
call's work comes behind the write and before the memory's next use."""
import numpy as np
import pytest

from tests.gpu_util import torch_dev

pytestmark = pytest.mark.gpu

N = 50_000
DELAY = 20_000_000                     # clock cycles: about 10 ms


def late(torch, t):
    """A tensor that holds t once the current stream gets there, zeros before."""
    out = torch.zeros_like(t)
    torch.cuda.synchronize()
    torch.cuda._sleep(DELAY)
    out.copy_(t)
    return out


def inputs(torch, dev, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    ids = torch.arange(N, dtype=torch.int32, device=dev)
    xy = torch.rand(N, 2, generator=g, device=dev)
    corner = torch.rand(2000, 2, generator=g, device=dev)
    rects = torch.cat([corner, corner + 0.02], 1).contiguous()
    inside = (xy[None, :, 0] >= rects[:, None, 0]) & (xy[None, :, 0] <= rects[:, None, 2])
    inside &= (xy[None, :, 1] >= rects[:, None, 1]) & (xy[None, :, 1] <= rects[:, None, 3])
    counts = inside.sum(1)
    torch.cuda.synchronize()
    return ids, xy, rects, counts.cpu().numpy()


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("side_stream", [False, True])
def test_calls_follow_the_current_stream(graph, side_stream):
    torch, dev = torch_dev()
    from paper_1411_3212_gb300 import mqr
    stream = torch.cuda.Stream() if side_stream else torch.cuda.default_stream()
    with torch.cuda.stream(stream):
        idx = mqr.Index(leaf_cap=32, max_objects=N)
        assert idx.stream == stream
        idx.set_graph(graph)
        for seed in range(3):
            ids, xy, rects, counts = inputs(torch, dev, seed)
            a, b = late(torch, ids), late(torch, xy)
            idx.apply_updates(a, b)
            del a, b                                           # the memory's next user writes it later
            for _ in range(4):
                torch.empty(N, dtype=torch.int32, device=dev).fill_(-1)
                torch.empty(N, 2, device=dev).fill_(-1.0)
            _, offs = idx.tick(late(torch, rects), kind="count")
            np.testing.assert_array_equal(np.diff(offs.cpu().numpy()), counts)
        idx.close()


@pytest.mark.parametrize("own_stream", [False, True])
def test_slot_joins_follow_the_current_stream(own_stream):
    torch, dev = torch_dev()
    from paper_1411_3212_gb300 import mqr
    idx = mqr.Index(leaf_cap=32, max_objects=N)
    slots = [idx.slot(torch.cuda.default_stream() if own_stream and k else None) for k in range(2)]
    for seed in range(3):
        ids, xy, rects, counts = inputs(torch, dev, seed)
        want = np.concatenate([[0], np.cumsum(counts)])
        a, b = late(torch, ids), late(torch, xy)
        idx.apply_updates(a, b)
        idx.snapshot()
        del a, b
        outs = []
        for s in slots:
            out = torch.empty(2 * int(want[-1]), dtype=torch.int32, device=dev)
            offs = torch.empty(len(want), dtype=torch.int64, device=dev)
            s.begin(late(torch, rects), "pairs", out, out.numel() * 4, offs)
            outs.append(offs)
            del out, offs                                      # the queries and the output have no other owner
            for _ in range(4):
                torch.empty(2000, 4, device=dev).fill_(-1.0)
                torch.empty(2 * int(want[-1]), dtype=torch.int32, device=dev).fill_(-1)
        for s, offs in zip(slots, outs):
            pairs = s._tensors[1]
            assert s.end() == (2000, int(want[-1])) and s._tensors is None
            np.testing.assert_array_equal(offs.cpu().numpy(), want)
            q = pairs.cpu().numpy().reshape(-1, 2)[:, 0]
            np.testing.assert_array_equal(np.bincount(q, minlength=2000), counts)
    for s in slots:
        s.close()
    idx.close()


def test_settings_do_not_depend_on_the_default_stream():
    """A model and a context's settings while torch's default stream is busy: the first is all zeros until
    it is given parameters, and both behave as they do with an idle one."""
    torch, dev = torch_dev()
    from paper_1411_3212_gb300 import mqr
    rng = np.random.default_rng(3)
    X, y = rng.uniform(-1, 1, (40, 5)).astype(np.float32), rng.uniform(-1, 1, 40).astype(np.float32)
    got = []
    for busy in (False, True):
        blocks = [torch.full((1 << 16,), 7.0, device=dev) for _ in range(64)]      # memory that is not zero
        del blocks
        torch.cuda.empty_cache()
        torch.cuda.synchronize()
        if busy:
            torch.cuda._sleep(DELAY)
        m = mqr.CostModel()
        first = m.predict(X)
        p = rng.standard_normal(m.P).astype(np.float32) * 0.1 if not busy else got[0][2]
        m.set_params(p)
        loss = m.train(X, y, epochs=3, lr=1e-2)
        got.append((first, loss, p, m.params()))
        m.close()
    assert not got[0][0].any() and not got[1][0].any()
    assert got[0][1] == got[1][1]
    np.testing.assert_array_equal(got[0][3], got[1][3])
