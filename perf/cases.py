"""Performance cases of the repeated-range-query library.

Each case is one pass that a user's program makes again and again: the position
updates of a tick and the tick itself (device buffers, host buffers, join slots,
batched worlds), the allocation-free object sort, and the training and
prediction of the tick-cost model.  Sizes and distributions are those of the
repository's workloads (`paper_1411_3212_gb300/workloads.py`, the tests and the
benchmark); inputs are drawn on the GPU from the seed alone.

A tick's outputs are whole numbers (ids, query indices, offsets) with no
rounding, so `exact` gives values for the cost model's passes only.
"""
import math

import numpy as np
import torch

from paper_1411_3212_gb300 import mqr
from paper_1411_3212_gb300.costmodel import he_uniform_params

BOUNDS = (0.0, 0.0, 1.0, 1.0)
TOP = 1.0 - 2.0 ** -24                 # largest float32 below 1
STEP = 0.0005                          # random-walk step of a moving object
ELEM = {"pairs": 8, "pairs_sorted": 8, "csr": 4, "csr_sorted": 4, "runs": 8, "count": 0}

TICK = {"call": "tick", "world": "uniform", "n": 0, "q": 0, "moved": 0, "side_lo": 0.0, "side_hi": 0.0,
        "hotspots": 0, "sigma_lo": 0.0, "sigma_hi": 0.0, "frac_hot": 0.0, "worlds": 0, "kind": "pairs",
        "leaf_cap": 128, "grid_level": 0, "covering": True, "graph": False, "slots": 0}


def tick_case(**kw):
    c = dict(TICK, **kw)
    c["moved"] = c["moved"] or c["n"]
    return c


def listed():
    return [
        # the smallest call: a few thousand objects, sorted id lists, plain launches; latency alone
        tick_case(name="tick-4k-csr-sorted", n=4096, q=256, side_lo=0.02, side_hi=0.02, leaf_cap=64, kind="csr_sorted"),
        # the small configuration (16,384 objects, 1,024 queries), replayed as a graph by a steady tick loop
        tick_case(name="uniform-16k-pairs", n=16384, q=1024, side_lo=0.01, side_hi=0.01, leaf_cap=64, graph=True),
        # an ordinary uniform population of which a third moved since the last tick, in arrival order
        # with repeated ids; id lists with offsets, plain launches
        tick_case(name="uniform-1m-csr", n=1_000_000, q=100_000, moved=333_333, side_lo=0.002, side_hi=0.002,
                  kind="csr"),
        # the uniform-grid index, counting results only (density monitoring)
        tick_case(name="uniform-1m-grid-count", n=1_000_000, q=100_000, side_lo=0.002, side_hi=0.002, kind="count",
                  grid_level=8, graph=True),
        # a skewed population of odd size, answered as pairs in (query, id) order
        hotspot(name="hotspot-1m-pairs-sorted", n=1_000_003, q=99_991, kind="pairs_sorted"),
        # the largest skewed tick: 4,000,000 objects, 400,000 queries, every pair written
        hotspot(name="hotspot-4m-pairs", n=4_000_000, q=400_000, graph=True),
        # 256 independent worlds of 1,000 to 262,144 objects answered as one tick
        tick_case(name="worlds-256-pairs", world="worlds", worlds=256, n=256, q=0, side_lo=0.003, side_hi=0.003,
                  hotspots=8, sigma_lo=0.01, sigma_hi=0.01, frac_hot=0.9, graph=True),
        # a served stream's tick: 10,000,000 objects, the queries of 10 ms split over two join slots,
        # covering-compressed output
        served(name="served-10m-runs-slots", n=10_000_000, q=100_000, slots=2),
        # host buffers in and out: updates and queries copied to the device, id lists copied back
        tick_case(name="host-1m-csr", call="host", n=1_000_000, q=100_000, side_lo=0.002, side_hi=0.002, kind="csr"),
        # the allocation-free sort of an embedder that owns all device memory
        {"name": "noalloc-200k", "call": "sort", "n": 200_000},
        # retraining of the per-tick index chooser on its logged ticks
        {"name": "train-80", "call": "train", "n": 80, "epochs": 400},
        # retraining of the per-region chooser on its full sample window
        {"name": "train-4096", "call": "train", "n": 4096, "epochs": 100},
    ]


def hotspot(**kw):
    return tick_case(**dict(dict(world="hotspot", side_lo=0.0005, side_hi=0.005, hotspots=64, sigma_lo=0.002,
                                 sigma_hi=0.02, frac_hot=0.9), **kw))


def served(**kw):
    return tick_case(**dict(dict(world="hotspot", side_lo=0.0005, side_hi=0.004, hotspots=16, sigma_lo=0.005,
                                 sigma_hi=0.005, frac_hot=0.95, kind="runs"), **kw))


def log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    what = rng.choice(["tick"] * 6 + ["served", "worlds", "host", "sort", "train", "predict"])
    if what == "sort":
        return {"call": "sort", "n": int(log_uniform(rng, 5, mqr.MQR_NOALLOC_MAX_OBJECTS))}
    if what == "train":
        n = int(log_uniform(rng, 8, 4096))
        return {"call": "train", "n": n, "epochs": rng.choice([1, 20, 100, 400]) if n < 1024 else rng.choice([1, 20, 100])}
    if what == "predict":
        return {"call": "predict", "n": int(log_uniform(rng, 4, 4096)), "epochs": 0}
    n = int(log_uniform(rng, 1000, 4_000_000))
    q = max(1, int(n * log_uniform(rng, 0.01, 0.1)))
    leaf_cap = rng.choice([32, 64, 128, 128, 256, 512])
    moved = rng.choice([n, n, max(1, int(n * log_uniform(rng, 0.01, 1.0)))])
    if what == "worlds":
        w = int(log_uniform(rng, 2, 256))
        return tick_case(world="worlds", worlds=w, n=w, side_lo=0.003, side_hi=0.003, hotspots=8, sigma_lo=0.01,
                         sigma_hi=0.01, frac_hot=0.9, kind=rng.choice(["pairs", "csr"]), leaf_cap=leaf_cap,
                         graph=rng.choice([True, False]))
    if what == "served":
        n = int(log_uniform(rng, 200_000, 10_000_000))
        return served(n=n, q=int(log_uniform(rng, 1000, 100_000)), slots=rng.choice([0, 0, 1, 2]),
                      kind=rng.choice(["runs", "runs", "csr"]))
    side = min(0.1, math.sqrt(log_uniform(rng, 0.5, 100.0) / n))       # 0.5 to 100 results of a query at the mean density
    if what == "host":
        n = min(n, 2_000_000)
        return tick_case(call="host", n=n, q=max(1, min(q, n // 10)), side_lo=side, side_hi=side, leaf_cap=leaf_cap,
                         kind=rng.choice(["csr", "pairs", "count"]))
    kind = rng.choice(["pairs", "pairs", "csr", "runs", "count", "csr_sorted", "pairs_sorted", "bitmap"])
    grid = rng.choice([0, 0, 0, max(1, min(9, int(math.log(n / 32, 4))))])
    covering = rng.choice([True, True, True, False])
    graph = rng.choice([True, False])
    if kind == "bitmap":
        q = max(1, min(q, 2 ** 31 // n))                                # at most 256 MB of words
    if rng.random() < 0.5:
        c = hotspot(n=n, q=q, moved=moved, kind=kind, leaf_cap=leaf_cap, covering=covering, graph=graph)
        if kind in ("csr_sorted", "pairs_sorted"):                      # at most 32M sorted results
            c["q"] = max(1, min(q, int(3.2e7 * q / max(results(c), 1.0))))
        return c
    return tick_case(n=n, q=q, moved=moved, side_lo=side, side_hi=side, kind=kind, leaf_cap=leaf_cap, grid_level=grid,
                     covering=covering, graph=graph)


# -- inputs ---------------------------------------------------------------------
def world_sizes(c):
    """Objects of every world: the quantiles of the log-uniform sizes 1,000 to 262,144."""
    w = c["worlds"]
    return [int(1000 * 262.144 ** ((k + 0.5) / w)) for k in range(w)]


def generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def log_uniform_t(g, n, lo, hi):
    return torch.exp(math.log(lo) + rand(g, n) * (math.log(hi) - math.log(lo)))


def clamp(xy):
    return xy.clamp_(0.0, TOP).to(torch.float32)


def positions(c, g, n):
    if c["world"] != "hotspot":
        return clamp(rand(g, n, 2))
    centres, sigmas = rand(g, c["hotspots"], 2), log_uniform_t(g, c["hotspots"], c["sigma_lo"], c["sigma_hi"])
    member = torch.randint(c["hotspots"], (n,), generator=g, device="cuda")
    hot = (rand(g, n) < c["frac_hot"]).unsqueeze(1)
    return clamp(torch.where(hot, centres[member] + randn(g, n, 2) * sigmas[member].unsqueeze(1), rand(g, n, 2)))


def squares(g, xy, lo, hi):
    """Closed squares around the issuing objects, sides log-uniform, corners rounded as the generators round them."""
    h = (log_uniform_t(g, xy.shape[0], lo, hi) / 2).to(torch.float32).unsqueeze(1)
    return torch.cat([xy - h, xy + h], 1).contiguous()


def world_inputs(c, g):
    """Objects and queries of all worlds in order, and their ranges; every second world is a hotspot walk."""
    sizes = world_sizes(c)
    sizes = [sizes[i] for i in torch.randperm(len(sizes), generator=torch.Generator().manual_seed(g.initial_seed())).tolist()]
    nq = [max(1, n // 10) for n in sizes]
    obj_base, q_base = (np.concatenate([[0], np.cumsum(v)]).astype(np.uint32) for v in (sizes, nq))
    w = torch.arange(len(sizes), device="cuda")
    wo, wq = (torch.repeat_interleave(w, torch.tensor(v, device="cuda")) for v in (sizes, nq))
    n = int(obj_base[-1])
    centres = rand(g, len(sizes) * c["hotspots"], 2)
    member = wo * c["hotspots"] + torch.randint(c["hotspots"], (n,), generator=g, device="cuda")
    hot = ((rand(g, n) < c["frac_hot"]) & (wo % 2 == 1)).unsqueeze(1)
    xy = clamp(torch.where(hot, centres[member] + randn(g, n, 2) * c["sigma_lo"], rand(g, n, 2)))
    base = torch.tensor(obj_base.astype(np.int64), device="cuda")
    iss = base[wq] + (rand(g, wq.shape[0]) * torch.tensor(sizes, device="cuda")[wq]).long()
    return xy, squares(g, xy[iss], c["side_lo"], c["side_hi"]), obj_base, q_base


def samples(c, seed):
    """Logged (features, log time) samples of a chooser, and the model's first parameters."""
    rng = np.random.default_rng(seed)
    x = rng.uniform(-1.0, 1.0, (c["n"], 5)).astype(np.float32)
    y = 0.5 * x[:, 0] - x[:, 1] ** 2 + 0.3 * x[:, 2] * x[:, 3] + 0.1 + 0.05 * rng.normal(size=c["n"])
    return x, y.astype(np.float32), he_uniform_params(seed % (1 << 31))


# -- what a program has in hand before the call -----------------------------------
def prepare(c, seed):
    if c["call"] in ("train", "predict"):
        x, y, p = samples(c, seed)
        return {"c": c, "x": x, "y": y, "p": p, "model": mqr.CostModel(p)}
    g = generator(seed)
    if c["call"] == "sort":
        n = c["n"]
        out = [torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2)]
        return {"c": c, "xy": positions({"world": "hotspot", "hotspots": 8, "sigma_lo": 0.002, "sigma_hi": 0.02,
                                         "frac_hot": 0.9}, g, n), "out": out}
    s = {"c": c}
    obj_base = None
    if c["world"] == "worlds":
        xy, s["rects"], obj_base, q_base = world_inputs(c, g)
        n = xy.shape[0]
    else:
        n = c["n"]
        xy = positions(c, g, n)
        iss = torch.randint(n, (c["q"],), generator=g, device="cuda").sort().values
        s["rects"] = squares(g, xy[iss], c["side_lo"], c["side_hi"])
    kind = mqr.MQR_INDEX_UNIFORM_GRID if c["grid_level"] else mqr.MQR_INDEX_QUADTREE
    idx = s["idx"] = mqr.Index(BOUNDS, leaf_cap=c["leaf_cap"], max_objects=n, index_kind=kind,
                               grid_level=c["grid_level"] or 8, covering=c["covering"])
    ids = torch.arange(n, dtype=torch.int32, device="cuda")
    idx.apply_updates(ids, xy)                              # the population before the tick
    if obj_base is not None:
        idx.set_worlds(obj_base)
        idx.set_query_worlds(q_base)
    if c["graph"]:
        idx.set_graph(True)
    if c["world"] != "worlds" and c["moved"] < n:           # a part of the objects, in arrival order, with repeats
        ids = torch.randint(n, (c["moved"],), generator=g, device="cuda", dtype=torch.int32)
        xy = clamp(xy[ids.long()].double() + STEP * randn(g, c["moved"], 2))
    s["ids"], s["xy"] = ids, xy
    if c["call"] == "host":
        def pinned(t, dtype):
            return t.cpu().pin_memory().numpy().view(dtype)
        s["ids"], s["xy"], s["rects"] = pinned(ids, np.uint32), pinned(xy, np.float32), pinned(s["rects"], np.float32)
        s["out"] = pinned(torch.zeros(out_words(c), dtype=torch.int32), np.uint32)
        s["offs"] = pinned(torch.zeros(c["q"] + 1, dtype=torch.int64), np.uint64)
        return s
    if c["world"] == "hotspot" and c["frac_hot"] == 0.95:   # served: bounded output memory per slot or tick
        k = max(1, c["slots"])
        s["slots"] = [idx.slot() for _ in range(c["slots"])]
        s["out"] = [torch.zeros((1 << 31) // 4 // k, dtype=torch.int32, device="cuda") for _ in range(k)]
        s["cut"] = [c["q"] * i // k for i in range(k + 1)]
        s["offs"] = [torch.zeros(s["cut"][i + 1] - s["cut"][i] + 1, dtype=torch.int64, device="cuda") for i in range(k)]
        torch.cuda.synchronize()                            # the slots' streams start after these
    else:
        s["out"] = torch.zeros(out_words(c), dtype=torch.int32, device="cuda")
        s["offs"] = torch.zeros(s["rects"].shape[0] + 1, dtype=torch.int64, device="cuda")
    return s


def out_words(c):
    """32-bit words of the output buffer: the whole bitmap, or twice the expected results (their number varies with
    the hotspots' spread); a program keeps one buffer for all its ticks."""
    if c["kind"] == "bitmap":
        return c["q"] * ((c["n"] + 31) // 32)
    return ELEM[c["kind"]] // 4 * (int(2.0 * results(c)) + 65536)


# -- one pass ---------------------------------------------------------------------
def run(s):
    c = s["c"]
    if c["call"] == "train":
        s["model"].set_params(s["p"])
        loss = s["model"].train(s["x"], s["y"], c["epochs"], 3e-3)
        return {"params": s["model"].params(), "loss": np.float32(loss)}
    if c["call"] == "predict":
        return {"y": s["model"].predict(s["x"])}
    if c["call"] == "sort":
        mqr.mqr_sort_objects_noalloc(BOUNDS, s["xy"], c["n"], s["out"][0], s["out"][1],
                                     torch.cuda.current_stream().cuda_stream)
        return s["out"]
    if c["call"] == "host":
        return run_host(s)
    idx = s["idx"]
    idx.apply_updates(s["ids"], s["xy"])
    if "cut" in s:
        return run_served(s)
    rects, out = s["rects"], s["out"] if c["kind"] != "count" else None
    st, n = mqr.mqr_tick(idx.ctx, rects, rects.shape[0], mqr.KINDS[c["kind"]], out, s["out"].numel() * 4, s["offs"])
    return answer(st, n, out, s["offs"])


def answer(st, n, out, offs):
    """A tick's status, count and buffers (words past the count are the caller's own)."""
    if st != mqr.MQR_OK:
        raise mqr.MqrError(st, mqr.mqr_last_error())
    return {"n": n, "offsets": offs} if out is None else {"n": n, "out": out, "offsets": offs}


def run_host(s):
    c = s["c"]
    mqr.mqr_apply_updates_host(s["idx"].ctx, s["ids"], s["xy"])
    kind = mqr.KINDS[c["kind"]]
    st, n = mqr.mqr_tick_host(s["idx"].ctx, s["rects"], c["q"], kind, s["out"], s["out"].nbytes, s["offs"])
    return answer(st, n, s["out"] if c["kind"] != "count" else None, s["offs"].view(np.int64))


def run_served(s):
    c, idx = s["c"], s["idx"]
    kind, got = mqr.KINDS[c["kind"]], []
    if not s["slots"]:
        got.append(mqr.mqr_tick_admit(idx.ctx, s["rects"], c["q"], kind, s["out"][0], s["out"][0].numel() * 4,
                                      s["offs"][0]))
    else:
        idx.snapshot()
        for i, slot in enumerate(s["slots"]):
            slot.begin(s["rects"][s["cut"][i]:s["cut"][i + 1]], kind, s["out"][i], s["out"][i].numel() * 4, s["offs"][i])
        got = [slot.end() for slot in s["slots"]]
    return [{"admitted": a, "n": m, "out": s["out"][i], "offsets": s["offs"][i]} for i, (a, m) in enumerate(got)]


# -- work and exact values ----------------------------------------------------------
def near(sigma, lo, hi):
    """Chance that another member of a Gaussian hotspot lies in the square around a member, over the sides' range."""
    k = 16
    sides = [lo * (hi / lo) ** ((i + 0.5) / k) for i in range(k)]
    return sum(math.erf(s / (4.0 * sigma)) ** 2 for s in sides) / k


def area(lo, hi):
    return lo * lo if hi <= lo else (hi * hi - lo * lo) / (2.0 * math.log(hi / lo))


def per_query(c, n, hot):
    r = 1.0 + n * area(c["side_lo"], c["side_hi"])
    if hot:
        k = 16
        sig = [c["sigma_lo"] * (c["sigma_hi"] / c["sigma_lo"]) ** ((i + 0.5) / k) for i in range(k)]
        r += c["frac_hot"] ** 2 * n / c["hotspots"] * sum(near(x, c["side_lo"], c["side_hi"]) for x in sig) / k
    return r


def results(c):
    """Expected results of a tick."""
    if c["world"] == "worlds":
        return sum(max(1, n // 10) * per_query(c, n, i % 2 == 1) for i, n in enumerate(world_sizes(c)))
    return c["q"] * per_query(c, c["n"], c["world"] == "hotspot")


def work(c):
    n = c["n"]
    if c["call"] in ("train", "predict"):
        macs = 5 * 64 + 64 * 64 + 64
        p = macs + 64 + 64 + 1
        if c["call"] == "predict":
            return {"bytes": 4.0 * (5 * n + n + p), "flops": 2.0 * macs * n}
        return {"bytes": 4.0 * (6 * n + 2 * p), "flops": (6.0 * macs * n + 12.0 * p) * c["epochs"]}
    if c["call"] == "sort":
        return {"bytes": 16.0 * n, "flops": 0.0}
    q, moved = c["q"], c["moved"]
    if c["world"] == "worlds":
        n = moved = sum(world_sizes(c))
        q = sum(max(1, k // 10) for k in world_sizes(c))
    r = results(c)
    if c["kind"] == "bitmap":
        out = 4.0 * q * ((n + 31) // 32)
    elif c["kind"] == "runs":
        out = 8.0 * 0.3 * r                                  # about a third of the results are not in covering runs
    else:
        out = float(ELEM[c["kind"]]) * r
    # updates in (id, position), the population's positions, queries in, results and offsets out
    return {"bytes": 12.0 * moved + 8.0 * n + 16.0 * q + out + 8.0 * (q + 1), "flops": 0.0}


def exact(c, seed):
    if c["call"] not in ("train", "predict"):
        return None
    x, y, p = (a.astype(np.float64) for a in samples(c, seed))
    m, v = np.zeros_like(p), np.zeros_like(p)
    loss = 0.0
    for t in range(1, max(1, c["epochs"]) + 1):
        w1, b1, w2, b2, w3, b3 = np.split(p, np.cumsum([320, 64, 4096, 64, 64]))
        w1, w2 = w1.reshape(64, 5), w2.reshape(64, 64)
        h1 = np.maximum(x @ w1.T + b1, 0.0)
        h2 = np.maximum(h1 @ w2.T + b2, 0.0)
        o = h2 @ w3 + b3[0]
        if c["call"] == "predict":
            return {"y": o}
        e = o - y
        loss = np.mean(e * e)
        d = (2.0 / len(y)) * e
        d2 = np.where(h2 > 0.0, d[:, None] * w3, 0.0)
        d1 = np.where(h1 > 0.0, d2 @ w2, 0.0)
        g = np.concatenate([(d1.T @ x).ravel(), d1.sum(0), (d2.T @ h1).ravel(), d2.sum(0), d @ h2, [d.sum()]])
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        p = p - 3e-3 * (m / (1.0 - 0.9 ** t)) / (np.sqrt(v / (1.0 - 0.999 ** t)) + 1e-8)
    return {"params": p, "loss": loss}
