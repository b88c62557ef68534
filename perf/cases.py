"""What this framework is measured on: contraction-hierarchy builds, s-t
queries, one-to-many and one-to-all distances, core tables, the query server
and the training of the learned priority, each through the public entry points
of ``paper_2412_18008_gb300.ch``.

Graphs are made on the device from the seed: geometric 3-nearest-neighbour
graphs with road-like weights (uniform points, 5% one-way edges, speed factors
1, 2, 4) and RMAT graphs (a = 0.57, b = c = 0.19, 16 edge samples per vertex,
weights 1-1000); perturbed grids come from the package's own host generator.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2412_18008_gb300 import ch
from paper_2412_18008_gb300 import inputs as I

# Build options of the power-law graphs: candidate bound (leaves a core),
# two-hop witnesses with a ball and a level-work bound, memoised distances.
RMAT = dict(hop_limit=2, max_candidates_per_vertex=256, witness_ball_limit=256,
            witness_level_work=1024, witness_memo_limit=1 << 30)


def listed():
    return [
        # A small road-like grid handed over as host arrays, built and read
        # back whole: the smallest build, where launches and host work count.
        dict(name="build_grid_64x64", kind="build_grid", rows=64, cols=64),
        # The headline: preprocessing of a road-like network of a million
        # vertices that is already in device memory.
        dict(name="build_geo_1M", kind="build", graph="geo", n=1_000_000, mode="plain"),
        # The same with the trained network in place of the edge difference,
        # at the size of its training graphs.
        dict(name="build_learned_geo_256K", kind="build", graph="geo", n=256_000, mode="learned"),
        # A power-law graph: hubs, a large candidate volume, memoised witness
        # distances, a core left uncontracted.
        dict(name="build_rmat_2e17", kind="build", graph="rmat", n=1 << 17, mode="rmat"),
        # One route request: the latency of a single query.
        dict(name="query_1_geo_1M", kind="query", graph="geo", n=1_000_000, mode="plain", k=1, call="device"),
        # A distance-matrix row: one source, a ragged number of targets.
        dict(name="one_to_many_777_geo_256K", kind="one_to_many", graph="geo", n=256_000, mode="plain", k=777),
        # Bulk routing: a million uniform random pairs.
        dict(name="query_1M_geo_1M", kind="query", graph="geo", n=1_000_000, mode="plain", k=1_000_000,
             call="device"),
        # Queries on a power-law hierarchy, which have to search its core.
        dict(name="query_96_rmat_2e15", kind="query", graph="rmat", n=1 << 15, mode="rmat", k=96,
             call="device"),
        # The core's distance table, then a batch of queries through it.
        dict(name="core_table_rmat_2e14", kind="core_table", graph="rmat", n=1 << 14, mode="rmat", k=20_000),
        # Distances from one full pass of sources to every vertex.
        dict(name="one_to_all_64_geo_1M", kind="one_to_all", graph="geo", n=1_000_000, mode="plain", k=64),
        # One epoch of the learned priority's training, minibatches of 8192
        # (a ragged last one), on the contraction trace of a road-like graph.
        dict(name="train_geo_100K", kind="train", n=100_000, batch=8192, epochs=1),
        # The device-resident server: a burst of mixed one-to-one and
        # one-to-many requests (1-1024 targets), all due at once.
        dict(name="serve_80K_geo_256K", kind="serve", graph="geo", n=256_000, mode="plain", targets=80_000),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["build_grid", "build", "build", "build", "query", "query", "query", "one_to_many",
                       "query_core", "core_table", "one_to_all", "train", "serve"])
    n = _log_int(rng, 2_000, 1_000_000)
    hier = rng.choice(["plain", "plain", "composite", "memo"])  # what a query kind's hierarchy is built with
    if kind == "build_grid":
        return dict(kind=kind, rows=_log_int(rng, 8, 96), cols=_log_int(rng, 8, 96))
    if kind == "build":
        mode = rng.choice(["plain", "plain", "learned", "composite", "memo", "prune", "hop3", "settle", "rmat"])
        if mode == "rmat":
            return dict(kind=kind, graph="rmat", n=1 << rng.randint(11, 17), mode=mode)
        return dict(kind=kind, graph="geo", n=min(n, 8_000) if mode == "settle" else n, mode=mode)
    if kind == "query":
        return dict(kind=kind, graph="geo", n=n, mode=hier, k=_log_int(rng, 1, 1_000_000),
                    call=rng.choice(["device", "device", "host", "graph"]))
    if kind == "query_core":
        return dict(kind="query", graph="rmat", n=1 << rng.randint(11, 15), mode="rmat", k=_log_int(rng, 1, 96),
                    call="device")
    if kind == "one_to_many":
        return dict(kind=kind, graph="geo", n=n, mode=hier, k=_log_int(rng, 1, 100_000))
    if kind == "core_table":
        return dict(kind=kind, graph="rmat", n=1 << rng.randint(11, 14), mode="rmat", k=_log_int(rng, 1, 20_000))
    if kind == "one_to_all":
        # rows of n distances: no more of them than the listed case returns
        return dict(kind=kind, graph="geo", n=n, mode=hier, k=_log_int(rng, 1, max(1, min(200, 64_000_000 // n))))
    if kind == "train":
        return dict(kind=kind, n=_log_int(rng, 2_000, 100_000), batch=rng.choice([256, 1000, 8192, 20_000]),
                    epochs=rng.choice([0, 1]))
    return dict(kind="serve", graph="geo", n=min(n, 256_000), mode=hier, targets=_log_int(rng, 250, 80_000))


# ---- inputs ---------------------------------------------------------------

def _csr(n, s, t, w):
    order = torch.argsort(s * n + t, stable=True)
    offsets = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    offsets[1:] = torch.cumsum(torch.bincount(s, minlength=n), 0)
    return dict(n=n, offsets=offsets, targets=t[order].to(torch.int32).contiguous(),
                weights=w[order].to(torch.int32).contiguous())


def _geo(n, gen):
    """Uniform points joined to their 3 nearest within the surrounding cells
    (4 points per cell on average), symmetrised."""
    pts = torch.rand((n, 2), generator=gen, device="cuda", dtype=torch.float64)
    side = max(1, int(math.sqrt(n / 4)))
    cell = (pts * side).long().clamp_(max=side - 1)
    cid = cell[:, 0] * side + cell[:, 1]
    counts = torch.bincount(cid, minlength=side * side)
    cap = int(counts.max())
    order = torch.argsort(cid, stable=True)
    first = torch.cumsum(counts, 0) - counts
    table = torch.full((side * side + 1, cap), -1, dtype=torch.int64, device="cuda")  # last row: outside
    table[cid[order], torch.arange(n, device="cuda") - first[cid[order]]] = order
    step = torch.tensor([(i, j) for i in (-1, 0, 1) for j in (-1, 0, 1)], device="cuda")
    nbrs = []
    for a in range(0, n, 1 << 18):
        b = min(n, a + (1 << 18))
        c = cell[a:b, None, :] + step
        inside = ((c >= 0) & (c < side)).all(-1)
        cand = table[torch.where(inside, c[..., 0] * side + c[..., 1], side * side)].reshape(b - a, -1)
        d2 = ((pts[cand.clamp(min=0)] - pts[a:b, None, :]) ** 2).sum(-1)
        d2[(cand < 0) | (cand == torch.arange(a, b, device="cuda")[:, None])] = math.inf
        d, i = torch.topk(d2, min(3, d2.shape[1]), largest=False)
        nb = torch.gather(cand, 1, i)
        nbrs.append(torch.where(torch.isinf(d), -1, nb))
    nb = torch.cat(nbrs)
    me = torch.arange(n, device="cuda")[:, None].expand_as(nb)
    ok = nb >= 0
    lo, hi = torch.minimum(me[ok], nb[ok]), torch.maximum(me[ok], nb[ok])
    key = torch.unique(lo * n + hi)
    a, b = key // n, key % n
    speed = torch.tensor([1.0, 2.0, 4.0], dtype=torch.float64, device="cuda")[
        torch.randint(0, 3, a.shape, generator=gen, device="cuda")]
    oneway = torch.rand(a.shape, generator=gen, device="cuda") < 0.05
    coin = torch.randint(0, 2, a.shape, generator=gen, device="cuda")
    length = ((pts[a] - pts[b]) ** 2).sum(-1).sqrt()
    w = torch.floor(1000.0 * length * speed + 0.5).long().clamp_(min=1)
    fwd, bwd = ~oneway | (coin == 0), ~oneway | (coin == 1)
    return _csr(n, torch.cat([a[fwd], b[bwd]]), torch.cat([b[fwd], a[bwd]]), torch.cat([w[fwd], w[bwd]]))


def _rmat(n, gen):
    """16 edge samples per vertex; duplicates and self-loops stay."""
    m, scale = 16 * n, n.bit_length() - 1
    u = torch.zeros(m, dtype=torch.int64, device="cuda")
    v = torch.zeros_like(u)
    for _ in range(scale):
        r = torch.rand(m, generator=gen, device="cuda")
        u = 2 * u + (r >= 0.76)
        v = 2 * v + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    return _csr(n, u, v, torch.randint(1, 1001, (m,), generator=gen, device="cuda"))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _graph(case, gen):
    return _rmat(case["n"], gen) if case.get("graph") == "rmat" else _geo(case["n"], gen)


def _network(seed):
    """A priority network of the kind training arrives at: the sum of the
    transformed edge difference and depth (positive and negative parts in
    three hidden units), everything else small."""
    w = 0.05 * ch.mlp_init(seed)
    w1, w2, w3 = w[:768].reshape(12, 64), w[832:4928].reshape(64, 64), w[4992:5056]
    for unit, (feature, sign) in enumerate(((4, 1.0), (4, -1.0), (6, 1.0))):
        w1[feature, unit] += sign
        w2[unit, unit] += 1.0
        w3[unit] += sign
    return w


def _options(mode, seed):
    return {"plain": dict(hop_limit=5), "learned": dict(hop_limit=5, mlp_weights=_network(seed)),
            "composite": dict(hop_limit=5, composite=True), "memo": dict(hop_limit=5, witness_memo_limit=1 << 30),
            "prune": dict(hop_limit=5, witness_memo_limit=1 << 30, witness_prune=True),
            "hop3": dict(hop_limit=3, tie_break=ch.CH_TIE_ID), "settle": dict(witness_settle_cap=100),
            "rmat": RMAT}[mode]


def _ids(n, k, gen):
    return torch.randint(0, n, (k,), generator=gen, device="cuda").to(torch.int32)


def prepare(case, seed):
    kind, gen = case["kind"], _gen(seed)
    if kind == "build_grid":
        return dict(kind=kind, graph=I.grid_graph(case["rows"], case["cols"], 0.10, 1, 100, seed=seed),
                    cells=case["rows"] * case["cols"])
    g = _graph(case, gen)
    if kind == "train":
        with ch.CH.build(**g, hop_limit=5, trace=True) as h:
            rows = torch.from_numpy(h.export_trace()["rows"]).cuda()
        rows = rows[torch.randperm(rows.shape[0], generator=gen, device="cuda")].contiguous()
        return dict(kind=kind, rows=rows, labels=ch.training_labels(rows), batch=case["batch"],
                    epochs=case["epochs"], weights=torch.from_numpy(ch.mlp_init(seed)).cuda())
    opt = _options(case["mode"], seed)
    if kind == "build":
        return dict(kind=kind, graph=g, options=opt)
    n, h = case["n"], ch.CH.build(**g, **opt)
    if kind == "serve":
        # requests until they have that many targets; the last one is cut short
        src, ks, targets = I.request_mix(n, case["targets"], seed)
        ends = np.cumsum(ks.astype(np.int64))
        count = int(np.searchsorted(ends, case["targets"])) + 1
        ks[count - 1] -= ends[count - 1] - case["targets"]
        return dict(kind=kind, ch=h, src=src[:count], ks=ks[:count], targets=targets[:case["targets"]],
                    due=np.zeros(count, np.uint64))
    src, dst = _ids(n, case["k"], gen), _ids(n, case["k"], gen)
    state = dict(kind=kind, ch=h, src=src, dst=dst)
    if kind == "one_to_many":
        state["source"] = int(src[0])
    if case.get("call") == "host":
        state.update(src=src.cpu().numpy().view(np.uint32), dst=dst.cpu().numpy().view(np.uint32))
    if case.get("call") == "graph":
        state["out"] = torch.empty_like(src)
        state["graph"] = h.query_graph(src, dst, state["out"])
    return state


# ---- one pass -------------------------------------------------------------

def _rows(a, count):
    """The array with zero rows up to ``count``: sizes that depend on the
    seed's graph become the same for every seed."""
    out = np.zeros((count,) + a.shape[1:], a.dtype)
    out[:len(a)] = a
    return out


def _summary(h):
    """The counters of the build that do not depend on how it was run, and
    its table of rounds."""
    st = h.stats()
    return dict(counts=np.array([st[k] for k in ("n", "m_input", "rounds", "shortcuts", "up_edges", "down_edges",
                                                 "core_vertices")], np.int64),
                rounds=_rows(h.round_stats().astype(np.int64), 1024))


def _order(h, n):
    """Level, priority and rank of every vertex through the C ABI (the whole
    export also sorts the edge lists on the host, which takes longer than the
    build of a large graph)."""
    out = [np.empty(n, np.int32) for _ in range(3)]
    rc = ch.load().ch_export(h._h, *(a.ctypes.data for a in out), None, None, None)
    if rc:
        raise RuntimeError(f"ch_export: {rc}")
    return dict(zip(("level", "priority", "rank"), out))


def run(state):
    kind = state["kind"]
    if kind == "build_grid":
        with ch.CH.build(state["graph"], hop_limit=5) as h:
            cells = state["cells"]
            out = {k: _rows(v.astype(np.int64), cells if v.ndim == 1 else 8 * cells) for k, v in h.export().items()}
            out.update(_summary(h))
        return out
    if kind == "build":
        with ch.CH.build(**state["graph"], **state["options"]) as h:
            return dict(_order(h, state["graph"]["n"]), **_summary(h))
    if kind == "train":
        w = state["weights"].clone()
        res = ch.mlp_train(state["rows"], state["labels"], w, epochs=state["epochs"], batch=state["batch"])
        return dict(grad=res[0], loss=res[1]) if state["epochs"] == 0 else dict(weights=w, loss=res)
    h = state["ch"]
    if kind == "serve":
        with ch.Server(h, ring=1 << 12, pool=1 << 18, idle_ms=200) as sv:
            return sv.replay(state["src"], state["ks"], state["targets"], state["due"])[0].astype(np.int64)
    if kind == "one_to_many":
        return h.query_one_to_many(state["source"], state["dst"])
    if kind == "one_to_all":
        return h.one_to_all(state["src"])
    if kind == "core_table":
        h.core_table()
    if "graph" in state:
        state["graph"].launch()
        return state["out"]
    out = h.query(state["src"], state["dst"])
    return out if isinstance(out, torch.Tensor) else out.astype(np.int64)


# ---- what a pass cannot do without ----------------------------------------

def _edges(case):
    """Edges of the input graph, about."""
    return 11 * case["n"] if case["graph"] == "rmat" else 3.6 * case["n"]


def work(case):
    """Inputs read once and outputs written once. A query is counted with the
    labels and edges that two upward Dijkstra searches would touch (about 90
    vertices of 10 edges each per direction at 10^5 vertices, growing with the
    fourth root of the size), but no hierarchy is read more than once; a
    relaxation (an addition and a minimum) is two operations."""
    kind = case["kind"]
    if kind == "build_grid":
        n = case["rows"] * case["cols"]
        return {"bytes": 8 * n + 8 * 3.6 * n + 12 * n + 12 * 8 * n, "flops": 2 * 100 * n}
    if kind == "train":
        rows, passes = 3.4 * case["n"], max(1, case["epochs"])
        if case["epochs"] == 0:
            rows = min(rows, case["batch"])
        mul = 12 * 64 + 64 * 64 + 64  # per row: forward, weight gradients, and back through the upper layers
        return {"bytes": rows * (12 * 8 + 4) * passes + 2 * 4 * 5057, "flops": 2.0 * rows * passes * (3 * mul - 12 * 64)}
    n, m = case["n"], _edges(case)
    hier = 2 * (4 * n + 8 * 1.6 * m)  # both rank-ordered CSRs
    if kind == "build":
        return {"bytes": 8 * n + 8 * m + 12 * n + hier, "flops": 2.0 * 60 * m}
    if kind == "one_to_all":
        return {"bytes": 4 * n + hier + 4.0 * n * case["k"], "flops": 2.0 * 2 * 1.6 * m * case["k"]}
    core = 0.2 * n if case["graph"] == "rmat" else 0
    if kind == "core_table":
        inner = 100 * core  # the core's own edges, about
        return {"bytes": 8 * inner + 4 * core * core + 12 * case["k"], "flops": 2.0 * core * inner}
    k = case["targets"] if kind == "serve" else case["k"]
    relax = 2 * 100 * core if core else 2 * 900 * (n / 1e5) ** 0.25
    return {"bytes": 12 * k + min(hier, 8.0 * relax * k), "flops": 2.0 * relax * k}


# ---- what a pass returns, in 64 bits --------------------------------------

def _transform(x):
    return torch.sign(x) * torch.log2(1 + x.abs())


def exact(case, seed):
    """Training: forward and backward passes and Adam in 64 bits, with the
    method's own BF16 roundings (inputs, both weight matrices, the first
    hidden layer). Everything else returns whole numbers."""
    if case["kind"] != "train":
        return None
    st = prepare(case, seed)
    rows = st["rows"]
    bf = lambda a: a.float().bfloat16().double()  # noqa: E731
    x, y = bf(_transform(rows[:, 2:].double())), st["labels"].double()
    w = st["weights"].double()
    cut = [0, 768, 832, 4928, 4992, 5056, 5057]

    def grad(w, x, y):
        w1, b1, w2, b2, w3, b3 = (w[a:b] for a, b in zip(cut, cut[1:]))
        w1, w2 = bf(w1).view(12, 64), bf(w2).view(64, 64)
        h1 = bf(torch.relu(x @ w1 + b1))
        h2 = torch.relu(h1 @ w2 + b2)
        diff = h2 @ w3 + b3 - y
        dy = 2 * diff / len(y)
        g2 = torch.where(h2 > 0, dy[:, None] * w3, 0.0)
        g1 = torch.where(h1 > 0, g2 @ w2.T, 0.0)
        return torch.cat([(x.T @ g1).ravel(), g1.sum(0), (h1.T @ g2).ravel(), g2.sum(0), h2.T @ dy,
                          dy.sum()[None]]), (diff * diff).sum()

    size, total = min(case["batch"], len(y)), 0.0
    if case["epochs"] == 0:
        g, loss = grad(w, x[:size], y[:size])
        return dict(grad=g, loss=np.array([float(loss) / size]))
    m, v, losses, step = torch.zeros_like(w), torch.zeros_like(w), [], 0
    for _ in range(case["epochs"]):
        total = 0.0
        for a in range(0, len(y), size):
            g, loss = grad(w, x[a:a + size], y[a:a + size])
            total += float(loss)
            step += 1
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            w = w - 2e-3 * (m / (1 - 0.9 ** step)) / ((v / (1 - 0.999 ** step)).sqrt() + 1e-8)
        losses.append(total / len(y))
    return dict(weights=w, loss=np.array(losses))
