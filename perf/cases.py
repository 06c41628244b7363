"""The calls whose time matters to a user of this library, from the smallest to the largest.

A case is one call (or one short sequence of calls) through the public binding, on a seeded
temporal graph of the structure the library is made for:

  exact     count_exact on a resident graph, one query: the least work a call can carry.
  noalloc   count_exact_noalloc, for callers that may not allocate.
  prepared  a fixed batch captured once and replayed: launch, then the results.
  batch     run_batch on a resident graph.
  step      graph from device arrays, one batch, graph freed: the benchmark's step.
  host      the same from pinned host arrays.
  stream    stream_run over pinned host arrays, never holding the whole graph on the device.
  serve     a burst of queries to a server, all their results.

The results come back whole, as arrays over the queries.  The library's work counters
(entries read, ranges closed) and its memory figure say how it went about a call, not what was
asked, and are not among them."""
import math

import numpy as np
import torch

from paper_1810_00980_gb300 import synth, tm

# the first four are the library's own workload motifs, the others its test shapes: a repeated
# out-star, a five-cycle, a path whose last edge reaches a new node, two edges out of one node
MOTIFS = {
    "cycle3": ([0, 1, 2], [1, 2, 0]),
    "outstar3": ([2, 2, 2], [0, 1, 0]),
    "pingpong": ([0, 1, 0], [1, 0, 1]),
    "cycle4": ([0, 1, 2, 3], [1, 2, 3, 0]),
    "star4": ([0, 0, 0, 0], [1, 2, 1, 2]),
    "cycle5": ([0, 1, 2, 3, 4], [1, 2, 3, 4, 0]),
    "path3": ([0, 2, 1], [1, 3, 2]),
    "fan2": ([0, 0], [1, 2]),
}
THREE = ("cycle3", "outstar3", "pingpong")
DELTAS = (600, 3600, 86400)
# the benchmark's calibrated (c, p, b) per motif and span
ESTIMATES = {
    ("cycle3", 600): (30, 0.85, 1), ("cycle3", 3600): (5, 0.7, 1), ("cycle3", 86400): (30, 1.0, 1),
    ("outstar3", 600): (10, 0.2, 1), ("outstar3", 3600): (2, 0.1, 4), ("outstar3", 86400): (30, 1.0, 1),
    ("pingpong", 600): (10, 0.2, 1), ("pingpong", 3600): (2, 0.3, 1), ("pingpong", 86400): (30, 1.0, 1),
}
FIELDS = (("status", np.int64), ("count", np.int64), ("estimate", np.float64), ("windows", np.int64),
          ("windows_kept", np.int64), ("var_hat", np.float64), ("shift_var", np.float64), ("p_used", np.float64))


def listed():
    return [
        # one exact count on a small graph (20,000 edges): launches and latency
        {"name": "count-20k", "call": "exact", "mix": "one:cycle3:86400", "m": 20_000, "n": 200, "graph": "bursty"},
        # the largest graph that the entry point without allocation takes
        {"name": "noalloc-262k", "call": "noalloc", "mix": "one:outstar3:3600", "m": 262_144, "n": 2_621, "graph": "bursty"},
        # a dashboard's fixed queries replayed on a graph of about 100,000 edges
        {"name": "replay-100k", "call": "prepared", "mix": "bench", "m": 99_991, "n": 1_009, "graph": "bursty"},
        # the benchmark's 18 queries on a resident graph of a million edges
        {"name": "batch-1m", "call": "batch", "mix": "bench", "m": 1_000_000, "n": 10_000, "graph": "bursty"},
        # deeper motifs, counted exactly: four and five edges, and last edges to a new node
        {"name": "deep-1m", "call": "batch", "mix": "deep", "m": 1_250_003, "n": 12_503, "graph": "bursty"},
        # the estimates on their own (no exact query beside them), ten million edges
        {"name": "estimates-10m", "call": "batch", "mix": "estimates", "m": 10_000_000, "n": 100_000, "graph": "bursty"},
        # the benchmark's step: build the graph, 18 queries, ten million edges
        {"name": "step-10m", "call": "step", "mix": "bench", "m": 10_000_000, "n": 100_000, "graph": "bursty"},
        # millisecond times (64-bit), an odd size, from host memory
        {"name": "host-3m-wide", "call": "host", "mix": "bench", "m": 3_333_331, "n": 33_331, "graph": "bursty", "ticks": 1000},
        # many seeds of one four-edge estimate in one launch, graph built for them
        {"name": "seeds-10m", "call": "step", "mix": "seeds:32", "m": 10_000_000, "n": 100_000, "graph": "bursty", "gamma": 2.0},
        # a hub-skewed graph built for a few sparse estimates: the build is the work
        {"name": "hubs-100m", "call": "step", "mix": "hub", "m": 100_000_000, "n": 1_000_000, "graph": "hubs"},
        # the same 18 queries over a list held on the host, a million edges at a time
        {"name": "stream-10m", "call": "stream", "mix": "bench", "m": 10_000_000, "n": 100_000, "graph": "bursty", "segment": 1_000_000},
        # a burst of mixed queries to a server over two graphs
        {"name": "serve-burst", "call": "serve", "mix": "serve:48", "m": 5_000_000, "n": 50_000, "graph": "bursty", "m2": 1_000_000, "n2": 10_000},
    ]


def _size(rng, lo, hi):
    m = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    return m | 1 if rng.random() < 0.7 else m


def draw(rng):
    kind = rng.choice(["exact", "noalloc", "prepared", "batch", "deep", "estimates", "step", "host", "seeds", "hubs",
                       "stream", "serve"])
    three, d = rng.choice(THREE + ("cycle4", "fan2")), rng.choice(DELTAS[1:])
    if kind == "exact":
        m = _size(rng, 8_000, 400_000)
        return {"call": "exact", "mix": "one:%s:%d" % (three, d), "m": m, "n": max(50, m // rng.choice([20, 50, 100])),
                "graph": rng.choice(["uniform", "bursty"])}
    if kind == "noalloc":
        m = _size(rng, 8_000, 262_144)
        return {"call": "noalloc", "mix": "one:%s:%d" % (three, d), "m": m, "n": max(50, m // 100), "graph": "bursty"}
    if kind == "prepared":
        m = _size(rng, 10_000, 1_000_000)
        return {"call": "prepared", "mix": rng.choice(["bench", "exacts", "estimates"]), "m": m, "n": m // 100, "graph": "bursty"}
    if kind in ("batch", "estimates"):
        m = _size(rng, 100_000, 10_000_000)
        return {"call": "batch", "mix": "estimates" if kind == "estimates" else rng.choice(["bench", "exacts", "auto"]),
                "m": m, "n": m // 100, "graph": "bursty"}
    if kind == "deep":
        m = _size(rng, 100_000, 1_250_000)
        return {"call": "batch", "mix": "deep", "m": m, "n": m // 100, "graph": "bursty"}
    if kind == "step":
        m = _size(rng, 100_000, 10_000_000)
        return {"call": "step", "mix": rng.choice(["bench", "exacts"]), "m": m, "n": m // rng.choice([20, 100, 300]), "graph": "bursty"}
    if kind == "host":
        m = _size(rng, 100_000, 4_000_000)
        return {"call": "host", "mix": "bench", "m": m, "n": m // 100, "graph": "bursty", "ticks": rng.choice([1, 1000])}
    if kind == "seeds":
        m = _size(rng, 500_000, 10_000_000)
        return {"call": rng.choice(["step", "batch"]), "mix": "seeds:%d" % rng.randint(2, 32), "m": m, "n": m // 100,
                "graph": "bursty", "gamma": 2.0}
    if kind == "hubs":
        m = _size(rng, 2_000_000, 50_000_000)
        return {"call": "step", "mix": "hub", "m": m, "n": m // 100, "graph": "hubs"}
    if kind == "stream":
        m = _size(rng, 1_000_000, 10_000_000)
        return {"call": "stream", "mix": rng.choice(["bench", "exacts"]), "m": m, "n": m // 100, "graph": "bursty",
                "segment": m // rng.randint(3, 12)}
    m = _size(rng, 500_000, 5_000_000)
    return {"call": "serve", "mix": "serve:%d" % rng.randint(16, 48), "m": m, "n": m // 100, "graph": "bursty",
            "m2": max(100_000, m // 5), "n2": max(1_000, m // 500)}


# ---------------------------------------------------------------- inputs
def _edges(case, seed, m, n):
    """Time-sorted device arrays (src, dst, t)."""
    if case["graph"] == "uniform":
        return tuple(torch.from_numpy(x).cuda() for x in synth.uniform_graph(n, m, 1_000_000, seed))
    if case["graph"] == "hubs":
        s, d, t = synth.chung_lu_hawkes_gpu(n, m, 1.8, seed, max_degree=m // 200, hub_bursts=max(1, m // 1_000_000))
    else:
        s, d, t = synth.chung_lu_hawkes_gpu(n, m, case.get("gamma", 2.1), seed)
    if case.get("ticks", 1) > 1:   # finer clock: each second's edges spread over its ticks, in order
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed + 17)
        t = t * case["ticks"] + torch.randint(0, case["ticks"], t.shape, generator=gen, device="cuda")
        t, order = torch.sort(t, stable=True)
        s, d = s[order].contiguous(), d[order].contiguous()
    return s, d, t


def _specs(case, seed):
    """(motif, delta, mode, c, p, seed, b, q_mode) of each query."""
    mix, k = case["mix"].split(":")[0], case.get("ticks", 1)
    ex = [(name, d * k, 0, 1, 1.0, 0, 1, 0) for name in THREE for d in DELTAS]
    es = [(name, d * k, 1, *ESTIMATES[name, d][:2], 1000 + 10 * i + j + seed, ESTIMATES[name, d][2], 0)
          for i, name in enumerate(THREE) for j, d in enumerate(DELTAS)]
    if mix == "one":
        _, name, d = case["mix"].split(":")
        return [(name, int(d), 0, 1, 1.0, 0, 1, 0)]
    if mix == "bench":
        return ex + es
    if mix == "exacts":
        return ex
    if mix == "estimates":
        return es
    if mix == "deep":
        return [("cycle4", 3600, 0, 1, 1.0, 0, 1, 0), ("star4", 600, 0, 1, 1.0, 0, 1, 0), ("cycle5", 600, 0, 1, 1.0, 0, 1, 0),
                ("path3", 600, 0, 1, 1.0, 0, 1, 0), ("fan2", 3600, 0, 1, 1.0, 0, 1, 0),
                ("cycle4", 600, 1, 10, 3000.0, seed + 5, 1, 1)]
    if mix == "seeds":
        n = int(case["mix"].split(":")[1])
        return [("cycle4", 3600, 1, c, p, 9000 + s + seed, 1, 0) for c in (10, 30, 100) for p in (0.01, 0.1) for s in range(n)]
    if mix == "hub":
        return [("outstar3", 1800, 1, 30, 0.01, 500 + s + seed, 1, 0) for s in range(8)]
    if mix == "auto":   # p chosen by a pilot for a 5 % error; one with q_j by window edges
        return [(name, d, 1, 10, 0.05, 77 + seed, 2, 2) for name in THREE for d in DELTAS[:2]] + \
               [("cycle3", 3600, 1, 10, 500.0, 78 + seed, 2, 1)]
    assert mix == "serve"
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(int(case["mix"].split(":")[1])):
        name, d = str(rng.choice(THREE + ("cycle4",))), int(rng.choice(DELTAS[:2]))
        c, p, s = int(rng.choice([10, 30])), float(rng.choice([0.01, 0.05, 0.1])), int(rng.integers(1 << 40))
        kind = rng.random()
        out.append((name, d, 0, 1, 1.0, 0, 1, 0) if kind < 0.5 else
                   (name, d, 1, c, p, s, 1, 0) if kind < 0.8 else (name, d, 1, c, 0.05, s, 1, 2))
    return out


def _queries(case, seed):
    motifs = {k: tm.Motif(*v) for k, v in MOTIFS.items()}
    return [tm.Query(motifs[name], d, mode, c, p, s, b, qm) for name, d, mode, c, p, s, b, qm in _specs(case, seed)]


def prepare(case, seed):
    call, n = case["call"], case["n"]
    qs = _queries(case, seed)
    src, dst, t = _edges(case, seed, case["m"], n)
    st = {"call": call, "queries": qs, "n": n}
    if call in ("host", "stream"):
        st["edges"] = tuple(x.cpu().pin_memory() for x in (src, dst, t))
        st["segment"] = case.get("segment", 0)
        return st
    if call == "step":
        st["edges"] = (src, dst, t)
        return st
    g = st["graph"] = tm.Graph(src, dst, t, n)
    if call == "prepared":
        st["batch"] = tm.PreparedBatch(g, qs)
    elif call == "batch":
        st["batch"] = tm.Batch(g, qs)
    elif call == "serve":
        g2 = st["graph2"] = tm.Graph(*_edges(case, seed + 1, case["m2"], case["n2"]), case["n2"])
        srv = st["server"] = tm.Server(n_streams=2, max_batch=64)
        st["ids"] = [srv.attach(g), srv.attach(g2)]
    return st


# ---------------------------------------------------------------- the calls
def _columns(rows):
    return {k: np.array([r[k] for r in rows], dtype) for k, dtype in FIELDS}


def run(state):
    call, qs = state["call"], state["queries"]
    if call == "exact":
        return {"count": tm.count_exact(state["graph"], qs[0].motif, qs[0].delta)}
    if call == "noalloc":
        return {"count": tm.count_exact_noalloc(state["graph"], qs[0].motif, qs[0].delta)}
    if call == "prepared":
        state["batch"].launch()
        return _columns(state["batch"].results())
    if call == "batch":
        state["batch"].run()
        return _columns(state["batch"].results())
    if call in ("step", "host"):
        with tm.Graph(*state["edges"], state["n"]) as g:
            info = g.info()
            out = _columns(tm.run_batch(g, qs))
        out["graph"] = np.array([info.m, info.n_nodes, info.n_pairs, info.t_min, info.t_max], np.int64)
        return out
    if call == "stream":
        return _columns(tm.stream_run(*state["edges"], qs, state["segment"], state["n"])[0])
    srv = state["server"]
    tickets = [srv.submit(state["ids"][i % 2], q) for i, q in enumerate(qs)]
    return _columns([srv.wait(k)[1] for k in tickets])


def work(case):
    """The edge list read once (12 bytes an edge resident, 16 where it comes in: two ids and a
    time) and a result written for each query; the arithmetic is on integers."""
    edges = case["m"] + case.get("m2", 0)
    per = 16 if case["call"] in ("step", "host", "stream") else 12
    nq = {"one": 1, "bench": 18, "exacts": 9, "estimates": 9, "deep": 6, "hub": 8, "auto": 7}.get(case["mix"].split(":")[0])
    if nq is None:
        nq = int(case["mix"].split(":")[1]) * (6 if case["mix"].startswith("seeds") else 1)
    return {"bytes": per * edges + 96 * nq, "flops": 0}


# ---------------------------------------------------------------- plain numpy
_EXACT_MOST = 300_000   # edges: beyond these, listing every instance in numpy takes minutes


def _instances(src, dst, t, mu, mv, delta):
    """First and last edge times of every instance, one motif edge at a time."""
    span = int(t.max()) + delta + 2
    n = int(max(src.max(), dst.max())) + 1

    def index(key):
        order = np.argsort(key * span + t, kind="stable")
        return order, (key * span + t)[order]

    views = {"out": index(src.astype(np.int64)), "in": index(dst.astype(np.int64)),
             "pair": None, "all": (np.arange(len(t)), t)}
    if n * n < (1 << 62) // span:
        views["pair"] = index(src.astype(np.int64) * n + dst)
    fine = np.flatnonzero(src != dst)
    bound = {mu[0]: src[fine].astype(np.int64), mv[0]: dst[fine].astype(np.int64)}
    t1, tp = t[fine], t[fine]
    for u, v in list(zip(mu, mv))[1:]:
        if u in bound and v in bound:
            (order, keys), node = views["pair"], bound[u] * n + bound[v]
        elif u in bound:
            (order, keys), node = views["out"], bound[u]
        elif v in bound:
            (order, keys), node = views["in"], bound[v]
        else:
            (order, keys), node = views["all"], np.zeros_like(t1)
        lo = np.searchsorted(keys, node * span + tp, "right")
        hi = np.searchsorted(keys, node * span + t1 + delta, "right")
        count = np.maximum(hi - lo, 0)
        who = np.repeat(np.arange(len(count)), count)
        e = order[np.arange(len(who)) - np.repeat(np.cumsum(count) - count, count) + lo[who]]
        s, d = src[e].astype(np.int64), dst[e].astype(np.int64)
        ok = s != d
        for new, x in ((u, s), (v, d)):
            if new not in bound:
                for label, y in bound.items():
                    ok &= x != y[who]
        who, e, s, d = who[ok], e[ok], s[ok], d[ok]
        was = set(bound)
        bound = {label: y[who] for label, y in bound.items()}
        if u not in was:
            bound[u] = s
        if v not in was:
            bound[v] = d
        t1, tp = t1[who], t[e]
    return t1, tp


def _mix64(x):
    x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return x ^ (x >> np.uint64(31))


def _draws(seed, k, j):
    step = np.uint64(0x9E3779B97F4A7C15)
    base = _mix64(np.uint64(seed & (2**64 - 1)) + np.uint64(k + 1) * step)
    return _mix64(base + (np.asarray(j, np.uint64) + np.uint64(1)) * step)


def exact(case, seed):
    """Algorithm 1 over every instance, listed in numpy; no value for the larger graphs, nor
    where p comes from a pilot."""
    specs = _specs(case, seed)
    if case["m"] > _EXACT_MOST or case["call"] in ("serve", "stream") or any(q[7] == 2 for q in specs):
        return None
    src, dst, t = (x.cpu().numpy() for x in _edges(case, seed, case["m"], case["n"]))
    info = np.array([len(t), case["n"], len(np.unique(src.astype(np.int64) * case["n"] + dst)), t[0], t[-1] - t[0]], np.int64)
    t = t - t[0]
    rows = []
    with np.errstate(over="ignore"):
        for name, delta, mode, c, p, s, b, q_mode in specs:
            t1, t3 = _instances(src, dst, t, *MOTIFS[name], delta)
            if mode == 0:
                rows.append((0, len(t1), float(len(t1)), 1, 1, 0.0, 0.0, 1.0))
                continue
            cd = c * delta
            J = 1 + -(-int(t[-1]) // cd)
            z, var, kept_n, inside_n = [], [], 0, 0
            for k in range(b):
                shift = -int(_draws(s, k, [0])[0] % np.uint64(cd))
                j = np.arange(1, J + 1)
                q = np.full(J, p)
                if q_mode == 1:
                    lo = np.searchsorted(t, shift + (j - 1) * cd, "left")
                    q = np.minimum(1.0, p * (np.searchsorted(t, shift + j * cd - 1, "right") - lo) / len(t))
                kept = (_draws(s, k, j) >> np.uint64(11)).astype(np.float64) * 2.0**-53 < q
                w = (t1 - shift) // cd
                inside = (t3 <= shift + (w + 1) * cd - 1) & kept[np.minimum(w, J - 1)]
                y = np.bincount(w[inside], cd / (cd - (t3 - t1)[inside]).astype(np.float64), minlength=J)
                qk, yk = q[kept], y[kept]
                z.append(float((yk / qk).sum()))
                var.append(float((yk * yk * (1 - qk) / (qk * qk)).sum()))
                kept_n += int(kept.sum())
                inside_n += int(inside.sum())
            rows.append((0, inside_n, float(np.mean(z)), b * J, kept_n, float(np.mean(var)),
                         float(np.var(z, ddof=1)) if b > 1 else 0.0, p))
    if case["call"] in ("exact", "noalloc"):
        return {"count": rows[0][1]}
    out = {k: np.array([r[i] for r in rows], dtype) for i, (k, dtype) in enumerate(FIELDS)}
    if case["call"] in ("step", "host"):
        out["graph"] = info
    return out
