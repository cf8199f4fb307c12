"""The workloads whose speed matters to a user of the engine, as plain-value cases.

A program loads a road network once and keeps it resident; queries then arrive over it with
new node sets.  So a case names a network (kept for the process, like the graph handle that
such a program keeps) and a query over it, and the seed draws the query's sets.  Networks
come from ``paper_1607_07696_gb300.inputs``: the jittered 64 x 64 lattice and the road-like
graphs whose sizes (264,000 / 730,000 and 1,070,000 / 2,700,000 nodes / edges) and sets
(256, 10,000 and 50,000 nodes a side) are those of the repository's tests and benchmark.
A radius is given in median arc weights (``hops``), which says the same on every network: a
search of h hops meets about 1 to 2 h^2 nodes, more where the map has more edges.

``listed()``  the cases;  ``draw(rng)``  one more of the same ranges;  ``prepare(case, seed)``
a query's inputs in hand;  ``run(state)``  one pass through the public entry points;
``work(case)``  the bytes and operations a pass cannot do without;  ``exact(case, seed)``  the
small lattice's answer by plain numpy.
"""
from __future__ import annotations

import collections
import math

import numpy as np
import torch

from paper_1607_07696_gb300 import inputs, rn

# -------------------------------------------------------------------------- cases ----

def listed() -> list[dict]:
    small = {"graph": "grid", "n": 4096, "m": 7400, "sets": "uniform", "nR": 256, "nS": 256}
    city = {"graph": "road", "n": 264_000, "m": 730_000, "sets": "uniform"}
    region = {"graph": "road", "n": 1_070_000, "m": 2_700_000, "sets": "clustered"}
    return [
        # the smallest query there is: a neighbourhood map, an interactive lookup
        {"name": "grid_join", "call": "join_dev", **small, "hops": 15.0},
        # an ordinary join on a city-sized network, everything on the device
        {"name": "city_join", "call": "join_dev", **city, "nR": 10_000, "nS": 10_000, "hops": 26.9},
        # the largest join: a million nodes, 50,000 clustered places a side
        {"name": "region_join", "call": "join_dev", **region, "nR": 50_000, "nS": 50_000, "hops": 20.8},
        # few sources with a wide radius (catchment areas): balls of thousands of nodes
        {"name": "region_wide_join", "call": "join_dev", **region, "nR": 5_000, "nS": 50_000, "hops": 52.0},
        # host arrays in and out, many customers against few depots (searched from the depots)
        {"name": "city_depots", "call": "join", **city, "nR": 20_011, "nS": 1_999, "hops": 24.0},
        # "the closest hundred": a short answer over a city, host arrays
        {"name": "city_kcp_100", "call": "kcp", **city, "nR": 10_000, "nS": 10_000, "k": 100},
        # k closest pairs on the large network, a short and a long answer
        {"name": "region_kcp_10k", "call": "kcp_dev", **region, "nR": 50_000, "nS": 50_000, "k": 10_000},
        {"name": "region_kcp_1m", "call": "kcp_dev", **region, "nR": 50_000, "nS": 50_000, "k": 1_000_000},
        # many small networks at once (one batch, replayed with its results read back)
        {"name": "towns_batch", "call": "batch", "instances": 20, "n_lo": 1_000, "n_hi": 50_000, "towns": 1},
        # a burst of mixed requests at a server over one resident network
        {"name": "region_serve", "call": "serve", "graph": "road", "n": 1_070_000, "m": 2_700_000, "sets": "uniform",
         "requests": 20, "lo": 100, "hi": 20_000, "stream": 1},
        # places along streets instead of at crossings
        {"name": "city_points", "call": "points", **city, "nR": 5_000, "nS": 5_000, "hops": 26.9},
        # the paper's own formulation, by parts of the partition hierarchy
        {"name": "city_hier", "call": "hier", **city, "nR": 10_000, "nS": 10_000, "hops": 26.9},
    ]


def _growth(n: int, m: int) -> float:
    """Nodes within h median arc weights of a node, over h^2: the lattice's, or a road-like
    network's, which grows with its edges per node."""
    return 1.9 if m < 2 * n else 1.13 + 2.64 * (m / n - 2.523)


def _log(rng, lo: float, hi: float) -> float:
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng) -> dict:
    call = rng.choice(["join_dev", "join_dev", "join", "kcp_dev", "kcp", "batch", "serve", "points", "hier"])
    if call == "batch":
        lo = int(_log(rng, 1_000, 8_000))
        return {"call": call, "instances": rng.randint(3, 20), "n_lo": lo, "n_hi": int(_log(rng, lo, 40_000)),
                "towns": rng.randint(2, 10_000)}
    n = int(_log(rng, 4_000, 1_000_000 if call in ("join_dev", "kcp_dev") else 264_000))
    c = {"call": call, "graph": "road", "n": n, "m": int(n * rng.uniform(2.5, 2.75)),
         "sets": rng.choice(["uniform", "clustered"])}
    if call == "serve":
        return {**c, "sets": "uniform", "requests": rng.randint(3, 20), "lo": 50, "hi": int(min(20_000, n // 4)),
                "stream": rng.randint(2, 10_000)}
    most = min(50_000, n // 3)
    c["nR"], c["nS"] = int(_log(rng, 64, most)), int(_log(rng, 64, most))
    if call in ("kcp_dev", "kcp"):
        # radii whose balls stay within a few thousand nodes, as the serving stream's do
        c["k"] = int(_log(rng, 10, min(1e6, max(11.0, c["nR"] * c["nS"] * 2_000 / n))))
        return c
    if call in ("points", "hier"):
        c["nR"], c["nS"] = min(c["nR"], 10_000), min(c["nS"], 10_000)
    # at most 24 million visited nodes and 2.8 million pairs
    ball = min(3_000, 24e6 / min(c["nR"], c["nS"]), 2.8e6 * n / (c["nR"] * c["nS"]) / (3 if c["sets"] == "clustered" else 1))
    c["hops"] = round(rng.uniform(4.0, max(5.0, math.sqrt(ball / _growth(n, c["m"])))), 2)
    return c


# ------------------------------------------------------------------------- inputs ----

_networks: collections.OrderedDict = collections.OrderedDict()  # the resident networks, the oldest dropped


def _network(kind: str, n: int, m: int, seed: int = inputs.BASE_SEED):
    """(handle, edge list, median weight) of a network, loaded once and kept."""
    at = (kind, n, m, seed)
    if at not in _networks:
        e = inputs.grid_graph(seed) if kind == "grid" else inputs.road_graph(n, m, seed)
        _networks[at] = (rn.rn_graph_load(e.src, e.dst, e.w, e.n), e, int(np.median(e.w)))
        while len(_networks) > 64:
            _networks.popitem(last=False)
    _networks.move_to_end(at)
    return _networks[at]


_servers: dict = {}  # one server per resident network, as a serving program keeps


def _server(g):
    if id(g) not in _servers:
        _servers.clear()
        _servers[id(g)] = rn.rn_serve_create(g, slab_bytes=1 << 30)
    return _servers[id(g)]


def _sets(case: dict, e, rng) -> tuple[np.ndarray, np.ndarray]:
    """Disjoint R and S: uniform nodes, or nodes drawn around 20 centres (standard deviation
    0.05 of the map's side)."""
    nR, nS = case["nR"], case["nS"]
    if case["sets"] == "clustered":
        xy = e.xy.astype(np.float32)
        density = np.zeros(e.n, np.float32)
        for c in rng.uniform(0.1, 0.9, size=(20, 2)).astype(np.float32):
            d = xy - c
            density += np.exp((d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) * np.float32(-1 / (2 * 0.05**2)))
        # the largest of log(density) + Gumbel noise: a draw without replacement by density
        score = np.log(density + 1e-30) - np.log(rng.exponential(size=e.n))
        pick = np.argpartition(score, e.n - nR - nS)[e.n - nR - nS:]
        pick = rng.permutation(pick)
    else:
        pick = rng.choice(e.n, size=nR + nS, replace=False)
    pick = pick.astype(np.uint32)
    return pick[:nR].copy(), pick[nR:].copy()


def _points(e, count: int, rng) -> np.ndarray:
    i = rng.integers(0, e.m, size=count)
    t = (rng.random(count) * (e.w[i] + 1.0)).astype(np.int64)
    return np.stack([e.src[i].astype(np.int64), e.dst[i].astype(np.int64), np.minimum(t, e.w[i])], axis=1)


def _towns(case: dict) -> list[dict]:
    """The batch's networks and query sizes: part of the case, so that seeds draw only sets."""
    rng = np.random.default_rng(case["towns"])
    specs = []
    for i in range(case["instances"]):
        n = int(inputs.log_uniform(rng, case["n_lo"], case["n_hi"] + 1))
        nR, nS = (int(min(inputs.log_uniform(rng, 64, 4096), n // 3)) for _ in range(2))
        ball = min(float(inputs.log_uniform(rng, 5, 200)) * n / nS, float(n))
        specs.append({"n": n, "m": int(2.77 * n), "nR": nR, "nS": nS, "sets": "uniform",
                      "hops": math.sqrt(ball / _growth(n, 2.77 * n)), "seed": case["towns"] * 100 + i})
    return specs


def _requests(case: dict) -> list[dict]:
    """The served stream's request sizes: seven joins to three k-closest-pairs queries."""
    rng = np.random.default_rng(case["stream"])
    n, specs = case["n"], []
    for _ in range(case["requests"]):
        nR, nS = (int(inputs.log_uniform(rng, case["lo"], case["hi"])) for _ in range(2))
        q = {"n": n, "m": case["m"], "nR": nR, "nS": nS, "sets": "uniform"}
        if rng.random() < 0.7:
            ball = min(float(inputs.log_uniform(rng, 5, 200)) * n / nS, inputs.C5_BALL_CAP, n)
            q["hops"] = math.sqrt(ball / _growth(n, case["m"]))
        else:
            q["k"] = max(1, min(int(inputs.log_uniform(rng, 10, 100_000)), int(nR * nS * 2_000 / n)))
        specs.append(q)
    return specs


def _ball(q: dict) -> float:
    """Nodes that one source's search of a query meets."""
    if "k" in q:
        return min(q["n"], q["k"] * q["n"] / (q["nR"] * q["nS"]))
    return min(q["n"], _growth(q["n"], q["m"]) * q["hops"]**2)


def _pairs(q: dict) -> float:
    """Pairs in a query's answer (clustered sets are denser where the sources are)."""
    dense = 3 if q["sets"] == "clustered" else 1
    return q["k"] if "k" in q else min(q["nR"] * q["nS"], dense * q["nR"] * q["nS"] * _ball(q) / q["n"])


def _room(q: dict, device: bool = False):
    """A caller's buffer for a query's answer, with room to spare."""
    shape = (3, q["k"] if "k" in q else int(min(q["nR"] * q["nS"], 3 * _pairs(q) + 4096)))
    if device:
        return torch.full(shape, -1, dtype=torch.int32, device="cuda")
    return np.full(shape, -1, np.int32)


def _theta(hops: float, median: int) -> int:
    return int(round(hops * median))


def prepare(case: dict, seed: int) -> dict:
    rng = np.random.default_rng(seed)
    call = case["call"]
    if call == "batch":
        towns, queries = _towns(case), []
        for t in towns:
            g, e, median = _network("road", t["n"], t["m"], t["seed"])
            queries.append((g, *_sets(t, e, rng), _theta(t["hops"], median)))
        b = rn.rn_batch_create(queries)
        rn.rn_batch_run(b)  # a prepared batch has met its instances once
        return {"call": call, "batch": b, "kept": [_room(t) for t in towns]}
    g, e, median = _network(case["graph"], case["n"], case["m"])
    if call == "serve":
        specs = _requests(case)
        stream = [(*_sets(q, e, rng), rn.RN_INF if "k" in q else _theta(q["hops"], median), q.get("k", 0)) for q in specs]
        return {"call": call, "server": _server(g), "requests": stream, "kept": [_room(q) for q in specs]}
    state = {"call": call, "g": g, "kept": _room(case, device=call.endswith("_dev"))}
    if "k" in case:
        state["k"] = case["k"]
    else:
        state["theta"] = _theta(case["hops"], median)
    if call == "points":
        state["R"], state["S"] = _points(e, case["nR"], rng), _points(e, case["nS"], rng)
        return state
    state["R"], state["S"] = _sets(case, e, rng)
    if call.endswith("_dev"):
        for x in "RS":
            state[x] = torch.as_tensor(state[x].astype(np.int32), device="cuda")
        state["out"] = rn.DevicePairs()
    return state


# ---------------------------------------------------------------------------- run ----

def _kept(pairs, buffer):
    """(count, buffer) with the pairs copied into the caller's buffer, which is as long
    whatever the seed: the library's own arrays last only until the next call."""
    n = len(pairs[0])
    for row, x in zip(buffer, pairs):
        row[:n] = x.view(np.int32) if isinstance(x, np.ndarray) else x
    return n, buffer


def run(s: dict):
    call = s["call"]
    if call == "batch":
        rn.rn_batch_run(s["batch"])
        return [_kept(rn.rn_batch_pairs(s["batch"], i), to) for i, to in enumerate(s["kept"])]
    if call == "serve":
        tickets = [rn.rn_serve_submit(s["server"], *request) for request in s["requests"]]
        return [_kept(rn.rn_serve_wait(s["server"], t), to) for t, to in zip(tickets, s["kept"])]
    if call == "join_dev":
        rn.rn_distance_join_dev(s["g"], s["R"], s["S"], s["theta"], s["out"])
        return _kept(s["out"].tensors(), s["kept"])
    if call == "kcp_dev":
        rn.rn_kcp_dev(s["g"], s["R"], s["S"], s["k"], rn.RN_INF, s["out"])
        return _kept(s["out"].tensors(), s["kept"])
    if call == "join":
        return _kept(rn.rn_distance_join(s["g"], s["R"], s["S"], s["theta"]), s["kept"])
    if call == "kcp":
        return _kept(rn.rn_kcp(s["g"], s["R"], s["S"], s["k"]), s["kept"])
    if call == "points":
        return _kept(rn.rn_distance_join_points(s["g"], s["R"], s["S"], s["theta"]), s["kept"])
    return _kept(rn.rn_distance_join_hier(s["g"], s["R"], s["S"], s["theta"]), s["kept"])


# --------------------------------------------------------------------------- work ----

def work(case: dict) -> dict:
    """Bytes: the sets once, the rows and arcs of the touched part of the network once, the
    pairs once.  Operations: an addition and a comparison for every arc of every source's
    ball, searched from the smaller set."""
    call, nbytes, ops = case["call"], 0.0, 0.0
    for q in _towns(case) if call == "batch" else _requests(case) if call == "serve" else [case]:
        sources, degree = min(q["nR"], q["nS"]), 2 * q["m"] / q["n"]
        touched = min(q["n"], sources * _ball(q))
        nbytes += (12 if call == "points" else 4) * (q["nR"] + q["nS"]) + touched * (4 + 8 * degree) + 12 * _pairs(q)
        ops += 2 * sources * _ball(q) * degree
    return {"bytes": nbytes, "flops": ops}


def exact(case: dict, seed: int):
    """The join's (u, v, d) by Bellman-Ford over all sources at once, in 64 bits; None where
    that would take long."""
    if case["call"] != "join_dev" or case["nR"] * case["n"] > 1 << 21:
        return None
    e = inputs.grid_graph(inputs.BASE_SEED) if case["graph"] == "grid" else inputs.road_graph(case["n"], case["m"], inputs.BASE_SEED)
    R, S = _sets(case, e, np.random.default_rng(seed))
    theta = _theta(case["hops"], int(np.median(e.w)))
    src, dst, w = (np.concatenate(x).astype(np.int64) for x in ((e.src, e.dst), (e.dst, e.src), (e.w, e.w)))
    order = np.argsort(dst, kind="stable")
    src, w = src[order], w[order]
    node, start = np.unique(dst[order], return_index=True)  # the arcs into each node, one run each
    R, S = np.sort(R).astype(np.int64), np.sort(S).astype(np.int64)
    dist = np.full((e.n, len(R)), 1 << 40, np.int64)
    dist[R, np.arange(len(R))] = 0
    while True:
        least = np.minimum(dist[node], np.minimum.reduceat(dist[src] + w[:, None], start, axis=0))
        if np.array_equal(least, dist[node]):
            break
        dist[node] = least
    d = dist[S].T
    i, j = np.nonzero(d <= theta)
    kept = np.full((3, int(min(case["nR"] * case["nS"], 3 * _pairs(case) + 4096))), -1, np.int64)
    kept[:, :len(i)] = R[i], S[j], d[i, j]
    return len(i), kept
