"""The workloads this library's speed is judged on, at the sizes they are used at.

A case is one call of the public API by a program that keeps its graph on the
device: a single query (``opmos_solve``), a batch of queries
(``opmos_solve_batch``), a stream of queries through the server
(``opmos_server``), or the heuristic alone (``opmos_heur``). Graphs are made
from a seed here: 8-connected grids with random or ship-routing costs,
time-expanded ship routes of many objectives, road-like graphs. Fronts and
paths come back whole; where several paths carry one cost vector the library
keeps the same one for the same call, so paths are part of the results.
"""
import heapq
import math
import time

import numpy as np

from paper_2411_16667_gb300 import opmos

SERVE_MEMORY = 16 << 30  # frontier and open-list budget of the served cases
SERVE_SECONDS = 60  # a served burst that takes longer is given up


# ---------------------------------------------------------------------------
# graphs: (n, rowptr, col, cost[d, m])
# ---------------------------------------------------------------------------
def _grid(rows, cols, is_open):
    """Arcs of the 8-connected grid between open cells, in CSR order:
    rowptr, source and target of every arc, and whether it is diagonal."""
    r, c = np.divmod(np.arange(rows * cols), cols)
    step = [(a, b) for a in (-1, 0, 1) for b in (-1, 0, 1) if a or b]
    rr = r[:, None] + np.array([a for a, _ in step])
    cc = c[:, None] + np.array([b for _, b in step])
    there = (rr >= 0) & (rr < rows) & (cc >= 0) & (cc < cols) & is_open[:, None]
    to = np.where(there, rr * cols + cc, 0)
    there &= is_open[to]
    src = np.nonzero(there)[0]
    diagonal = np.broadcast_to(np.array([a != 0 and b != 0 for a, b in step]), there.shape)[there]
    rowptr = np.zeros(rows * cols + 1, np.uint64)
    np.cumsum(there.sum(1), out=rowptr[1:])
    return rowptr, src, to[there], diagonal


def _field(rng, rows, cols, blobs=32):
    """A smooth field in [0, 1]: a sum of Gaussian blobs of 8 to 48 cells."""
    y, x = rng.random(blobs) * rows, rng.random(blobs) * cols
    sigma, height = 8 + 40 * rng.random(blobs), 0.5 + 0.5 * rng.random(blobs)
    fy = np.exp(-((np.arange(rows)[:, None] - y) ** 2) / (2 * sigma**2)) * height
    fx = np.exp(-((np.arange(cols)[:, None] - x) ** 2) / (2 * sigma**2))
    f = fy @ fx.T
    return ((f - f.min()) / max(f.max() - f.min(), 1e-9)).reshape(-1)


def _reached(rows, cols, is_open, start):
    """The open cells that 8-connected moves reach from start."""
    free = is_open.reshape(rows, cols)
    seen = np.zeros((rows + 2, cols + 2), bool)
    inner = seen[1:-1, 1:-1]
    inner[divmod(start, cols)] = True
    count = 0
    while inner.sum() != count:
        count = inner.sum()
        for _ in range(16):
            wide = seen[:-2] | seen[1:-1] | seen[2:]
            inner[...] = (wide[:, :-2] | wide[:, 1:-1] | wide[:, 2:]) & free
    return inner.reshape(-1).copy()


def _ship(rng, rows, cols, d):
    """A ship-routing grid with 5% land: move length, length x current, length
    x wave, exposure and move count (the first d of them); the two opposite
    corners are open and connected. Also the cells reached from the first."""
    n = rows * cols
    while True:
        land = _field(rng, rows, cols)
        is_open = np.ones(n, bool)
        is_open[np.argsort(-land, kind="stable")[: n // 20]] = False
        is_open[0] = is_open[n - 1] = True
        reached = _reached(rows, cols, is_open, 0)
        if reached[n - 1]:
            break
    rowptr, src, dst, diagonal = _grid(rows, cols, is_open)
    length = np.where(diagonal, 14, 10)

    def factor():
        f = _field(rng, rows, cols)
        return np.clip(np.floor(1.5 + 3.5 * (f[src] + f[dst])), 1, 8).astype(np.int64)

    costs = [length, length * factor(), length * factor(), factor(), np.ones_like(length)][:d]
    return (n, rowptr, dst.astype(np.uint32), np.stack(costs).astype(np.uint32)), reached


def _random_grid(rng, rows, cols, d):
    """A grid whose arcs cost U[1, 10] under every objective."""
    rowptr, src, dst, _ = _grid(rows, cols, np.ones(rows * cols, bool))
    return rows * cols, rowptr, dst.astype(np.uint32), rng.integers(1, 11, (d, len(src)), dtype=np.uint32)


def _csr(n, src, dst, cost):
    order = np.lexsort((dst, src))
    rowptr = np.zeros(n + 1, np.uint64)
    np.cumsum(np.bincount(src, minlength=n), out=rowptr[1:])
    return n, rowptr, dst[order].astype(np.uint32), np.ascontiguousarray(cost[:, order]).astype(np.uint32)


def _route(rng, rows, cols, windows, d):
    """A time-expanded ship route: cells x time windows, three speeds, weather
    that drifts from window to window; a goal node that the destination cell
    reaches at no cost in every window. The d objectives of a move are its
    length, then the length times a weather response of its own each."""
    _, src, dst, diagonal = _grid(rows, cols, np.ones(rows * cols, bool))
    cells, length = rows * cols, np.where(diagonal, 14.0, 10.0)
    y, x = np.divmod(np.arange(cells), cols)
    weather = np.zeros((d, windows, cells))
    for f in weather:
        for _ in range(6):
            cy, cx, sigma, height = rng.random() * rows, rng.random() * cols, 1.5 + 2.5 * rng.random(), 0.5 + 0.5 * rng.random()
            vy, vx = rng.uniform(-0.6, 0.6, 2)
            w = np.arange(windows)[:, None]
            f += height * np.exp(-((y - cy - vy * w) ** 2 + (x - cx - vx * w) ** 2) / (2 * sigma**2))
        f /= f.max()
    tails, heads, costs = [], [], []
    for speed, took in ((3, 1), (2, 2), (1, 3)):
        for w in range(windows - took):
            f = 0.5 * (weather[:, w][:, src] + weather[:, w][:, dst])
            c = [length]
            for k in range(1, d):
                c.append(rng.integers(1, 101, len(src)) if k == 11 else length * ((speed if k % 3 == 1 else 1) + (8 if k % 2 else 4) * f[k]))
            tails.append(src * windows + w)
            heads.append(dst * windows + w + took)
            costs.append(np.floor(np.stack(c) + 0.5).astype(np.int64))
    goal = cells * windows
    tails.append((cells - 1) * windows + np.arange(windows))
    heads.append(np.full(windows, goal))
    costs.append(np.zeros((d, windows), np.int64))
    return _csr(goal + 1, np.concatenate(tails), np.concatenate(heads), np.concatenate(costs, 1))


def _road(rng, side, d):
    """A road-like graph: side x side jittered points, each joined both ways
    to its 4 nearest; length, length x U{1..4}, U[0, 50], U[1, 100]."""
    y, x = np.mgrid[0:side, 0:side] + rng.uniform(-0.5, 0.5, (2, side, side))
    near = [(a, b) for a in (-2, -1, 0, 1, 2) for b in (-2, -1, 0, 1, 2) if a or b]
    far = np.full((len(near), side, side), np.float32(1e9))
    for f, (a, b) in zip(far, near):
        here = (slice(max(0, -a), side - max(0, a)), slice(max(0, -b), side - max(0, b)))
        there = (slice(max(0, a), side - max(0, -a)), slice(max(0, b), side - max(0, -b)))
        f[here] = (y[there] - y[here]) ** 2 + (x[there] - x[here]) ** 2
    pick = np.argpartition(far, 4, axis=0)[:4].reshape(4, -1)
    shift = np.array([a * side + b for a, b in near])
    u = np.tile(np.arange(side * side), 4)
    v = u + shift[pick].reshape(-1)
    pair = np.unique(np.minimum(u, v) * (side * side) + np.maximum(u, v))
    u, v = np.divmod(pair, side * side)
    y, x = y.reshape(-1), x.reshape(-1)
    length = np.floor(1e4 * np.hypot(y[u] - y[v], x[u] - x[v]) / side + 0.5).astype(np.int64)
    m = len(pair)
    cost = np.stack([length, length * rng.integers(1, 5, m), rng.integers(0, 51, m), rng.integers(1, 101, m)][:d])
    return _csr(side * side, np.concatenate([u, v]), np.concatenate([v, u]), np.concatenate([cost, cost], 1))


def _graph(case, rng):
    """(graph, start, goal, cells reached from the start or None)."""
    d = case["d"]
    if case["graph"] == "ship":
        g, reached = _ship(rng, case["rows"], case["cols"], d)
        return g, 0, g[0] - 1, reached
    if case["graph"] == "grid":
        g = _random_grid(rng, case["rows"], case["cols"], d)
        return g, 0, g[0] - 1, None
    if case["graph"] == "route":
        g = _route(rng, case["rows"], case["cols"], case["windows"], d)
        return g, 0, g[0] - 1, None
    side, far = case["side"], case["far"]
    g = _road(rng, side, d)
    r, c = (int(q) for q in rng.integers(0, side - far, 2))
    return g, r * side + c, (r + far) * side + c + far // 2, None


def _pairs(case, rng, reached):
    """Start and goal of every query of a batch: reached cells, the goal at a
    Chebyshev distance of U[near, far] from its start."""
    rows, cols = case["rows"], case["cols"]
    cells = np.flatnonzero(reached)
    starts, goals = [], []
    while len(starts) < case["queries"]:
        s = int(rng.choice(cells))
        r, c = divmod(s, cols)
        h = int(rng.integers(case["near"], case["far"] + 1))
        a, b = (h if rng.random() < 0.5 else -h), int(rng.integers(-h, h + 1))
        a, b = (a, b) if rng.random() < 0.5 else (b, a)
        if 0 <= r + a < rows and 0 <= c + b < cols and reached[(r + a) * cols + c + b]:
            starts.append(s)
            goals.append((r + a) * cols + c + b)
    return np.array(starts, np.uint32), np.array(goals, np.uint32)


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # a short voyage on a small corridor, many objectives: the smallest call, all launches and latency
        {"name": "route-4x5x12-d8", "call": "solve", "graph": "route", "rows": 4, "cols": 5, "windows": 12, "d": 8},
        # the plain two-objective grid query of the first benchmark workload
        {"name": "grid-32-d2", "call": "solve", "graph": "grid", "rows": 32, "cols": 32, "d": 2},
        # an ordinary ship-routing query at an odd size, library defaults
        {"name": "ship-97x89-d3", "call": "solve", "graph": "ship", "rows": 97, "cols": 89, "d": 3},
        # a longer one with the default window: thousands of steps
        {"name": "ship-160-d3", "call": "solve", "graph": "ship", "rows": 160, "cols": 160, "d": 3},
        # the benchmark's headline query at its tuned window: the largest single search
        {"name": "ship-256-d3-wide", "call": "solve", "graph": "ship", "rows": 256, "cols": 256, "d": 3, "window": 262144},
        # first-in first-out order and costs only, five objectives
        {"name": "ship-96-d5-fifo-costs", "call": "solve", "graph": "ship", "rows": 96, "cols": 96, "d": 5, "window": 4096, "fifo": True, "costs_only": True},
        # the twelve-objective time-expanded route: label processing dominates
        {"name": "route-6x8x24-d12", "call": "solve", "graph": "route", "rows": 6, "cols": 8, "windows": 24, "d": 12},
        # a query across a large sparse road-like graph: the heuristic is most of it
        {"name": "road-447-d2", "call": "solve", "graph": "road", "side": 447, "far": 100, "d": 2},
        # a captured batch of uneven queries on the five-objective grid
        {"name": "batch-128-ship-256-d5", "call": "batch", "graph": "ship", "rows": 256, "cols": 256, "d": 5, "queries": 128, "near": 16, "far": 64, "window": 1024, "captured": True},
        # a batch of more queries than run at once, library defaults
        {"name": "batch-400-ship-128-d3", "call": "batch", "graph": "ship", "rows": 128, "cols": 128, "d": 3, "queries": 400, "near": 16, "far": 64},
        # the heuristic alone, read back: planning that keeps it for many starts
        {"name": "heuristic-ship-256-d5", "call": "heuristic", "graph": "ship", "rows": 256, "cols": 256, "d": 5},
        # a session of the server: a burst of queries over a grid and a ship grid, of two to five objectives
        {"name": "serve-64", "call": "serve", "graph": "ship", "rows": 128, "cols": 128, "d": 5, "queries": 64, "near": 8, "far": 48, "window": 256},
    ]


def draw(rng):
    def size(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    call = rng.choice(["solve"] * 5 + ["batch", "batch", "heuristic", "serve"])
    if call == "solve":
        graph = rng.choice(["grid", "ship", "ship", "route", "road"])
        if graph == "route":
            rows, cols = size(3, 7), size(3, 9)
            return {"call": call, "graph": graph, "rows": rows, "cols": cols, "windows": size(8, min(26, 1200 // (rows * cols))), "d": rng.randint(6, 12)}
        if graph == "road":
            d = rng.choice([2, 2, 3, 4])
            return {"call": call, "graph": graph, "side": size(120, 447), "far": size(8, {2: 100, 3: 36, 4: 20}[d]), "d": d}
        if graph == "grid":
            d = rng.choice([2, 3])
            most = 64 if d == 2 else 17
            return {"call": call, "graph": graph, "rows": size(5, most), "cols": size(5, most), "d": d}
        d = rng.choice([1, 2, 3, 3, 4, 5])
        window = rng.choice([0, 0, 4096, 65536])
        rows = size(16, {1: 256, 2: 224, 3: 176, 4: 120, 5: 96}[d])
        case = {"call": call, "graph": graph, "rows": rows, "cols": max(12, rows - rng.randint(0, 9)), "d": d, "window": window}
        return dict(case, fifo=True, costs_only=True) if rng.random() < 0.25 else case
    rows = size(64, 256)
    cols = max(56, rows - rng.randint(0, 9))
    if call == "heuristic":
        if rng.random() < 0.4:
            return {"call": call, "graph": "road", "side": size(60, 447), "far": 8, "d": rng.randint(1, 4)}
        return {"call": call, "graph": "ship", "rows": rows, "cols": cols, "d": rng.randint(1, 5)}
    near = rng.randint(4, 16)
    case = {"call": call, "graph": "ship", "rows": rows, "cols": cols, "d": rng.randint(2, 5), "near": near, "far": size(near + 8, min(64, cols // 2))}
    if call == "serve":
        return dict(case, rows=min(rows, 160), cols=min(cols, 160), far=min(case["far"], 40), queries=size(8, 64), window=256)
    case = dict(case, queries=size(4, 400), window=rng.choice([0, 0, 1024]))
    return dict(case, captured=True) if rng.random() < 0.4 else case


def _inputs(case, seed):
    rng = np.random.default_rng(seed)
    return _graph(case, rng) + (rng,)


def prepare(case, seed):
    (n, rowptr, col, cost), start, goal, reached, rng = _inputs(case, seed)
    state = {"call": case["call"], "graph": opmos.opmos_graph(n, case["d"], rowptr, col, cost), "start": start, "goal": goal}
    options = {"window": case.get("window") or None}
    flags = opmos.FLAG_NO_PATHS * bool(case.get("costs_only")) | opmos.FLAG_FIFO * bool(case.get("fifo")) | opmos.FLAG_GRAPH * bool(case.get("captured"))
    options["flags"] = flags or None
    state["options"] = options
    if case["call"] != "heuristic":
        state["out"], state["used"] = _buffers(case), {}
    if case["call"] in ("batch", "serve"):
        state["starts"], state["goals"] = _pairs(case, rng, reached)
    if case["call"] == "serve":  # a second graph beside it, and the graph and objectives of each query
        side = 24
        n2, rowptr2, col2, cost2 = _random_grid(rng, side, side, 2)
        state["graphs"] = [state["graph"], opmos.opmos_graph(n2, 2, rowptr2, col2, cost2)]
        queries = []
        for s, t in zip(state["starts"].tolist(), state["goals"].tolist()):
            if rng.random() < 0.25:
                a, b = (int(q) for q in rng.integers(0, side * side, 2))
                queries.append((1, 2, a, b))
            else:
                queries.append((0, int(rng.integers(2, case["d"] + 1)) if case["d"] > 2 else case["d"], s, t))
        state["queries"] = queries
    return state


def _room(case):
    """How many solutions and path nodes a program keeps room for: it takes
    the results of its queries into arrays of its own, one after the other."""
    if case["call"] != "solve":
        return 64 * case["queries"], 4096 * case["queries"]
    long = {"grid": 1.5, "ship": 1.5, "route": 0.5, "road": 2.5}[case["graph"]] * max(case.get(k, 0) for k in ("rows", "cols", "windows", "far"))
    solutions = 4096 if case["d"] <= 2 else 16384
    return solutions, int(min(4_000_000, solutions * (long + 16)))


def _buffers(case):
    solutions, nodes = _room(case)
    queries = case.get("queries", 1)
    out = {"counts": np.zeros(queries, np.int64), "costs": np.zeros(solutions * case["d"], np.uint32)}
    if not case.get("costs_only"):
        out |= {"offsets": np.zeros(solutions + queries, np.uint32), "nodes": np.zeros(nodes, np.uint32), "edges": np.zeros(nodes, np.uint64)}
    return out


def _keep(state, results):
    """The results, one after the other, in the program's own arrays."""
    out, used = state["out"], {}

    def put(name, values):
        at = used.get(name, 0)
        used[name] = at + values.size
        if used[name] > out[name].size:
            raise RuntimeError(f"no room for {used[name]} values of {name}")
        out[name][at : used[name]] = values.reshape(-1)

    for i, r in enumerate(results):
        out["counts"][i] = len(r.costs)
        put("costs", r.costs)
        if r.paths is not None:
            put("offsets", r.paths.offsets)
            put("nodes", r.paths.nodes)
            put("edges", r.paths.edges)
    for name, before in state["used"].items():  # what an earlier, longer answer left
        out[name][used[name] : before] = 0
    state["used"] = used
    return out


def _serve(state):
    server = opmos.opmos_server(state["graphs"], mem_budget_bytes=SERVE_MEMORY, **state["options"])
    try:
        queries, done, waiting, at, began = state["queries"], {}, [], 0, time.monotonic()
        while len(done) < len(queries):
            if at < len(queries):
                try:
                    waiting.append((at, server.submit(*queries[at])))
                    at += 1
                except opmos.OpmosError as e:  # the queue is full: collect first
                    if e.code != opmos.ERR_CAPACITY:
                        raise
            left = []
            for i, ticket in waiting:
                status, result = server.poll(ticket)
                if status == opmos.PENDING:
                    left.append((i, ticket))
                elif status != opmos.OK:
                    raise RuntimeError(f"served query {i} ended with status {status}")
                else:
                    done[i] = result
            waiting = left
            if time.monotonic() - began > SERVE_SECONDS:
                raise RuntimeError("the server does not finish")
        return [done[i] for i in range(len(queries))]
    finally:
        server.close()


def run(state):
    call, graph = state["call"], state["graph"]
    if call == "heuristic":
        return opmos.opmos_heur(graph, state["goal"]).copy()
    if call == "batch":
        out = opmos.opmos_solve_batch(graph, state["starts"], state["goals"], **state["options"])
        for i, (status, _) in enumerate(out):
            if status != opmos.OK:
                raise RuntimeError(f"batch query {i} ended with status {status}")
        return _keep(state, [r for _, r in out])
    if call == "serve":
        return _keep(state, _serve(state))
    result = opmos.opmos_solve(graph, state["start"], state["goal"], **state["options"])
    return _keep(state, [result])


def work(case):
    """The graph read once, and what comes out of a known size: a front's size
    is not known before the search, so results other than the heuristic's are
    left out. Comparisons and additions of integers are not counted."""
    d = case["d"]
    if case["graph"] == "road":
        n, m = case["side"] ** 2, 4.9 * case["side"] ** 2
    else:
        cells = case["rows"] * case["cols"]
        arcs = 8 * cells - 6 * (case["rows"] + case["cols"]) + 4
        n, m = cells, arcs
        if case["graph"] == "ship":
            m *= 0.93
        if case["graph"] == "route":
            n, m = cells * case["windows"] + 1, arcs * (3 * case["windows"] - 6) + case["windows"]
    bytes_ = 4 * (n + 1) + 4 * m * (d + 1)
    if case["call"] == "heuristic":
        bytes_ += 4 * d * n
    return {"bytes": bytes_ + 8 * case.get("queries", 1), "flops": 0}


# ---------------------------------------------------------------------------
# the same results in plain Python
# ---------------------------------------------------------------------------
def _shortest(n, tails, arcs, goal):
    """Shortest distance of every node to goal: tails[v] and arcs[v] list the
    arcs that enter v as (tail, cost)."""
    far = [0xFFFFFFFF] * n
    far[goal] = 0
    heap = [(0, goal)]
    while heap:
        at, v = heapq.heappop(heap)
        if at > far[v]:
            continue
        for u, c in zip(tails[v], arcs[v]):
            if at + c < far[u]:
                far[u] = at + c
                heapq.heappush(heap, (at + c, u))
    return far


def _distances(g, goal, d):
    n, rowptr, col, cost = g
    src = np.repeat(np.arange(n), np.diff(rowptr).astype(np.int64))
    order = np.argsort(col, kind="stable")
    cut = np.cumsum(np.bincount(col, minlength=n))[:-1]
    tails = [t.tolist() for t in np.split(src[order], cut)]
    return np.array([_shortest(n, tails, [a.tolist() for a in np.split(cost[k][order], cut)], goal) for k in range(d)], np.uint32)


def _front(g, start, goal, d):
    """The cost-unique Pareto front from start to goal, in lexicographic
    order: labels leave a heap in that order, and one stays unless a cost at
    its node is as low in every objective."""
    n, rowptr, col, cost = g
    rowptr, col, cost = rowptr.tolist(), col.tolist(), cost.T.tolist()
    kept = [np.zeros((0, d), np.int64) for _ in range(n)]
    heap = [((0,) * d, start)]
    while heap:
        at, v = heapq.heappop(heap)
        if (kept[v] <= at).all(1).any() or (kept[goal] <= at).all(1).any():
            continue
        kept[v] = np.vstack([kept[v], np.array(at, np.int64)])
        if v != goal:
            for e in range(rowptr[v], rowptr[v + 1]):
                heapq.heappush(heap, (tuple(a + b for a, b in zip(at, cost[e])), col[e]))
    return kept[goal].astype(np.uint32)


def exact(case, seed):
    if case["call"] == "heuristic":
        g, _, goal, _, _ = _inputs(case, seed)
        return _distances(g, goal, case["d"])
    small = {"grid": case.get("rows", 0) * case.get("cols", 0) <= 1100 and case["d"] == 2,
             "route": case.get("rows", 0) * case.get("cols", 0) <= 20 and case.get("windows", 99) <= 12}
    if case["call"] == "solve" and small.get(case["graph"]):
        g, start, goal, _, _ = _inputs(case, seed)
        # several paths may carry one cost vector: only the costs are one answer
        front = _front(g, start, goal, case["d"])
        costs = np.zeros_like(_buffers(case)["costs"])
        costs[: front.size] = front.reshape(-1)
        return {"counts": np.array([len(front)], np.int64), "costs": costs, "offsets": None, "nodes": None, "edges": None}
    return None
