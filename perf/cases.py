"""The work a user of the framework has it do, as timed cases.

A case is a dict of plain values.  ``listed()`` gives the named ones,
``draw(rng)`` another one of the same ranges, ``prepare(case, seed)`` what a
program holds before the call (device inputs made from the seed, solvers,
servers, workspaces), ``run(state)`` one pass through the public entry points,
``work(case)`` the bytes and integer operations a pass cannot do without, and
``exact(case, seed)`` the same outputs from plain torch and numpy.

Kinds of case:
  solve   a whole solve (or its first `rounds` rounds) on a resident solver:
          reset, solve, and the objective, allotment, loads and table read;
  strict  the same with no overload allowed (Alg. 5);
  batch   many instances advanced by one planned, captured launch set;
  serve   requests submitted to the request server, every result taken;
  scan    the best-transfer table of a given allotment;
  road    the cost matrix of a road network.
"""
import math

import numpy as np
import torch

import paper_2304_06543_gb300 as lb

TINF = 2**31 - 1

# ------------------------------------------------------------------ cases ---


def listed():
    return [
        # the tiny configuration (2,000 x 20): an interactive what-if solve
        {"name": "solve_tiny", "kind": "solve", "n": 2000, "k": 20, "layout": "uniform",
         "scale": 100, "caps": "uniform", "cap_frac": 0.9, "pen_lo": 50, "pen_hi": 500,
         "qlen": 1, "rounds": -1},
        # a mid-size instance of the batched mix, solved alone
        {"name": "solve_mix", "kind": "solve", "n": 6007, "k": 126, "layout": "uniform",
         "scale": 100, "caps": "uniform", "cap_frac": 0.9, "pen_lo": 50, "pen_hi": 500,
         "qlen": 1, "rounds": -1},
        # the city configuration's centers, capacities and penalties, its units thinned out
        {"name": "solve_city", "kind": "solve", "n": 8000, "k": 500, "layout": "gmm",
         "scale": 1000, "caps": "zipf", "cap_frac": 0.8, "pen_lo": 200, "pen_hi": 2000,
         "qlen": 1, "rounds": -1},
        # the first rounds of the wide configuration (20,000 x 2,000): a
        # resumable solve whose table does not fit a cluster's shared memory
        {"name": "solve_wide", "kind": "solve", "n": 20000, "k": 2000, "layout": "gmm",
         "scale": 1000, "caps": "uniform", "cap_frac": 0.3, "pen_lo": 100, "pen_hi": 5000,
         "qlen": 1, "rounds": 800},
        # hard capacities, and costs past 32,767 (kept as int32)
        {"name": "strict_wide_costs", "kind": "strict", "n": 1500, "k": 40, "layout": "uniform",
         "scale": 50000, "caps": "uniform", "cap_frac": 0.9},
        # the batched mix: uneven instances in one captured launch set
        {"name": "batch_24", "kind": "batch", "m": 24, "n_lo": 500, "n_hi": 5000,
         "k_lo": 10, "k_hi": 400},
        # the serving stream's small requests, all at once, matrices on the device
        {"name": "serve_24", "kind": "serve", "m": 24, "n_lo": 500, "n_hi": 5000,
         "k_lo": 10, "k_hi": 400},
        # the table of one small instance: launch-bound
        {"name": "scan_tiny_i32", "kind": "scan", "n": 2000, "k": 20, "elem": 4,
         "layout": "uniform", "scale": 100},
        # short rows: an instance of the batched mix
        {"name": "scan_mix_i32", "kind": "scan", "n": 50001, "k": 126, "elem": 4,
         "layout": "uniform", "scale": 100},
        # the city-scale table
        {"name": "scan_city_i16", "kind": "scan", "n": 200000, "k": 500, "elem": 2,
         "layout": "gmm", "scale": 1000},
        # the memory-bound table (8 GB of costs)
        {"name": "scan_large_i16", "kind": "scan", "n": 2000000, "k": 2000, "elem": 2,
         "layout": "gmm", "scale": 1000},
        # the road-network pipeline's cost matrix
        {"name": "road_256", "kind": "road", "w": 256, "h": 256, "k": 109},
    ]


def _log(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choices(["solve", "scan", "strict", "batch", "serve", "road"],
                       [8, 6, 1, 2, 2, 1])[0]
    city = rng.random() < 0.5
    layout, scale = ("gmm", 1000) if city else ("uniform", rng.choice([100, 100, 50000]))
    if kind == "solve":
        k = _log(rng, 8, 600)
        n = _log(rng, 500, int(170000 / math.sqrt(k)))   # no more than the city-shaped solve
        lo, hi = (200, 2000) if city else (50, 500)
        if scale == 50000:
            lo, hi = 500 * lo, 500 * hi
        return {"kind": kind, "n": max(n, 2 * k), "k": k, "layout": layout, "scale": scale,
                "caps": "zipf" if city else "uniform",
                "cap_frac": rng.choice([0.3, 0.8, 0.85, 0.9, 1.1]), "pen_lo": lo, "pen_hi": hi,
                "qlen": rng.choice([1, 1, 1, 8]), "rounds": -1}
    if kind == "strict":
        k = _log(rng, 8, 100)
        return {"kind": kind, "n": max(_log(rng, 300, 4000), 2 * k), "k": k, "layout": layout,
                "scale": scale, "caps": "uniform", "cap_frac": rng.choice([0.7, 0.9, 1.2])}
    if kind in ("batch", "serve"):
        lo = _log(rng, 300, 1500)
        return {"kind": kind, "m": _log(rng, 3, 24), "n_lo": lo, "n_hi": 3 * lo,
                "k_lo": _log(rng, 8, 30), "k_hi": _log(rng, 60, 400)}
    if kind == "scan":
        k = _log(rng, 8, 2000)
        n = max(_log(rng, 1000, min(2000000, int(1.6e9 / k))), k)
        elem = 4 if scale == 50000 else rng.choice([2, 4])
        return {"kind": kind, "n": n, "k": k, "elem": elem, "layout": layout, "scale": scale}
    return {"kind": kind, "w": _log(rng, 24, 256), "h": _log(rng, 24, 256), "k": _log(rng, 5, 109)}


# ----------------------------------------------------------------- inputs ---


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _points(g, n, layout):
    """n demand points of the unit square: uniform, or 30 Gaussian clusters."""
    if layout == "uniform":
        return torch.rand(n, 2, generator=g, device="cuda")
    mean = torch.rand(30, 2, generator=g, device="cuda")
    sigma = 0.02 + 0.06 * torch.rand(30, 1, generator=g, device="cuda")
    comp = torch.randint(0, 30, (n,), generator=g, device="cuda")
    xy = mean[comp] + sigma[comp] * torch.randn(n, 2, generator=g, device="cuda")
    return xy.clamp_(0.0, 1.0)


def _costs(g, n, k, layout, scale, dtype, ld):
    """(n, ld) costs, columns 0..k filled: max(1, round(scale * distance *
    road factor)), road factor in [1, 1.5] per pair with clustered demand."""
    d, s = _points(g, n, layout), torch.rand(k, 2, generator=g, device="cuda")
    out = torch.zeros(n, ld, dtype=dtype, device="cuda")
    step = max(1, 100_000_000 // k)
    for a in range(0, n, step):
        b = min(n, a + step)
        x = torch.hypot(d[a:b, :1] - s[:, 0], d[a:b, 1:] - s[:, 1])
        if layout == "gmm":
            x *= 1.0 + 0.5 * torch.rand(b - a, k, generator=g, device="cuda")
        out[a:b, :k] = x.mul_(float(scale)).add_(0.5).floor_().clamp_(min=1.0).to(dtype)
    return out


def _split(weights, total):
    """`total` split over the weights in whole numbers, at least 1 each."""
    k = len(weights)
    total = max(total, k)
    cap = 1 + np.floor((total - k) * weights / weights.sum()).astype(np.int64)
    cap[:total - int(cap.sum())] += 1
    return cap.astype(np.int32)


def _caps_pens(rs, c):
    n, k = c["n"], c["k"]
    if c["caps"] == "zipf":
        wts = rs.permutation(1.0 / np.arange(1, k + 1) ** 1.2)
    else:
        wts = rs.random_sample(k) + 1e-3
    cap = _split(wts, int(c["cap_frac"] * n))
    pen = rs.randint(c.get("pen_lo", 1), c.get("pen_hi", 1) + 1, k).astype(np.int32)
    qtab = None
    if c.get("qlen", 1) > 1:     # a growing penalty per unit past capacity
        steps = rs.randint(0, c["pen_lo"] // 4 + 2, (k, c["qlen"])).astype(np.int32)
        steps[:, 0] = pen
        qtab = np.cumsum(steps, axis=1).astype(np.int32)
    return cap, pen, qtab


def _instance(c, seed):
    g, rs = _gen(seed), np.random.RandomState(seed % (1 << 31))
    cm = _costs(g, c["n"], c["k"], c["layout"], c["scale"], torch.int32, c["k"])
    return (cm,) + _caps_pens(rs, c)


def _mix(c, seed):
    """Instances of the batched mix: sizes log-uniform in the case's ranges,
    spread evenly so that every seed has about the same work; odd k among them."""
    out = []
    m = c["m"]
    for i in range(m):
        # low-discrepancy spread of the two sizes
        fn, fk = (i + 0.5) / m, (i * 0.6180339887498949 + 0.5) % 1.0
        n = int(c["n_lo"] * (c["n_hi"] / c["n_lo"]) ** fn)
        k = int(c["k_lo"] * (c["k_hi"] / c["k_lo"]) ** fk)
        one = {"n": n, "k": k, "layout": "uniform", "scale": 100, "caps": "uniform",
               "cap_frac": 0.9, "pen_lo": 50, "pen_hi": 500}
        out.append(_instance(one, seed * 64 + i) + (one,))
    return out


def _scan_inputs(c, seed):
    """Padded costs and an allotment: most units at their cheapest center,
    one in ten at the second cheapest (moved there by a full center)."""
    n, k = c["n"], c["k"]
    dtype = torch.int16 if c["elem"] == 2 else torch.int32
    ld = lb.cm_pitch(k, lb.CM_I16 if c["elem"] == 2 else lb.CM_I32)
    g = _gen(seed)
    cm = _costs(g, n, k, c["layout"], c["scale"], dtype, ld)
    assign = torch.empty(n, dtype=torch.int32, device="cuda")
    step = max(1, 50_000_000 // k)
    for a in range(0, n, step):
        x = cm[a:a + step, :k].to(torch.int32)
        first = x.argmin(dim=1, keepdim=True)
        x.scatter_(1, first, TINF)
        second = x.argmin(dim=1)
        moved = torch.rand(x.shape[0], generator=g, device="cuda") < 0.1
        assign[a:a + step] = torch.where(moved, second, first[:, 0]).to(torch.int32)
    return cm, ld, assign


def _road_graph(c, seed):
    """A w x h grid of jittered intersections, 4-neighbour roads and 15 % of
    the diagonals, length = 100 x distance x factor in [1, 1.5]; CSR, both
    directions.  k intersections hold a center, every other one a demand."""
    w, h, k = c["w"], c["h"], c["k"]
    rs = np.random.RandomState(seed % (1 << 31))
    V = w * h
    x, y = np.meshgrid(np.arange(w), np.arange(h))
    at = np.stack([x.ravel(), y.ravel()], 1) + 0.35 * (rs.random_sample((V, 2)) - 0.5)
    idx = np.arange(V).reshape(h, w)
    diag = rs.random_sample((h - 1, w - 1)) < 0.15
    a = np.concatenate([idx[:, :-1].ravel(), idx[:-1].ravel(), idx[:-1, :-1][diag]])
    b = np.concatenate([idx[:, 1:].ravel(), idx[1:].ravel(), idx[1:, 1:][diag]])
    length = np.hypot(*(at[a] - at[b]).T) * (1.0 + 0.5 * rs.random_sample(len(a)))
    wt = np.maximum(1, np.floor(100.0 * length + 0.5)).astype(np.int32)
    src, dst, wt = np.concatenate([a, b]), np.concatenate([b, a]), np.concatenate([wt, wt])
    o = np.lexsort((dst, src))
    row_ptr = np.zeros(V + 1, np.int32)
    row_ptr[1:] = np.cumsum(np.bincount(src, minlength=V))
    centers = np.sort(rs.permutation(V)[:k]).astype(np.int32)
    demand = np.setdiff1d(np.arange(V, dtype=np.int32), centers)
    return row_ptr, dst[o].astype(np.int32), wt[o], centers, demand


# -------------------------------------------------------- prepare and run ---


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "solve":
        cm, cap, pen, qtab = _instance(case, seed)
        st["solver"] = lb.Solver(cm, cap, pen, qtab=qtab)
        st["out"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
    elif kind == "strict":
        cm, cap, _, _ = _instance(case, seed)
        st["solver"] = lb.Solver(cm.cpu().numpy(), cap, None, strict=True)
        st["out"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
    elif kind == "batch":
        mix = _mix(case, seed)
        st["solvers"] = [lb.Solver(cm, cap, pen) for cm, cap, pen, _, _ in mix]
        st["batch"] = lb.Batch(st["solvers"])
        st["out"] = [torch.empty(s.n, dtype=torch.int32, device="cuda") for s in st["solvers"]]
    elif kind == "serve":
        st["requests"] = [x[:3] for x in _mix(case, seed)]
        st["server"] = lb.Server(8 << 30)
    elif kind == "scan":
        cm, ld, assign = _scan_inputs(case, seed)
        k = case["k"]
        wsb = lb.best_transfer_workspace(case["n"], k)
        st.update(cm=cm, ld=ld, assign=assign, wsb=wsb,
                  tc=torch.empty(k, k, dtype=torch.int32, device="cuda"),
                  td=torch.empty(k, k, dtype=torch.int32, device="cuda"),
                  ws=torch.empty(wsb, dtype=torch.uint8, device="cuda"))
    else:
        rp, col, w, cen, dem = (torch.from_numpy(x).cuda() for x in _road_graph(case, seed))
        st.update(rp=rp, col=col, w=w, cen=cen, dem=dem,
                  cm=torch.empty(len(dem), len(cen), dtype=torch.int32, device="cuda"))
    torch.cuda.synchronize()
    return st


def run(st):
    c = st["case"]
    kind = c["kind"]
    if kind in ("solve", "strict"):
        s = st["solver"]
        s.reset()
        s.solve(c.get("rounds", -1))
        tc, td = s.table()
        return {"objective": s.objective, "allotment": s.assignment(st["out"]),
                "loads": s.loads(), "tc": tc, "td": td}
    if kind == "batch":
        for s in st["solvers"]:
            s.reset()
        st["batch"].run()
        return {"objective": np.array([s.objective for s in st["solvers"]]),
                "allotment": [s.assignment(o) for s, o in zip(st["solvers"], st["out"])]}
    if kind == "serve":
        tickets = [st["server"].submit(*r) for r in st["requests"]]
        done = [st["server"].result(t) for t in tickets]
        return {"objective": np.array([info.objective for info, _ in done]),
                "allotment": [a for _, a in done]}
    if kind == "scan":
        lb.best_transfer(c["n"], c["k"], st["cm"], lb.CM_I16 if c["elem"] == 2 else lb.CM_I32,
                         st["ld"], st["assign"], st["tc"], st["td"], st["ws"], st["wsb"])
        return {"tc": st["tc"], "td": st["td"]}
    return lb.road_cm(st["rp"], st["col"], st["w"], st["cen"], st["dem"], st["cm"])


# ------------------------------------------------------------------- work ---


def _solve_work(n, k, scale, rounds=-1):
    """The costs once to find every unit's cheapest center, the allotted
    units' rows once more to enter the table, and the results."""
    w = 2 if scale * 1.5 * 1.42 < 32767 else 4
    r = n if rounds < 0 else min(n, rounds)
    return (n + r) * k * w + 4 * (n + k) + 8 * k * k, (n + r) * k


def work(case):
    kind = case["kind"]
    if kind in ("solve", "strict"):
        b, f = _solve_work(case["n"], case["k"], case["scale"], case.get("rounds", -1))
    elif kind in ("batch", "serve"):
        b = f = 0
        m = case["m"]
        for i in range(m):
            fn, fk = (i + 0.5) / m, (i * 0.6180339887498949 + 0.5) % 1.0
            n = int(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** fn)
            k = int(case["k_lo"] * (case["k_hi"] / case["k_lo"]) ** fk)
            x, y = _solve_work(n, k, 100)
            b, f = b + x, f + y
    elif kind == "scan":
        n, k = case["n"], case["k"]
        b, f = n * k * case["elem"] + 4 * n + 8 * k * k, n * k
    else:
        V, k = case["w"] * case["h"], case["k"]
        edges = int(2 * 2.15 * V)
        b, f = 4 * (V + 1 + 2 * edges + V) + 4 * (V - k) * k, edges * k
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ exact ---


def _exact_scan(c, seed):
    """The lexicographic minimum of (transfer cost, unit) per pair, as one
    64-bit key."""
    n, k = c["n"], c["k"]
    cm, _, assign = _scan_inputs(c, seed)
    none = torch.iinfo(torch.int64).max
    best = torch.full((k, k), none, dtype=torch.int64, device="cuda")
    step = max(1, 20_000_000 // k)
    for a in range(0, n, step):
        x = cm[a:a + step, :k].to(torch.int64)
        j = assign[a:a + step].to(torch.int64)
        key = (x - x.gather(1, j[:, None])) * (1 << 32)
        key += torch.arange(a, a + x.shape[0], device="cuda")[:, None]
        best.scatter_reduce_(0, j[:, None].expand(-1, k), key, "amin")
    best.fill_diagonal_(none)
    empty = best == none
    tc = torch.where(empty, TINF, best >> 32).to(torch.int32)
    td = torch.where(empty, -1, best & 0xFFFFFFFF).to(torch.int32)
    return {"tc": tc, "td": td}


def _exact_road(c, seed):
    """Shortest distances from every center by whole relaxation sweeps."""
    rp, col, w, cen, dem = _road_graph(c, seed)
    V, k = c["w"] * c["h"], c["k"]
    src = torch.from_numpy(np.repeat(np.arange(V), np.diff(rp))).cuda()
    dst, wt = torch.from_numpy(col).cuda().long(), torch.from_numpy(w).cuda().long()
    dist = torch.full((V, k), 1 << 40, dtype=torch.int64, device="cuda")
    dist[torch.from_numpy(cen).cuda().long(), torch.arange(k, device="cuda")] = 0
    at = dst[:, None].expand(-1, k)
    for sweep in range(V):
        old = dist.clone()
        dist.scatter_reduce_(0, at, old[src] + wt[:, None], "amin")
        if torch.equal(old, dist):
            break
    return dist[torch.from_numpy(dem).cuda().long()].to(torch.int32)


def _exact_solve(c, seed):
    """Alg. 2 (Alg. 5 when strict) as the paper states it, on whole arrays:
    the table row of every center that changed is rebuilt from its members."""
    strict = c["kind"] == "strict"
    cm, cap, pen, qtab = _instance(c, seed)
    cm = cm.cpu().numpy().astype(np.int64)
    cap = cap.astype(np.int64)
    n, k = cm.shape
    if strict and cap.sum() < n:     # a dummy center for what does not fit
        cm = np.hstack([cm, np.full((n, 1), cm.max() + 1)])
        cap = np.append(cap, n - cap.sum())
        k += 1
    q = (qtab if qtab is not None else pen[:, None]).astype(np.int64) if not strict else None
    INF = 1 << 60
    tc, td = np.full((k, k), INF), np.full((k, k), -1)
    assign, load = np.full(n, -1, np.int32), np.zeros(k, np.int64)
    low = cm.argmin(1)
    order = np.arange(n) if strict else np.argsort(cm.min(1), kind="stable")
    delta = 0

    def penalty(s, x):
        return q[s, min(x, q.shape[1]) - 1] if x >= 1 else 0

    def rebuild(s):
        d = np.nonzero(assign == s)[0]
        tc[s], td[s] = INF, -1
        if len(d):
            t = cm[d] - cm[d, s][:, None]
            i = t.argmin(0)
            tc[s], td[s] = t[i, np.arange(k)], d[i]
        tc[s, s], td[s, s] = INF, -1

    def search(W, sink, j):
        """Whole sweeps from j; `sink` holds the costs into the sink."""
        dist, par = np.full(k + 1, INF), np.full(k + 1, -1)
        full = np.hstack([W, sink[:, None]])
        full[:, j] = INF
        dist[j] = 0
        for _ in range(k + 2):
            lab = dist[:k].copy()
            cand = np.where((lab[:, None] >= INF) | (full >= INF), INF, lab[:, None] + full)
            u = cand.argmin(0)
            best = cand[u, np.arange(k + 1)]
            up = best < dist
            if not up.any():
                break
            dist[up], par[up] = best[up], u[up]
        path, v = [], par[k]
        if dist[k] < 0:
            while v != j:
                path.append(v)
                v = par[v]
            path.append(j)
        return int(dist[k]), [int(p) for p in path[::-1]]

    def move(path, to_last, free=()):
        ends = path[1:] + to_last
        units = [(-1 if (u, v) in free else int(td[u, v])) for u, v in zip(path, ends)]
        for x, v in zip(units, ends):
            if x >= 0:
                load[assign[x]] -= 1
                assign[x] = v
                load[v] += 1
        for s in set(path):
            rebuild(s)

    rounds = c.get("rounds", -1)
    for d in order[:n if rounds < 0 else rounds]:
        j = int(np.where(load < cap, cm[d], INF).argmin()) if strict else int(low[d])
        over = not strict and load[j] >= cap[j]
        delta += int(cm[d, j]) + (int(penalty(j, int(load[j] - cap[j] + 1))) if over else 0)
        assign[d], load[j] = j, load[j] + 1
        t = cm[d] - cm[d, j]
        t[j] = INF
        up = (t < tc[j]) | ((t == tc[j]) & (d < td[j]) & (t < INF))
        tc[j, up], td[j, up] = t[up], d
        W = tc
        free = ()
        if strict:      # a vacancy passes on for nothing
            room = load < cap
            W = np.where(room[:, None] & (tc > 0), 0, tc)
            W[np.arange(k), np.arange(k)] = INF
        cost, path = search(W, W[:, j].copy(), j)
        if path:
            if strict:
                free = {(u, v) for u, v in zip(path, path[1:] + [j]) if room[u] and tc[u, v] > 0}
            move(path, [j], free)
            delta += cost
        if over:
            qu = np.array([penalty(s, int(load[s] - cap[s] + 1)) for s in range(k)])
            sink = qu - penalty(j, int(load[j] - cap[j]))
            sink[j] = INF
            cost, path = search(tc, sink, j)
            if path:
                move(path, [])
                delta += cost
    tc[tc >= INF] = TINF
    return {"objective": int(delta), "allotment": assign, "loads": load.astype(np.int32),
            "tc": tc.astype(np.int32), "td": td.astype(np.int32)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "scan":
        return _exact_scan(case, seed)
    if kind == "road":
        return _exact_road(case, seed)
    if kind in ("solve", "strict") and case["n"] * case["k"] <= 100_000:
        return _exact_solve(case, seed)
    return None     # larger solves take minutes on whole arrays
