"""Performance cases: what a program that uses this library has it do, through
its public entry points.

A case is one kind of call on one seeded synthetic graph (R-MAT, grid or
Erdos-Renyi, the shapes of the library's tests and benchmark):

  call "query"  one device-output BFS or SSSP query on a resident graph
  call "batch"  a list of sources through the batched host-output call
  call "serve"  a burst of queries over a mix of resident graphs through the
                serving engine

Graphs are generated on the GPU from the seed (every seed is another graph and
another source) and handed to the library as device arrays.
"""
import math

import torch

from paper_1711_00231_gb300 import lb, serve

# R-MAT quadrant probabilities a, b, c (d = 1 - a - b - c)
A, B, C = 0.57, 0.19, 0.19


def listed():
    return [
        # The smallest call: a BFS on a small skewed graph, a handful of levels
        # of a few microseconds each, where latency and launches count.
        dict(name="bfs_rmat14", call="query", kind="bfs", strategy="WD", graph="rmat", scale=14, ef=16),
        # An ordinary skewed graph, both kinds, from its largest hub.
        dict(name="bfs_rmat20", call="query", kind="bfs", strategy="WD", graph="rmat", scale=20, ef=16),
        dict(name="sssp_rmat20", call="query", kind="sssp", strategy="WD", graph="rmat", scale=20, ef=16),
        # The largest skewed graph: the throughput case of both kinds.
        dict(name="bfs_rmat24", call="query", kind="bfs", strategy="WD", graph="rmat", scale=24, ef=32),
        dict(name="sssp_rmat24", call="query", kind="sssp", strategy="WD", graph="rmat", scale=24, ef=32),
        # Road-network-like graphs: thousands of small worklists.  One of
        # ordinary size with ragged sides, one at the full size.
        dict(name="bfs_grid_1000x1537", call="query", kind="bfs", strategy="WD", graph="grid", rows=1000, cols=1537),
        dict(name="sssp_grid_4096x4096", call="query", kind="sssp", strategy="WD", graph="grid", rows=4096, cols=4096),
        # A uniform random graph: no hubs, every worklist entry short.
        dict(name="sssp_er_8m", call="query", kind="sssp", strategy="WD", graph="er", n=1 << 23, m=33554432),
        # The other ways of handing out the work, which programs that compare
        # the strategies run beside WD: edge-based and hierarchical.
        dict(name="sssp_ep_rmat20", call="query", kind="sssp", strategy="EP", graph="rmat", scale=20, ef=16),
        dict(name="bfs_hp_rmat20", call="query", kind="bfs", strategy="HP", graph="rmat", scale=20, ef=16),
        # Results wanted on the host: several sources in one call, each
        # result copied to pinned memory.
        dict(name="batch_bfs_rmat18", call="batch", kind="bfs", strategy="WD", graph="rmat", scale=18, ef=16, k=16),
        # Serving: a burst of BFS and SSSP queries over a mix of resident
        # graphs of uneven sizes.
        dict(name="serve_mix", call="serve", graphs=12, lo=12, hi=18, queries=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any call, kind and graph shape of the listed ones, with
    sizes spread over their whole ranges."""
    call = rng.choices(["query", "batch", "serve"], [0.76, 0.12, 0.12])[0]
    if call == "serve":
        return dict(call="serve", graphs=rng.randint(3, 12), lo=12, hi=rng.randint(14, 18),
                    queries=_log_int(rng, 8, 128))
    case = dict(call=call, kind=rng.choice(["bfs", "sssp"]))
    case["strategy"] = rng.choices(["WD", "EP", "HP"], [0.8, 0.1, 0.1])[0] if call == "query" else "WD"
    case["graph"] = rng.choice(["rmat", "grid", "er"])
    small = call == "batch" or case["strategy"] != "WD"
    if case["graph"] == "rmat":
        case["scale"] = rng.randint(14, 20 if small else 24)
        case["ef"] = rng.randint(8, 16 if small else 32)
    elif case["graph"] == "grid":
        top = 600 if small else 4096
        case["rows"] = _log_int(rng, 64, top)
        case["cols"] = _log_int(rng, 64, top)
    else:
        n = _log_int(rng, 20000, (1 << 20) if small else (1 << 23))
        case["n"] = n
        case["m"] = n * rng.randint(2, 8)
        if not small:
            case["m"] = min(case["m"], 33554432)
    if call == "batch":
        case["k"] = rng.randint(2, 16)
    return case


# ------------------------------------------------------------------ graphs


def _csr(keys, n, shift):
    """CSR arrays of the distinct edges keys = u << shift | v without
    self-loops, adjacency sorted by destination."""
    mask = (1 << shift) - 1
    keys = torch.unique(keys[(keys >> shift) != (keys & mask)])
    bounds = torch.arange(n + 1, dtype=torch.int64, device="cuda") << shift
    off = torch.searchsorted(keys, bounds)
    return off, (keys & mask).to(torch.int32)


def _rmat(scale, ef, gen):
    total, chunk = ef << scale, 1 << 26
    parts = []
    for k in range(0, total, chunk):
        cnt = min(chunk, total - k)
        key = torch.zeros(cnt, dtype=torch.int64, device="cuda")
        for level in range(scale):
            r = torch.rand(cnt, generator=gen, device="cuda")
            u = r >= A + B
            v = ((r >= A) & ~u) | (r >= A + B + C)
            key += (u.to(torch.int64) << (2 * scale - 1 - level)) + (v.to(torch.int64) << (scale - 1 - level))
        parts.append(key)
    off, col = _csr(torch.cat(parts) if len(parts) > 1 else parts[0], 1 << scale, scale)
    w = torch.randint(1, 256, (col.numel(),), generator=gen, device="cuda", dtype=torch.int32)
    return off, col, w


def _er(n, m, gen):
    shift = max(1, (n - 1).bit_length())
    u = torch.randint(0, n, (m,), generator=gen, device="cuda")
    v = torch.randint(0, n, (m,), generator=gen, device="cuda")
    off, col = _csr((u << shift) | v, n, shift)
    w = torch.randint(1, 256, (col.numel(),), generator=gen, device="cuda", dtype=torch.int32)
    return off, col, w


def _grid_weights(rows, cols, gen, wmax):
    right = torch.randint(1, wmax + 1, (rows, cols - 1), generator=gen, device="cuda", dtype=torch.int32)
    down = torch.randint(1, wmax + 1, (rows - 1, cols), generator=gen, device="cuda", dtype=torch.int32)
    return right, down


def _grid(rows, cols, gen, wmax):
    """4-neighbour grid, vertex r * cols + c, one weight per undirected edge."""
    right, down = _grid_weights(rows, cols, gen, wmax)
    v = torch.arange(rows * cols, dtype=torch.int32, device="cuda").view(rows, cols)
    # neighbours in the order of their ids: up, left, right, down
    nb = torch.stack([v - cols, v - 1, v + 1, v + cols], dim=2)
    w = torch.zeros(rows, cols, 4, dtype=torch.int32, device="cuda")
    w[1:, :, 0] = down
    w[:, 1:, 1] = right
    w[:, :-1, 2] = right
    w[:-1, :, 3] = down
    have = w > 0
    off = torch.zeros(rows * cols + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(have.sum(dim=2).reshape(-1), 0)
    return off, nb[have], w[have]


def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return gen


def _arrays(case, seed):
    gen = _generator(seed)
    if case["graph"] == "rmat":
        return _rmat(case["scale"], case["ef"], gen)
    if case["graph"] == "er":
        return _er(case["n"], case["m"], gen)
    return _grid(case["rows"], case["cols"], gen, case.get("wmax", 1000))


def _graph(arrays):
    off, col, w = arrays
    torch.cuda.synchronize()  # the library copies them on a stream of its own
    return lb.Graph(off, col, w, off.numel() - 1, col.numel(), device_arrays=True)


def _sources(case, arrays, seed, k):
    """R-MAT query: the largest hub at scales 15 to 20; SSSP query on a grid: a
    corner; else uniform among vertices with out-edges."""
    off = arrays[0]
    deg = off[1:] - off[:-1]
    if case["graph"] == "grid" and k == 1 and case["kind"] == "sssp":
        return [0]
    if case["graph"] == "rmat" and k == 1 and 14 < case["scale"] <= 20:
        return [int(torch.argmax(deg))]
    cand = torch.nonzero(deg > 0).view(-1)
    pick = torch.randint(0, cand.numel(), (k,), generator=_generator(seed + 7919), device="cuda")
    return cand[pick].tolist()


def _mix(case, seed):
    """The serving mix: two thirds R-MAT (scales lo..hi, edge factor 8, 16 or
    32), one third grids, weights U[1,255]; the sizes depend on the case
    alone, the edges on the seed."""
    specs = []
    for i in range(case["graphs"]):
        if i % 3 == 2:
            side = (256, 512, 384, 200)[(i // 3) % 4]
            specs.append(dict(graph="grid", rows=side, cols=side + 31 * (i % 2), wmax=255))
        else:
            specs.append(dict(graph="rmat", scale=case["lo"] + (5 * i) % (case["hi"] - case["lo"] + 1),
                              ef=(8, 16, 32)[i % 3 + i % 2]))
    arrays = [_arrays(s, seed * 1000 + i) for i, s in enumerate(specs)]
    reqs, place = [], 0
    for q in range(case["queries"]):
        g = (q * 5 + q // 7) % len(arrays)
        src = _sources(specs[g], arrays[g], seed * 1000 + q, 2)[0]
        n = arrays[g][0].numel() - 1
        reqs.append((g, src, "sssp" if (q // len(arrays) + q) % 2 else "bfs", place, n))
        place += n
    return specs, arrays, reqs, place


# ------------------------------------------------------------ the interface


def prepare(case, seed):
    if case["call"] == "serve":
        _, arrays, reqs, total = _mix(case, seed)
        graphs = [_graph(a) for a in arrays]
        out = torch.empty(total, dtype=torch.int32, device="cuda")
        server = serve.Server(graphs, slots=64, mem_fraction=0.05)
        return dict(call="serve", server=server, out=out, views=[out[p:p + n] for _, _, _, p, n in reqs],
                    reqs=[serve.Request(0.0, g, src, kind) for g, src, kind, _, _ in reqs])
    arrays = _arrays(case, seed)
    state = dict(call=case["call"], kind=case["kind"], strategy=case["strategy"], graph=_graph(arrays))
    n = arrays[0].numel() - 1
    if case["call"] == "batch":
        state["sources"] = _sources(case, arrays, seed, case["k"])
        state["pinned"] = torch.empty(case["k"], n, dtype=torch.int32, pin_memory=True)
        state["out"] = state["pinned"].numpy() if case["kind"] == "bfs" else state["pinned"].numpy().view("u4")
    else:
        state["source"] = _sources(case, arrays, seed, 1)[0]
        state["out"] = torch.empty(n, dtype=torch.int32, device="cuda")
    return state


def run(state):
    if state["call"] == "serve":
        state["server"].run_batch(state["reqs"], state["views"])
        return state["out"]
    g = state["graph"]
    if state["call"] == "batch":
        if state["kind"] == "bfs":
            g.bfs_batch(state["sources"], state["strategy"], state["out"])
        else:
            g.sssp_batch(state["sources"], state["strategy"], state["out"])
        return state["pinned"]
    query = g.bfs_dev if state["kind"] == "bfs" else g.sssp_dev
    query(state["source"], state["strategy"], state["out"], None, torch.cuda.current_stream())
    return state["out"]


def _sizes(case):
    if case["graph"] == "rmat":
        return 1 << case["scale"], case["ef"] << case["scale"]
    if case["graph"] == "er":
        return case["n"], case["m"]
    rows, cols = case["rows"], case["cols"]
    return rows * cols, 2 * (rows * (cols - 1) + (rows - 1) * cols)


def _work(case, kind, times=1):
    """Every offset, column (and weight) read once, every result written
    once; one comparison per edge (and one sum with weights)."""
    n, m = _sizes(case)
    sssp = kind == "sssp"
    return times * (8 * (n + 1) + (8 if sssp else 4) * m + 4 * n), times * (2 if sssp else 1) * m


def work(case):
    if case["call"] == "serve":
        by = fl = 0
        shapes = []
        for i in range(case["graphs"]):
            if i % 3 == 2:
                side = (256, 512, 384, 200)[(i // 3) % 4]
                shapes.append(dict(graph="grid", rows=side, cols=side + 31 * (i % 2)))
            else:
                shapes.append(dict(graph="rmat", scale=case["lo"] + (5 * i) % (case["hi"] - case["lo"] + 1),
                                   ef=(8, 16, 32)[i % 3 + i % 2]))
        for q in range(case["queries"]):
            b, f = _work(shapes[(q * 5 + q // 7) % len(shapes)], "sssp" if (q // len(shapes) + q) % 2 else "bfs")
            by, fl = by + b, fl + f
        return {"bytes": by, "flops": fl}
    by, fl = _work(case, case["kind"], case.get("k", 1))
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------- exact values


def _exact_one(arrays, src, kind):
    """Least fixed point of d[v] = min(d[u] + w(u, v)) in 64-bit integers by
    full sweeps over the edges; -1 where unreachable."""
    off, col, w = arrays
    n = off.numel() - 1
    u = torch.repeat_interleave(torch.arange(n, device="cuda"), off[1:] - off[:-1])
    far = 1 << 60
    d = torch.full((n,), far, dtype=torch.int64, device="cuda")
    d[src] = 0
    to = col.to(torch.int64)
    step = 1 << 27
    while True:
        new = d.clone()
        for k in range(0, to.numel(), step):
            s = slice(k, k + step)
            cost = d[u[s]] + (w[s].to(torch.int64) if kind == "sssp" else 1)
            new.scatter_reduce_(0, to[s], cost, "amin")
        if torch.equal(new, d):
            break
        d = new
    d[d >= far] = -1
    return d


def _exact_grid(rows, cols, right, down, src):
    """The same on a grid, by shifted minima instead of edge lists."""
    far = 1 << 60
    d = torch.full((rows, cols), far, dtype=torch.int64, device="cuda")
    d.view(-1)[src] = 0
    while True:
        before = d.clone()
        for _ in range(64):
            d[:, 1:] = torch.minimum(d[:, 1:], d[:, :-1] + right)
            d[:, :-1] = torch.minimum(d[:, :-1], d[:, 1:] + right)
            d[1:] = torch.minimum(d[1:], d[:-1] + down)
            d[:-1] = torch.minimum(d[:-1], d[1:] + down)
        if torch.equal(before, d):
            return d.view(-1)


def _exact(case, arrays, src, kind, seed):
    if case["graph"] != "grid":
        return _exact_one(arrays, src, kind)
    rows, cols = case["rows"], case["cols"]
    if kind == "bfs":
        r = torch.arange(rows, device="cuda").view(-1, 1) - src // cols
        c = torch.arange(cols, device="cuda").view(1, -1) - src % cols
        return (r.abs() + c.abs()).reshape(-1)
    if rows * cols * (rows + cols) > 3e9:  # over about 20 seconds of sweeps
        return None
    right, down = _grid_weights(rows, cols, _generator(seed), case.get("wmax", 1000))
    return _exact_grid(rows, cols, right, down, src)


def exact(case, seed):
    if case["call"] == "serve":
        specs, arrays, reqs, total = _mix(case, seed)
        if case["queries"] > 64:
            return None
        out = torch.empty(total, dtype=torch.int64, device="cuda")
        for g, src, kind, place, n in reqs:
            out[place:place + n] = _exact(specs[g], arrays[g], src, kind, seed * 1000 + g)
        return out
    arrays = _arrays(case, seed)
    if case["call"] == "batch":
        rows = [_exact(case, arrays, s, case["kind"], seed) for s in _sources(case, arrays, seed, case["k"])]
        return None if any(r is None for r in rows) else torch.stack(rows)
    return _exact(case, arrays, _sources(case, arrays, seed, 1)[0], case["kind"], seed)
