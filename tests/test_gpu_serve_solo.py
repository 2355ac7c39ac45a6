"""Queries that one CTA of the serving kernel runs alone (short lists), with
the distance threshold of SSSP: results must equal the oracle's when lists
move between the single CTA and many, at the rule's sizes, across launches
that end part way, and with saturated distances."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from paper_1711_00231_gb300 import lb
from paper_1711_00231_gb300 import serve as sv

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1711_00231_gb300 import _build
    _build.build()


def fan(k, deg):
    """A source, k middle vertices of out-degree deg, a shared layer, a tail."""
    mid = 1 + np.arange(k)
    low = 1 + k + np.arange(max(deg, 1))
    src = np.concatenate([np.zeros(k, int), np.repeat(mid, deg), low])
    dst = np.concatenate([mid, np.tile(low, k)[:k * deg], np.full(low.size, 1 + k + low.size)])
    n = 2 + k + low.size
    return gg.from_edges(n, src, dst, 1 + (np.arange(src.size) * 37) % 200)


def graphs():
    over = gg.grid(40, 40, seed=1)
    over.weights[:] = np.random.default_rng(0).integers(1 << 27, 1 << 30, over.m)
    heavy = gg.grid(160, 170, seed=4)
    heavy.weights[:] = np.where(np.random.default_rng(1).random(heavy.m) < 0.5, 0, 100000)
    return [gg.grid(300, 333, seed=2), gg.grid(700, 650, seed=3), gg.rmat(13, 8, seed=5), gg.erdos_renyi(40000, 160000, seed=6),
            fan(8, 64), fan(8, 65), fan(1000, 8), fan(1100, 8), gg.from_edges(3, [0, 1], [1, 2], [4, 5]),
            gg.from_edges(1, [], [], []), over, heavy]


@pytest.mark.parametrize("launch_ms", [0, 1])
def test_solo_levels_match_oracle(launch_ms):
    import torch
    cg = graphs()
    G = [lb.Graph.from_csr(g) for g in cg]
    S = sv.Server(G, slots=24, mem_fraction=0.05, launch_ms=launch_ms)
    try:
        reqs = []
        for gi, g in enumerate(cg):
            for src in sorted({0, g.n // 2, g.n - 1}):
                reqs += [sv.Request(0.0, gi, int(src), "bfs"), sv.Request(0.0, gi, int(src), "sssp")]
        outs = [torch.empty(cg[r.graph].n, dtype=torch.int32, device="cuda") for r in reqs]
        status = S.run_batch(reqs, outs, timeout_s=120.0)
        torch.cuda.synchronize()
        for r, o, st in zip(reqs, outs, status):
            g, got = cg[r.graph], o.cpu().numpy()
            if r.kind == "bfs":
                assert st == lb.LB_OK and np.array_equal(got, oracle.bfs(g, r.src)[0]), (r.graph, r.src)
            else:
                ref, ov = oracle.dijkstra(g, r.src)
                assert st == (lb.LB_ERR_OVERFLOW if ov else lb.LB_OK), (r.graph, r.src, st)
                assert np.array_equal(got.view(np.uint32), ref), (r.graph, r.src)
    finally:
        S.close()
        for g in G:
            g.close()


@pytest.mark.parametrize("launch_ms", [0, 3])
def test_wide_fronts_match_oracle(launch_ms):
    # fronts of over a thousand vertices: the pulls cost more than the lists,
    # so intervals widen until their lists pass what one CTA takes
    import torch
    g = gg.grid(1500, 1400, seed=8)
    G = lb.Graph.from_csr(g)
    S = sv.Server([G], slots=4, mem_fraction=0.05, launch_ms=launch_ms)
    try:
        src = [0, g.n // 2 + 700]
        outs = [torch.empty(g.n, dtype=torch.int32, device="cuda") for _ in src]
        status = S.run_batch([sv.Request(0.0, 0, s, "sssp") for s in src], outs, timeout_s=120.0)
        torch.cuda.synchronize()
        for s, o, st in zip(src, outs, status):
            assert st == lb.LB_OK and np.array_equal(o.cpu().numpy().view(np.uint32), oracle.dijkstra(g, s)[0]), s
    finally:
        S.close()
        G.close()


def test_launch_limit_is_seen_after_every_pull():
    # 190,000 far vertices in blocks of their own, nearly all at one distance:
    # every pull reads all of their blocks (milliseconds) and queues ten
    # vertices.  A launch of 1 ms has to end after each.
    import torch
    chain, mids, far, groups, pads = 33, 5000, 190000, 24, 1000
    hub = chain + 1 + mids
    fv = hub + 32 * (1 + np.arange(far))
    sink = int(fv[-1]) + 1
    n = sink + 1 + pads
    deg = np.zeros(n, np.int64)
    deg[:chain] = 1
    deg[chain] = mids
    deg[chain + 1:hub] = 1
    deg[hub] = far
    deg[fv] = 1
    deg[sink + 1:] = 13000  # not reached: the mean weight stays 1
    off = np.concatenate([[0], np.cumsum(deg)])
    col = np.zeros(off[-1], np.int32)
    w = np.ones(off[-1], np.uint32)
    col[:chain] = 1 + np.arange(chain)
    col[off[chain]:off[chain + 1]] = chain + 1 + np.arange(mids)
    col[off[chain + 1]:off[hub]] = hub
    heavy = slice(off[hub], off[hub + 1])
    col[heavy] = fv
    dist = np.full(far, 1 << 30)
    dist[:10 * groups] = 64 << (np.arange(10 * groups) // 10)
    w[heavy] = dist
    col[off[fv]] = sink
    col[off[sink + 1]:] = np.tile(np.arange(13000), pads)
    sample = (np.arange(64) * off[-1]) >> 6
    assert (w[sample] == 1).all()
    g = gg.CSRGraph(n, int(off[-1]), off, col, w, "far", {})
    G = lb.Graph.from_csr(g)
    S = sv.Server([G], slots=4, mem_fraction=0.05, launch_ms=1)
    try:
        out = torch.empty(n, dtype=torch.int32, device="cuda")
        status = S.run_batch([sv.Request(0.0, 0, 0, "sssp")], [out], timeout_s=120.0)
        torch.cuda.synchronize()
        assert status[0] == lb.LB_OK and np.array_equal(out.cpu().numpy().view(np.uint32), oracle.dijkstra(g, 0)[0])
        assert S.info()["kernel_launches"] >= groups // 2
    finally:
        S.close()
        G.close()


def test_no_threshold_in_a_random_graphs_tail():
    # the lists of iterations 32 and on are the query's last, short ones: no
    # more iterations than in plain order (the host loop's)
    import torch
    g = gg.erdos_renyi(300000, 480000, seed=1)
    src = 73589
    G = lb.Graph.from_csr(g)
    G.set_options(loop_mode=1)
    ref, rc = G.sssp(src, "WD")
    assert rc == lb.LB_OK and np.array_equal(ref, oracle.dijkstra(g, src)[0])
    plain = G.stats()["iterations"]
    t = G.trace()["edges"]
    assert plain > 36 and ((t[32:] >= 4096) & (t[32:] <= 32768)).any()
    S = sv.Server([G], slots=2, mem_fraction=0.05)
    try:
        out = torch.empty(g.n, dtype=torch.int32, device="cuda")
        S.submit(0, src, "sssp", out)
        done = []
        while not done:
            done = S.poll()
        assert done[0][1] == lb.LB_OK and np.array_equal(out.cpu().numpy().view(np.uint32), ref)
        assert done[0][3] <= plain + 3  # the order inside an iteration may change its number by a few
    finally:
        S.close()
        G.close()


def test_far_set_spread_over_the_graph():
    # 1% of the edges heavy: their far ends keep thousands of blocks alive, so
    # that pulls outweigh lists and intervals widen
    import torch
    g = gg.grid(1024, 1024, seed=1)
    g.weights[:] = np.where(np.random.default_rng(1).random(g.m) < 0.01, 1000000, 1)
    G = lb.Graph.from_csr(g)
    S = sv.Server([G], slots=4, mem_fraction=0.05)
    try:
        src = [0, g.n // 2 + 300]
        outs = [torch.empty(g.n, dtype=torch.int32, device="cuda") for _ in src]
        status = S.run_batch([sv.Request(0.0, 0, s, "sssp") for s in src], outs, timeout_s=120.0)
        torch.cuda.synchronize()
        for s, o, st in zip(src, outs, status):
            assert st == lb.LB_OK and np.array_equal(o.cpu().numpy().view(np.uint32), oracle.dijkstra(g, s)[0]), s
    finally:
        S.close()
        G.close()


@pytest.mark.parametrize("k,deg", [(512, 8), (513, 8), (4095, 1), (4096, 1), (4097, 1)])
def test_bfs_lists_at_the_single_cta_limit(k, deg):
    import torch
    g = fan(k, deg)
    G = lb.Graph.from_csr(g)
    S = sv.Server([G], slots=4, mem_fraction=0.05)
    try:
        outs = [torch.empty(g.n, dtype=torch.int32, device="cuda") for _ in range(2)]
        status = S.run_batch([sv.Request(0.0, 0, 0, "bfs"), sv.Request(0.0, 0, 1, "bfs")], outs, timeout_s=60.0)
        torch.cuda.synchronize()
        for s, (o, st) in enumerate(zip(outs, status)):
            assert st == lb.LB_OK and np.array_equal(o.cpu().numpy(), oracle.bfs(g, s)[0]), s
    finally:
        S.close()
        G.close()


@pytest.mark.parametrize("policy", [0, 1])
def test_stop_with_queries_in_flight(policy):
    # strips of half a second and more, one of them an SSSP whose threshold is
    # in force, beside a graph of long lists: a stop returns at once, and the
    # queries go on at the next poll
    import time
    import torch
    cg = [gg.grid(4, 20000, seed=1), gg.grid(64, 8000, seed=2), gg.erdos_renyi(1 << 20, 1 << 23, seed=3)]
    G = [lb.Graph.from_csr(g) for g in cg]
    S = sv.Server(G, slots=16, mem_fraction=0.1, launch_ms=5000, policy=policy)
    try:
        for wanted in ([(0, "sssp")], [(0, "bfs")], [(1, "sssp")], [(2, "sssp"), (0, "sssp"), (1, "bfs"), (0, "bfs")]):
            outs = [torch.empty(cg[g].n, dtype=torch.int32, device="cuda") for g, _ in wanted]
            torch.cuda.synchronize()
            tick = {S.submit(g, 0, kind, o): i for i, ((g, kind), o) in enumerate(zip(wanted, outs))}
            for pause in (0.0, 0.004, 0.05):
                time.sleep(pause)
                t0 = time.perf_counter()
                S.stop()
                assert time.perf_counter() - t0 < 1.0
                for c in S.poll():  # starts the engine again
                    assert c[1] == lb.LB_OK
                    del tick[c[0]]
            end = time.perf_counter() + 60
            while tick and time.perf_counter() < end:
                for c in S.poll():
                    assert c[1] == lb.LB_OK
                    del tick[c[0]]
            assert not tick
            torch.cuda.synchronize()
            for (gi, kind), o in zip(wanted, outs):
                got = o.cpu().numpy()
                ref = oracle.bfs(cg[gi], 0)[0] if kind == "bfs" else oracle.dijkstra(cg[gi], 0)[0].view(np.int32)
                assert np.array_equal(got, ref), (gi, kind)
        # an engine is destroyed with a query in flight
        last = torch.empty(cg[1].n, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        S.submit(1, 0, "sssp", last)
        time.sleep(0.02)
        t0 = time.perf_counter()
        S.close()
        assert time.perf_counter() - t0 < 1.0
    finally:
        S.close()
        for g in G:
            g.close()
