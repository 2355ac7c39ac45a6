"""The whole-query WD launch (the WD device loop): one cooperative launch per
query with a grid barrier per level, and a team of CTAs for small lists.
Cases sit at the edges of its own rules; results must equal the oracle's."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from paper_1711_00231_gb300 import lb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1711_00231_gb300 import _build
    _build.build()


def check(G, g, src):
    assert np.array_equal(G.bfs(src, "WD"), oracle.bfs(g, src)[0]), src
    d, rc = G.sssp(src, "WD")
    ref, ov = oracle.dijkstra(g, src)
    assert rc == (lb.LB_ERR_OVERFLOW if ov else lb.LB_OK) and np.array_equal(d, ref), src


@pytest.mark.parametrize("deg", [8 * 256 - 1, 8 * 256, 8 * 256 + 1, 9 * 256 + 1, 20000])
def test_hub_spanning_many_tile_starts(deg):
    # hubs found in level 1 whose lists cover 8 or more 256-edge grains: the
    # grain starts of a longer entry are written by the whole warp
    hubs = np.arange(1, 41)
    leaves = 41 + np.arange(deg)
    src = np.concatenate([np.zeros(40, int)] + [np.full(deg, h) for h in hubs[::7]] + [hubs])
    dst = np.concatenate([hubs] + [leaves for _ in hubs[::7]] + [np.full(40, 41)])
    g = gg.from_edges(41 + deg, src, dst, 1 + np.arange(src.size) % 250)
    G = lb.Graph.from_csr(g)
    try:
        check(G, g, 0)
        check(G, g, 8)
    finally:
        G.close()


def test_failed_queries_leave_the_next_one_clean():
    # every query has synchronisation words of its own: two that end at the
    # barrier's time limit in a row, then exact ones
    g = gg.grid(40, 50, seed=1)
    G = lb.Graph.from_csr(g)
    try:
        check(G, g, 7)
        for _ in range(2):
            G.set_options(test_barrier_skip=1)
            with pytest.raises(lb.LbError) as ei:
                G.bfs(0, "WD")
            assert ei.value.status == lb.LB_ERR_TIMEOUT
        G.set_options(test_barrier_skip=0)
        check(G, g, 0)
        check(G, g, 1999)
    finally:
        G.close()


@pytest.mark.parametrize("opts", [dict(ctas_per_sm=1), dict(ctas_per_sm=2, wd_tile=256), dict(small_edges=1),
                                  dict(small_edges=1 << 24)])
def test_grid_and_team_sizes(opts):
    for g, src in ((gg.rmat(15, 16, seed=2), 3), (gg.grid(150, 70, seed=5), 33), (gg.from_edges(1, [], [], []), 0)):
        G = lb.Graph.from_csr(g)
        try:
            G.set_options(**opts)
            check(G, g, src)
        finally:
            G.close()


@pytest.mark.parametrize("deg", [1, 2, 4, 8, 32, 33])
def test_fast_levels_at_their_degree_limits(deg):
    # layered graphs whose entries have exactly deg edges: lists that fit the
    # team's segments, that just do not (33), and that grow past them
    L, width = 30, 3000
    r = np.random.default_rng(deg)
    n = 1 + L * width
    src, dst = [np.zeros(min(width, 40), int)], [1 + np.arange(min(width, 40))]
    for k in range(L - 1):
        u = np.repeat(1 + k * width + np.arange(width), deg)
        src.append(u)
        dst.append(1 + (k + 1) * width + (u * 7 + r.integers(0, 60, u.size)) % width)
    src, dst = np.concatenate(src), np.concatenate(dst)
    g = gg.from_edges(n, src, dst, r.integers(1, 1000, src.size), clean=False)
    G = lb.Graph.from_csr(g)
    try:
        check(G, g, 0)
        G.set_options(small_edges=100)
        check(G, g, 0)
        check(G, g, 1 + 5 * width)
    finally:
        G.close()


def test_fast_levels_on_small_and_large_graphs():
    # the segments' size changes at 32768 vertices
    for R, C in ((181, 181), (182, 181), (64, 5000), (3, 40000)):
        g = gg.grid(R, C, seed=R)
        G = lb.Graph.from_csr(g)
        try:
            check(G, g, 0)
            check(G, g, R * C // 2)
        finally:
            G.close()


def far_graph(kind):
    # uniform random graphs whose lists grow past the threshold rule's size
    # early; n is not a multiple of the far set's 128-vertex blocks
    g = gg.erdos_renyi(300001, 1200000, seed=6)
    r = np.random.default_rng(4)
    if kind == "zero":
        g.weights[:] = r.integers(0, 9, g.m)
    elif kind == "gaps":
        g.weights[:] = np.where(r.random(g.m) < 0.5, 1, 1 << 20)
    elif kind == "equal":
        g.weights[:] = 1
    elif kind == "overflow":
        g.weights[:] = r.integers(1 << 28, 1 << 31, g.m)
    return g


@pytest.mark.parametrize("kind", ["uniform", "zero", "gaps", "equal", "overflow"])
def test_sssp_distance_threshold(kind):
    import torch
    g = far_graph(kind)
    G = lb.Graph.from_csr(g)
    try:
        src = int(gg.pick_sources(g, 1, seed=3)[0])
        ref, ov = oracle.dijkstra(g, src)
        d, rc = G.sssp(src, "WD")
        assert rc == (lb.LB_ERR_OVERFLOW if ov else lb.LB_OK) and np.array_equal(d, ref)
        assert ov == (kind == "overflow")
        relaxed = G.stats()["edges_relaxed"]
        # any 4-byte alignment of the caller's buffer
        buf = torch.empty(g.n + 1, dtype=torch.int32, device="cuda")
        G.sssp_dev(src, "WD", buf[1:], None, torch.cuda.current_stream())
        torch.cuda.synchronize()
        assert np.array_equal(buf[1:].cpu().numpy().view(np.uint32), ref)
        if kind == "uniform":
            # the host loop keeps the plain order: the threshold was in force
            G.set_options(loop_mode=1)
            G.sssp(src, "WD")
            assert relaxed < 0.8 * G.stats()["edges_relaxed"]
    finally:
        G.close()


def test_sssp_distance_threshold_on_a_grid():
    # high diameter: the threshold comes in after 32 iterations, the intervals
    # widen, and lists move between the team and the whole grid
    g = gg.grid(900, 1100, seed=2)
    G = lb.Graph.from_csr(g)
    try:
        for opts in (dict(), dict(small_edges=0), dict(small_edges=2000, ctas_per_sm=1)):
            G.set_options(**opts)
            d, rc = G.sssp(450 * 1100 + 7, "WD")
            assert rc == lb.LB_OK and np.array_equal(d, oracle.dijkstra(g, 450 * 1100 + 7)[0])
    finally:
        G.close()


@pytest.mark.parametrize("off", ["line-1", "line", "line+255", "rounds"])
def test_lists_walked_in_claimed_slices(off):
    # one CTA per SM: lists of 16 grains of 256 edges per warp and more are
    # claimed in slices; level 1 has exactly E list edges, over ragged entries
    import torch
    warps = 8 * torch.cuda.get_device_properties(0).multi_processor_count
    line = 16 * 256 * warps
    E = {"line-1": line - 1, "line": line, "line+255": line + 255, "rounds": 2 * line + line // 3 + 77}[off]
    r = np.random.default_rng(len(off))
    leaves = 200000
    deg = []
    while sum(deg) < E:
        deg.append(int(min(r.choice([1, 2, 31, 33, 255, 257, 5000, 150000]), E - sum(deg))))
    deg = np.array(deg)
    H = deg.size
    first = np.repeat(np.cumsum(deg) - deg, deg)
    dst = 1 + H + (np.repeat(r.integers(0, leaves, H), deg) + np.arange(E) - first) % leaves
    src = np.repeat(1 + np.arange(H), deg)
    g = gg.from_edges(1 + H + leaves, np.concatenate([np.zeros(H, int), src]), np.concatenate([1 + np.arange(H), dst]),
                      1 + r.integers(0, 200, H + E))
    G = lb.Graph.from_csr(g)
    ref, ov = oracle.dijkstra(g, 0)
    lev = oracle.bfs(g, 0)[0]
    try:
        for tile in (256, 512, 8192, 32768):
            G.set_options(ctas_per_sm=1, wd_tile=tile)
            assert np.array_equal(G.bfs(0, "WD"), lev), tile
            assert list(G.trace()["edges"][:2]) == [H, E]
            d, rc = G.sssp(0, "WD")
            assert not ov and rc == lb.LB_OK and np.array_equal(d, ref), tile
    finally:
        G.close()


def swinging(rounds, width, chain, arms):
    """Lists that swing between the whole grid and the team: a hub's `width`
    edges, as many one-edge entries, one entry, then `chain` vertices of `arms`
    edges (too many for a fast level: regular levels of the team), the next hub."""
    src, dst, at = [], [], 0
    for _ in range(rounds):
        leaves = at + 1 + np.arange(width)
        end = at + 1 + width
        src += [np.full(width, at), leaves]
        dst += [leaves, np.full(width, end)]
        at = end
        for _ in range(chain):
            src.append(np.full(arms, at))
            dst.append(at + 1 + np.arange(arms))
            at += arms
        src.append(np.array([at]))
        dst.append(np.array([at + 1]))
        at += 1
    src, dst = np.concatenate(src), np.concatenate(dst)
    return gg.from_edges(at + 1, src, dst, 1 + (np.arange(src.size) * 31) % 500)


@pytest.mark.parametrize("width", [40000, 70000])
@pytest.mark.parametrize("chain", [0, 1, 2, 3, 4, 5])
def test_late_reads_of_a_steps_counters(width, chain):
    # CTAs outside the team read a step's counters when the team is levels
    # ahead: nothing may have cleared them
    g = swinging(12, width, chain, 50)
    G = lb.Graph.from_csr(g)
    try:
        for opts in (dict(), dict(small_edges=100)):
            G.set_options(test_barrier_skip=2, **opts)
            check(G, g, 0)
            modes = G.trace()["mode"]
            assert (modes == 4).sum() >= 12 and (modes == 0).sum() >= 12
    finally:
        G.close()


@pytest.mark.parametrize("kind", ["uniform", "gaps"])
def test_late_reads_with_a_distance_threshold(kind):
    g = far_graph(kind)
    src = int(gg.pick_sources(g, 1, seed=3)[0])
    ref, _ = oracle.dijkstra(g, src)
    G = lb.Graph.from_csr(g)
    try:
        for opts in (dict(), dict(small_edges=2000)):
            G.set_options(test_barrier_skip=2, **opts)
            d, rc = G.sssp(src, "WD")
            assert rc == lb.LB_OK and np.array_equal(d, ref)
    finally:
        G.close()


def test_failed_query_reports_nothing_of_the_one_before():
    g = gg.grid(40, 50, seed=1)
    G = lb.Graph.from_csr(g)
    try:
        for kind, query in (("bfs", G.bfs), ("sssp", G.sssp)):
            check(G, g, 7)
            assert G.stats()["iterations"] > 0 and len(G.trace()) > 0
            G.set_options(test_barrier_skip=1)
            with pytest.raises(lb.LbError):
                query(0, "WD")
            st = G.stats()
            assert st["status"] == lb.LB_ERR_TIMEOUT, kind
            assert [st[k] for k in ("iterations", "steps", "edges_relaxed", "pushes")] == [0, 0, 0, 0], kind
            assert len(G.trace()) == 0, kind
            G.set_options(test_barrier_skip=0)
    finally:
        G.close()


@pytest.mark.parametrize("before,edges,engages", [(6, 10.5, True), (6, 16, True), (6, 7.5, False), (5, 16, False)])
def test_threshold_rule_on_fast_levels(before, edges, engages):
    # `before` lists, then one of W one-edge entries that the team runs as a
    # fast level.  The threshold comes in there if at least 6 iterations and
    # fewer than a quarter of the graph's `edges` * W edges have been listed
    # with it: W by the hub's list, W by this one.  Behind it 50 vertices at
    # far distances: one list in plain order, many with a threshold.
    W, far = 20000, 50
    mids = before + np.arange(W)
    c = before + W
    y = c + 1 + np.arange(far)
    src = [np.arange(before - 1), np.full(W, before - 1), mids, np.full(far, c), y]
    dst = [1 + np.arange(before - 1), mids, np.full(W, c), y, np.full(far, c + far + 1)]
    w = [np.ones(before - 1), np.ones(W), np.ones(W), 100000 * (1 + np.arange(far)), np.ones(far)]
    m = int(edges * W)
    pad = m - sum(len(x) for x in src)
    u = c + far + 2 + np.arange(-(-pad // 4))  # not reached
    src.append(np.repeat(u, 4)[:pad])
    dst.append(np.tile(np.arange(4), u.size)[:pad])
    w.append(np.ones(pad))
    src, dst, w = (np.concatenate(x).astype(np.int64) for x in (src, dst, w))
    g = gg.from_edges(int(u[-1]) + 1, src, dst, w)
    assert g.m == m
    # the first width comes from 1024 evenly spaced weights: none of the far ones
    assert (g.weights[(np.arange(1024) * m) >> 10] == 1).all()
    G = lb.Graph.from_csr(g)
    try:
        d, rc = G.sssp(0, "WD")
        assert rc == lb.LB_OK and np.array_equal(d, oracle.dijkstra(g, 0)[0])
        t = G.trace()
        assert list(t["edges"][before - 1:before + 1]) == [W, W] and t["mode"][before] == 4
        plain = before + 3  # the lists before, of the W, of c, of the far vertices
        assert len(t) == plain if not engages else len(t) > plain + 3
    finally:
        G.close()


@pytest.mark.parametrize("hook,graph", [(3, "spokes"), (3, "swing"), (4, "grid"), (4, "swing"), (5, "grid"), (5, "spokes")])
def test_bounded_waits_of_the_team(hook, graph):
    # a CTA of the team that never arrives (3: regular steps, 4: fast levels)
    # or a team that never publishes (5): the waits run out, those of the CTAs
    # outside the team too, and the next queries are exact
    import time
    g = {"grid": lambda: gg.grid(40, 50, seed=1), "spokes": lambda: swinging(1, 100, 4, 60),
         "swing": lambda: swinging(3, 40000, 3, 50)}[graph]()
    G = lb.Graph.from_csr(g)
    try:
        check(G, g, 0)
        for query in (G.bfs, G.sssp):
            G.set_options(test_barrier_skip=hook)
            t = time.perf_counter()
            with pytest.raises(lb.LbError) as ei:
                query(0, "WD")
            assert ei.value.status == lb.LB_ERR_TIMEOUT
            assert 1.5 < time.perf_counter() - t < 8.0
            G.set_options(test_barrier_skip=0)
            check(G, g, 0)
    finally:
        G.close()


def test_bounded_wait_of_the_host_loops_small_levels():
    g = gg.grid(64, 64, seed=1)
    G = lb.Graph.from_csr(g)
    try:
        G.set_options(test_barrier_skip=1, loop_mode=1)
        for query in (G.bfs, G.sssp):
            with pytest.raises(lb.LbError) as ei:
                query(0, "WD")
            assert ei.value.status == lb.LB_ERR_TIMEOUT
        G.set_options(test_barrier_skip=0, loop_mode=1)
        check(G, g, 0)
        G.set_options(loop_mode=0)
        check(G, g, 0)
    finally:
        G.close()
