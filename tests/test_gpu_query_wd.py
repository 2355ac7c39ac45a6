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
