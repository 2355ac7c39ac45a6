"""EP's edge-id flush entry by entry (entries averaging 16 edges or more) and
HP's sub-iterations served by threads, warps and CTAs over spread entries, at
the edges of their rules; results must equal the oracle's."""
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


def layered(deg, width=700, layers=6, seed=0):
    """Layers of vertices of out-degree deg (one vertex in ten: ten times that)."""
    r = np.random.default_rng(seed)
    src, dst = [np.zeros(width, int)], [1 + np.arange(width)]
    for k in range(layers - 1):
        d = np.where(np.arange(width) % 10 == 0, 10 * deg, deg)
        u = np.repeat(1 + k * width + np.arange(width), d)
        src.append(u)
        dst.append(1 + (k + 1) * width + r.integers(0, width, u.size))
    src, dst = np.concatenate(src), np.concatenate(dst)
    return gg.from_edges(1 + layers * width, src, dst, r.integers(1, 256, src.size), clean=False)


def check(G, g, src, strategies):
    lev = oracle.bfs(g, src)[0]
    dist = oracle.dijkstra(g, src)[0]
    for s in strategies:
        assert np.array_equal(G.bfs(src, s), lev), s
        d, rc = G.sssp(src, s)
        assert rc == lb.LB_OK and np.array_equal(d, dist), s


@pytest.mark.parametrize("deg", [1, 8, 9, 15, 16, 17, 61])
def test_ep_runs_of_edge_ids(deg):
    # averages on both sides of 16 edges per entry, runs that start at every
    # 16-byte phase of the list
    g = layered(deg, seed=deg)
    G = lb.Graph.from_csr(g)
    try:
        check(G, g, 0, ["EP", "EP_NOCHUNK"])
    finally:
        G.close()


@pytest.mark.parametrize("opts", [dict(mdt_override=1), dict(mdt_override=33), dict(mdt_override=100, thread_max=1),
                                  dict(mdt_override=100, hp_warp_max=32), dict(mdt_override=5000, hp_warp_max=64),
                                  dict(mdt_override=7, hp_depth=2)])
@pytest.mark.parametrize("deg", [3, 40])
def test_hp_sub_iterations_binned(deg, opts):
    g = layered(deg, seed=deg)
    G = lb.Graph.from_csr(g)
    try:
        G.set_options(hp_threshold=-1, **opts)
        check(G, g, 0, ["HP"])
        G.set_options(hp_threshold=256)
        check(G, g, 3, ["HP"])
    finally:
        G.close()
