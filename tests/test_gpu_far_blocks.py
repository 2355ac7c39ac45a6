"""The far set of an SSSP with a distance threshold on graphs of more than
2^24 vertices, where a bit stands for a block of 64 or 128 vertices: distances
equal those of the same graph with its vertices packed."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from paper_1711_00231_gb300 import lb
from paper_1711_00231_gb300 import serve as sv

pytestmark = pytest.mark.gpu

SIZES = [1 << 24, (1 << 24) + 1, (1 << 24) + 63, (1 << 25) - 1, 1 << 25, (1 << 25) + 1, (1 << 25) + 129]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1711_00231_gb300 import _build
    _build.build()


def spread(g, n):
    """g with its vertices spread over n, the last one at n - 1: (graph, new
    ids).  Vertex 1, which nothing reaches, gets n / 2 (or n) edges of
    weight 1, so that the first interval's width (32 * mean weight / mean degree)
    stays about that of g."""
    new = np.arange(g.n, dtype=np.int64) * ((n - 1) // (g.n - 1))
    new[-1] = n - 1
    pad, first = n // 2 if g.name == "uniform" else n, int(g.offsets[1])
    off = np.zeros(n + 1, np.int64)
    off[new + 1] = g.degrees()
    off[2] = pad
    join = lambda x, y: np.concatenate([x[:first], y, x[first:]])
    cols = join(new[g.cols].astype(np.int32), np.arange(pad, dtype=np.int32))
    w = join(g.weights, np.ones(pad, np.uint32))
    return gg.CSRGraph(n, g.m + pad, np.cumsum(off), cols, w, g.name, {}), new


@pytest.fixture(scope="module")
def packed():
    """Graph, source and distances: a uniform graph (long lists, the threshold
    after a few iterations) and a grid (after 32)."""
    out = {}
    for name, g, src in (("uniform", gg.erdos_renyi(300001, 1200000, seed=6), None), ("grid", gg.grid(900, 1100, seed=2), 450 * 1100 + 7)):
        src = int(gg.pick_sources(g, 1, seed=3)[0]) if src is None else src
        ref, ov = oracle.dijkstra(g, src)
        assert not ov
        g.name = name
        out[name] = (g, src, ref)
    return out


def same(got, ref, new):
    want = np.full(got.size, 0xFFFFFFFF, np.uint32)
    want[new] = ref
    return np.array_equal(got, want)


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("name", ["uniform", "grid"])
def test_blocks_of_every_size(packed, name, n):
    g, src, ref = packed[name]
    big, new = spread(g, n)
    G = lb.Graph.from_csr(big)
    try:
        d, rc = G.sssp(int(new[src]), "WD")
        assert rc == lb.LB_OK and same(d, ref, new)
        relaxed = G.stats()["edges_relaxed"]
        G.set_options(loop_mode=1)  # plain order: the threshold was in force
        G.sssp(int(new[src]), "WD")
        assert relaxed < 0.8 * G.stats()["edges_relaxed"]
    finally:
        G.close()


@pytest.mark.parametrize("n", [(1 << 24) + 63, (1 << 25) + 129])
def test_blocks_in_the_engine(packed, n):
    import torch
    g, src, ref = packed["grid"]
    big, new = spread(g, n)
    G = lb.Graph.from_csr(big)
    S = sv.Server([G], slots=2, mem_fraction=0.05)
    try:
        out = torch.empty(n, dtype=torch.int32, device="cuda")
        status = S.run_batch([sv.Request(0.0, 0, int(new[src]), "sssp")], [out], timeout_s=120.0)
        torch.cuda.synchronize()
        assert status[0] == lb.LB_OK and same(out.cpu().numpy().view(np.uint32), ref, new)
    finally:
        S.close()
        G.close()
