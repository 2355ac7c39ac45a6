"""Queries beside a serving engine that holds 3 CTAs per SM: what fits in the
room it leaves runs at once, not when the engine goes idle."""
import time

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


@pytest.fixture
def busy():
    """An engine with one query of half a second and more in flight."""
    import torch
    g = gg.grid(4, 100000, seed=1)
    G = lb.Graph.from_csr(g)
    S = sv.Server([G], slots=2, ctas_per_sm=3, mem_fraction=0.05)
    out = torch.empty(g.n, dtype=torch.int32, device="cuda")
    ref = oracle.dijkstra(g, 0)[0]
    torch.cuda.synchronize()

    class Busy:
        def start(self):
            S.submit(0, 0, "sssp", out)
            # under way: the engine's kernel has taken it
            while S.state()["active"] < 1:
                time.sleep(0.001)

        def still(self):
            return not S.poll()

        def finish(self):
            done, end = [], time.perf_counter() + 30
            while not done and time.perf_counter() < end:
                done = S.poll()
            assert done and done[0][1] == lb.LB_OK
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy().view(np.uint32), ref)

    yield Busy()
    S.close()
    G.close()


@pytest.mark.parametrize("strategy", ["EP", "HP", "NS", "BS"])
def test_first_query_of_a_strategy_beside_a_busy_engine(busy, strategy):
    g = gg.rmat(12, 8, seed=3)
    W = lb.Graph.from_csr(g)
    W.bfs(5, strategy)  # the driver loads a kernel at its first launch, which waits for the GPU
    G = lb.Graph.from_csr(g)
    try:
        busy.start()
        lev = G.bfs(5, strategy)
        assert busy.still()
        assert np.array_equal(lev, oracle.bfs(g, 5)[0])
    finally:
        G.close()
        W.close()


def test_wd_query_beside_a_busy_engine(busy):
    # it waits for the engine to go idle; both results are exact
    g = gg.rmat(14, 8, seed=4)
    G = lb.Graph.from_csr(g)
    try:
        for kind in ("bfs", "sssp"):
            busy.start()
            if kind == "bfs":
                assert np.array_equal(G.bfs(5, "WD"), oracle.bfs(g, 5)[0])
            else:
                d, rc = G.sssp(5, "WD")
                assert rc == lb.LB_OK and np.array_equal(d, oracle.dijkstra(g, 5)[0])
            busy.finish()
    finally:
        G.close()


def test_wd_queries_of_several_threads_and_streams():
    # their launches fill the GPU and wait for one another as wholes
    import threading
    import torch
    graphs = [gg.grid(150, 170, seed=1), gg.rmat(15, 16, seed=2), gg.erdos_renyi(50000, 300000, seed=3)]
    ref = [(oracle.bfs(g, 7)[0], oracle.dijkstra(g, 7)[0].view(np.int32)) for g in graphs]
    G = [lb.Graph.from_csr(g) for g in graphs]
    wrong = []

    def work(k):
        g, st = graphs[k], torch.cuda.Stream()
        outs = [torch.empty(g.n, dtype=torch.int32, device="cuda") for _ in range(2)]
        torch.cuda.synchronize()
        for _ in range(20):
            G[k].bfs_dev(7, "WD", outs[0], None, st)
            G[k].sssp_dev(7, "WD", outs[1], None, st)
            st.synchronize()
            if G[k].stats()["status"] != lb.LB_OK or not all(np.array_equal(o.cpu().numpy(), r) for o, r in zip(outs, ref[k])):
                wrong.append(k)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(graphs))]
    try:
        for t in threads:
            t.start()
        for t in threads:
            t.join(60)
        assert not wrong and not any(t.is_alive() for t in threads)
    finally:
        for g in G:
            g.close()
