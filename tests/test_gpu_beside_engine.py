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
    torch.cuda.synchronize()

    class Busy:
        def start(self):
            S.submit(0, 0, "sssp", out)
            # under way: the engine's kernel has taken it
            while S.state()["consumed"] < 1:
                time.sleep(0.001)

        def still(self):
            return not S.poll()

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
