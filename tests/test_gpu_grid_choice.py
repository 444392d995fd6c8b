"""The number of CTAs the library chooses for a graph: enough for its arcs and
for its vertices."""
import numpy as np
import pytest

import oracle
from workloads import generators as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,least", [(1 << 20, 5000, 1 << 20), (200_000, 4000, 48), (30_000, 500, 7), (1000, 8000, 7)])
def test_vertices_count_too(n, m, least):
    import paper_2511_05895_gb300 as mf
    rng = np.random.default_rng(n)
    g = gen.from_edges(n, rng.integers(0, m // 50, m), rng.integers(0, m // 50, m), rng.integers(1, 100, m), 0, 1)
    full = mf.MaxFlowGraph(g.n, g.row_ptr, g.col, g.cap, g.s, g.t, grid_blocks=1 << 20)
    G = mf.MaxFlowGraph(g.n, g.row_ptr, g.col, g.cap, g.s, g.t)
    assert min(least, full.stats()["grid_blocks"]) <= G.stats()["grid_blocks"] <= full.stats()["grid_blocks"]
    G.solve()
    assert G.flow_value() == oracle.maxflow_fifo(g.n, g.row_ptr, g.col, g.cap, g.s, g.t)
    full.close()
    G.close()
