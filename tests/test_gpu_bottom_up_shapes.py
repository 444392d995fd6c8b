"""Bottom-up BFS levels in both shapes (64-vertex pieces when every warp gets
one, else 32-vertex pieces): vertex counts around the line between them for a
given grid, ragged last pieces, short rows, long rows and rows of more than 64
arcs, in the plain and in the push-pull search."""
import numpy as np
import pytest

import oracle
from tests._helpers import certify_gpu
from workloads import generators as gen

pytestmark = pytest.mark.gpu

LINE = 64 * 24   # vertices at which one CTA of 24 warps has a 64-vertex piece for each


@pytest.mark.parametrize("n", [65, LINE - 1, LINE, LINE + 1, LINE + 33, 3 * LINE + 17])
@pytest.mark.parametrize("deg", [3, 12, 70])
@pytest.mark.parametrize("mode", [0, 2])
def test_shapes(n, deg, mode):
    import paper_2511_05895_gb300 as mf
    rng = np.random.default_rng(n + deg)
    m = n * deg
    g = gen.from_edges(n, rng.integers(0, n, m), rng.integers(0, n, m), rng.integers(1, 60, m), 0, n - 1)
    cap = g.cap.copy()
    G = mf.MaxFlowGraph(g.n, g.row_ptr, g.col, cap, g.s, g.t, mode=mode, grid_blocks=1)
    G.solve()
    levels = G.stats()["bfs_bottom_up_levels"]
    assert G.flow_value() == oracle.maxflow_fifo(g.n, g.row_ptr, g.col, cap, g.s, g.t)
    for i in range(2):
        b = gen.mixed_batch(cap, max(1, g.m // 8), 1, 60, seed=5, index=i)
        G.apply_updates(b.edge_id, b.new_cap)
        gen.apply_batch(cap, b)
        f = G.flow_value()
        levels += G.stats()["bfs_bottom_up_levels"]
        assert f == oracle.maxflow_fifo(g.n, g.row_ptr, g.col, cap, g.s, g.t)
        certify_gpu(G, g, cap, f)
    assert levels > 0 or n * deg < 16_384   # (smaller ones may be searched by one CTA alone)
    G.close()
