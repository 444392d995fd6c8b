"""Visits that relabel their vertex without moving anything and put it back in
the activation queue: with one step per visit (kernel_cycles=1) that is every
relabel.  Short rows, staged rows (more than 128 arcs) and both directions."""
import numpy as np
import pytest

import oracle
from tests._helpers import certify_gpu
from workloads import generators as gen

pytestmark = pytest.mark.gpu


def _wide(left, right, deg, seed):
    """s -> left -> right -> t with `deg` arcs at every left vertex."""
    rng = np.random.default_rng(seed)
    s, t = left + right, left + right + 1
    u = np.repeat(np.arange(left), deg)
    v = left + np.concatenate([rng.permutation(right)[:deg] for _ in range(left)])
    tails = np.concatenate([np.full(left, s), u, left + np.arange(right)])
    heads = np.concatenate([np.arange(left), v, np.full(right, t)])
    caps = np.concatenate([rng.integers(1, 400, left), rng.integers(1, 20, u.size), rng.integers(0, 60, right)])
    return gen.from_edges(t + 1, tails, heads, caps, s, t)


GRAPHS = [lambda: gen.random_graph(n=2000, m=9000, seed=71), lambda: gen.grid_segmentation(120, 90, seed=72),
          lambda: _wide(300, 700, 200, 73)]


@pytest.mark.parametrize("make", range(len(GRAPHS)))
@pytest.mark.parametrize("mode", [0, 2])
def test_relabels_alone(make, mode):
    import paper_2511_05895_gb300 as mf
    g = GRAPHS[make]()
    cap = g.cap.copy()
    G = mf.MaxFlowGraph(g.n, g.row_ptr, g.col, cap, g.s, g.t, mode=mode, kernel_cycles=1, debug_checks=True)
    G.solve()
    for i in range(4):
        f = G.flow_value()
        assert f == oracle.maxflow_fifo(g.n, g.row_ptr, g.col, cap, g.s, g.t)
        certify_gpu(G, g, cap, f)
        b = gen.mixed_batch(cap, g.m // 8, 1, 60, seed=74, index=i)
        G.apply_updates(b.edge_id, b.new_cap)
        gen.apply_batch(cap, b)
    G.close()
