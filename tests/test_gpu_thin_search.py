"""BFS levels of small frontiers (run by one CTA): deep thin graphs, frontiers
around the sizes at which the search goes back to the whole grid, vertices of
many arcs among thin ones, and active vertices found along the way."""
import numpy as np
import pytest

import oracle
from tests._helpers import certify_gpu
from workloads import generators as gen

pytestmark = pytest.mark.gpu


def _layers(widths, cap_hi, seed, fan=2):
    """s -> layer 0 -> layer 1 -> ... -> t, every vertex with `fan` arcs into the next layer."""
    rng = np.random.default_rng(seed)
    start = np.concatenate([[0], np.cumsum(widths)])
    s, t = int(start[-1]), int(start[-1]) + 1
    tails, heads = [np.full(widths[0], s)], [np.arange(widths[0])]
    for i in range(len(widths) - 1):
        u = np.repeat(np.arange(start[i], start[i + 1]), fan)
        tails.append(u)
        heads.append(rng.integers(start[i + 1], start[i + 2], u.size))
    tails.append(np.arange(start[-2], start[-1]))
    heads.append(np.full(widths[-1], t))
    tails, heads = np.concatenate(tails), np.concatenate(heads)
    return gen.from_edges(t + 1, tails, heads, rng.integers(1, cap_hi, tails.size), s, t)


WIDTHS = {"path": [1] * 300, "thin": [7] * 120, "edge": [100, 4095, 4096, 4097, 100, 5], "wide": [3, 9000, 3, 9000, 3],
          "mixed": [1, 64, 65, 1, 130, 1, 2000, 1, 1, 600] * 3}


@pytest.mark.parametrize("name", sorted(WIDTHS))
@pytest.mark.parametrize("mode", [0, 2])
def test_thin_search(name, mode):
    import paper_2511_05895_gb300 as mf
    g = _layers(WIDTHS[name], 50, len(name))
    cap = g.cap.copy()
    G = mf.MaxFlowGraph(g.n, g.row_ptr, g.col, cap, g.s, g.t, mode=mode, debug_checks=True)
    G.solve()
    f = G.flow_value()
    assert f == oracle.maxflow_fifo(g.n, g.row_ptr, g.col, cap, g.s, g.t)
    certify_gpu(G, g, cap, f)
    for i in range(3):
        b = gen.mixed_batch(cap, max(1, g.m // 10), 1, 40, seed=3, index=i)
        G.apply_updates(b.edge_id, b.new_cap)
        gen.apply_batch(cap, b)
        f = G.flow_value()
        assert f == oracle.maxflow_fifo(g.n, g.row_ptr, g.col, cap, g.s, g.t)
        certify_gpu(G, g, cap, f)
    G.close()
