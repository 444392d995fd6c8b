"""Batches that meet s and t in every entry: clamped and raised terminal arcs,
both kinds in one warp and in every CTA, against the oracle, with the excess of
every vertex accounted for by the certificate."""
import numpy as np
import pytest

import oracle
from tests._helpers import certify_gpu
from workloads import generators as gen

pytestmark = pytest.mark.gpu


def _star(mid, seed):
    """s -> every middle vertex -> t, a ring through the middle and one arc s -> t."""
    rng = np.random.default_rng(seed)
    v = np.arange(mid)
    s, t = mid, mid + 1
    tails = np.concatenate([np.full(mid, s), v, v, [s]])
    heads = np.concatenate([v, np.full(mid, t), (v + 1) % mid, [t]])
    return gen.from_edges(mid + 2, tails, heads, rng.integers(1, 1000, tails.size), s, t)


@pytest.mark.parametrize("mid", [3, 33, 1000, 40_000])
@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("top", [0, 1000, 1 << 20])
def test_terminal_entries(mid, mode, top):
    import paper_2511_05895_gb300 as mf
    g = _star(mid, mid)
    cap = g.cap.copy()
    rng = np.random.default_rng(top + mode)
    G = mf.MaxFlowGraph(g.n, g.row_ptr, g.col, cap, g.s, g.t, mode=mode)
    G.solve()
    for _ in range(3):
        ids = rng.permutation(g.m)[: max(1, g.m * 2 // 3)].astype(np.int32)
        new = rng.integers(0, top + 1, ids.size).astype(np.int32)
        G.apply_updates(ids, new)
        cap[ids] = new
        f = G.flow_value()
        assert f == oracle.maxflow_fifo(g.n, g.row_ptr, g.col, cap, g.s, g.t)
        certify_gpu(G, g, cap, f)
    G.close()
