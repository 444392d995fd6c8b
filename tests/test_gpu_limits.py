"""Solves and repairs that end on max_iters or on the wall-clock limit: every
CTA leaves the loop on the same decision, so the call ends at once with that
limit's message (a CTA that missed it would wait for the others until the
barrier's own limit of 20 s)."""
import time

import pytest

import oracle
from workloads import generators as gen

pytestmark = pytest.mark.gpu


def _ends(mf, G, what):
    t0 = time.perf_counter()
    with pytest.raises(mf.MFError) as ei:
        G.flow_value()
    assert ei.value.code == mf.MF_ETIMEOUT and what in str(ei.value)
    assert time.perf_counter() - t0 < 5.0


@pytest.mark.parametrize("mode", [0, 1, 2])
def test_iteration_limit(mode):
    import paper_2511_05895_gb300 as mf
    g = gen.grid_segmentation(300, 300, seed=81)
    G = mf.MaxFlowGraph(g.n, g.row_ptr, g.col, g.cap, g.s, g.t, mode=mode, max_iters=1, kernel_cycles=1)
    for _ in range(100):
        G.solve()
        _ends(mf, G, "max_iters")
    G.close()


@pytest.mark.parametrize("mode", [0, 2])
def test_wall_clock_limit(mode):
    import paper_2511_05895_gb300 as mf
    g = gen.grid_segmentation(1024, 1024, seed=82)
    want = oracle.maxflow_fifo(g.n, g.row_ptr, g.col, g.cap, g.s, g.t)
    G = mf.MaxFlowGraph(g.n, g.row_ptr, g.col, g.cap, g.s, g.t, mode=mode)
    for _ in range(20):
        G.set_time_limit(1)
        G.solve()
        _ends(mf, G, "wall-clock")
    G.set_time_limit(0)
    G.solve()
    assert G.flow_value() == want
    G.set_time_limit(1)
    G.apply_updates([], [], recompute=True)   # the recompute of a graph whose flow stands
    _ends(mf, G, "wall-clock")
    G.set_time_limit(0)
    G.solve()
    assert G.flow_value() == want
    G.close()
