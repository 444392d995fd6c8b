"""A failed debug check of a renumbered graph names the vertex or the arc by the
caller's numbers (an arc: its place in the exported arc arrays)."""
import re

import numpy as np
import pytest

from workloads import generators as gen

pytestmark = pytest.mark.gpu


def _fails(mf, G, g, seed):
    b = gen.mixed_batch(g.cap, 20, 1, 50, seed=seed, index=0)
    G.apply_updates(b.edge_id, b.new_cap)
    with pytest.raises(mf.MFError) as ei:
        G.flow_value()
    assert ei.value.code == mf.MF_ECHECK
    return str(ei.value), int(re.search(r"\(index (\d+)\)", str(ei.value)).group(1))


@pytest.mark.parametrize("seed", [3, 4, 5])
def test_arc_and_vertex_are_the_callers(seed):
    import paper_2511_05895_gb300 as mf
    g = gen.rmat(scale=10, seed=seed)
    G = mf.MaxFlowGraph(g.n, g.row_ptr, g.col, g.cap, g.s, g.t, debug_checks=True)
    G.solve()
    G.flow_value()
    b = mf.bicsr_host(g.n, g.row_ptr, g.col, g.cap, g.s, g.t)
    deg = np.diff(b["arc_row"])
    big = np.flatnonzero((deg > 64) & ~np.isin(np.arange(g.n), (g.s, g.t)))
    assert 4 * deg[big].sum() >= deg.sum()   # the rule by which the graph is renumbered
    r, e, h = G.export_state()
    tail = np.repeat(np.arange(g.n), deg)
    # one unit too many on a pair, the excess of its tail in step with it
    a = int(np.random.default_rng(seed).choice(np.flatnonzero(~np.isin(tail, (g.s, g.t)) & (b["head"] != g.s) & (b["head"] != g.t))))
    r2, e2 = r.copy(), e.copy()
    r2[a] += 1
    e2[tail[a]] += 1
    G.import_state(r2, e2, h)
    text, at = _fails(mf, G, g, seed)
    assert "residual pair" in text and at in (a, int(b["rev"][a]))
    # an excess of its own
    G.solve()
    G.flow_value()
    v = int(tail[a])
    r, e, h = G.export_state()
    e[v] += 1
    G.import_state(r, e, h)
    text, at = _fails(mf, G, g, seed + 10)
    assert "excess differs" in text and at == v
    G.close()
