"""PushRelabel visits at the sizes where a vertex changes its path: one arc
round per lane, several, the staged range, and the cooperative hub cycles; with
excess above 2^31 - 1, which one step cannot move whole."""
import numpy as np
import pytest

from workloads import generators as gen

pytestmark = pytest.mark.gpu


def _gadget(deg, big, seed):
    """s -> a_i -> u -> b_j -> t with deg arcs at u; the b_j also form a ring
    (excess that one cannot pass on goes round), and half of them have a narrow
    arc to t, so that flow returns through u."""
    rng = np.random.default_rng(seed)
    k = max(1, deg // 3)
    a, b = list(range(k)), list(range(k, deg + 1 if deg == 1 else deg))
    u, s, t = deg + 1, deg + 2, deg + 3
    hi = (1 << 28) if big else 50
    E = [(s, x, int(rng.integers(hi // 2, hi))) for x in a] + [(x, u, int(rng.integers(hi // 2, hi))) for x in a]
    E += [(u, y, int(rng.integers(1, hi))) for y in b]
    E += [(y, t, int(rng.integers(0, hi if j % 2 else 3))) for j, y in enumerate(b)]
    E += [(b[j], b[(j + 1) % len(b)], int(rng.integers(0, hi))) for j in range(len(b)) if len(b) > 1]
    E += [(x, t, 1) for x in a[:2]]
    return gen.from_edges(deg + 4, [e[0] for e in E], [e[1] for e in E], [e[2] for e in E], s, t)


@pytest.mark.parametrize("deg", [2, 31, 32, 33, 127, 128, 129, 300, 512, 513, 1100])
@pytest.mark.parametrize("big", [False, True])
def test_visit_sizes(deg, big):
    import oracle
    import paper_2511_05895_gb300 as mf
    for mode in (mf.MF_MODE_DATA_DRIVEN, mf.MF_MODE_TOPOLOGY, mf.MF_MODE_PUSH_PULL):
        g = _gadget(deg, big, 7 * deg + big)
        cap = g.cap.copy()
        G = mf.MaxFlowGraph(g.n, g.row_ptr, g.col, cap, g.s, g.t, mode=mode, debug_checks=True)
        G.solve()
        assert G.flow_value() == oracle.maxflow_fifo(g.n, g.row_ptr, g.col, cap, g.s, g.t)
        for i in range(3):
            bt = gen.mixed_batch(cap, max(2, g.m // 4), 1, (1 << 27) if big else 40, seed=deg, index=i)
            new = np.minimum(bt.new_cap, G.cap_limit()).astype(np.int32)
            G.apply_updates(bt.edge_id, new)
            cap[bt.edge_id] = new
            assert G.flow_value() == oracle.maxflow_fifo(g.n, g.row_ptr, g.col, cap, g.s, g.t)
        G.close()
