"""The learned policy on a stream of its own (non-blocking: it does not wait for
the legacy stream): the batch after set_policy is decided by the new network."""
import numpy as np
import pytest

import oracle
from oracle import mlp as omlp
from workloads import generators as gen

pytestmark = pytest.mark.gpu


def test_parameters_are_in_place_for_the_next_batch():
    import torch

    import paper_2511_05895_gb300 as mf
    g = gen.rmat(scale=12, seed=95)
    cap = g.cap.copy()
    with torch.cuda.stream(torch.cuda.Stream()):
        G = mf.MaxFlowGraph(g.n, g.row_ptr, g.col, cap, g.s, g.t)
        G.solve()
        P = np.zeros(omlp.N_TOTAL, np.float32)
        P[omlp.O_SD:] = 1e6
        for j, (repair, log2kc) in enumerate([(4.0, 3.0), (4.0, 0.0), (-4.0, 2.0), (4.0, 1.0), (-4.0, 4.0), (4.0, 4.0)]):
            P[omlp.O_B3:omlp.N_TRAINED] = [repair, log2kc, 1.0, 0.0, 0.0]
            G.set_policy(mf.MF_POLICY_LEARNED, P)
            b = gen.mixed_batch(cap, 100, 1, 500, seed=95, index=j)
            G.apply_updates(b.edge_id, b.new_cap)
            gen.apply_batch(cap, b)
            assert G.flow_value() == oracle.maxflow_fifo(g.n, g.row_ptr, g.col, cap, g.s, g.t)
            s = G.stats()
            assert (s["policy_kind"], s["policy_kernel_cycles"], s["policy_fallback"]) == (int(repair < 0), 2 ** log2kc, 0)
        G.close()
