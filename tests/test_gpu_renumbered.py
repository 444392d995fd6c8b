"""A power-law graph is renumbered by degree inside the library; everything
that crosses the C ABI stays in the caller's vertex ids and arc order."""
import ctypes

import numpy as np
import pytest

import oracle
from tests._helpers import certify_gpu
from workloads import generators as gen

pytestmark = pytest.mark.gpu


def _star(n, seed):
    """A few centres that most edges touch, s and t ordinary vertices."""
    rng = np.random.default_rng(seed)
    m = 6 * n
    u = np.where(rng.random(m) < 0.5, rng.integers(n - 4, n, m), rng.integers(0, n, m))
    v = np.where(rng.random(m) < 0.5, rng.integers(n - 4, n, m), rng.integers(0, n, m))
    return gen.from_edges(n, u, v, rng.integers(1, 100, m), 3, n // 2)


GRAPHS = [lambda: gen.rmat(scale=10, seed=5), lambda: gen.rmat(scale=13, edge_factor=9, seed=6),
          lambda: _star(4001, 7), lambda: gen.random_graph(n=3000, m=20_000, seed=8)]


@pytest.mark.parametrize("make", range(len(GRAPHS)))
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_ids_stay_the_callers(make, mode):
    import torch

    import paper_2511_05895_gb300 as mf
    g = GRAPHS[make]()
    cap = g.cap.copy()
    G = mf.MaxFlowGraph(g.n, g.row_ptr, g.col, cap, g.s, g.t, mode=mode)
    G.solve()
    b = gen.mixed_batch(cap, min(500, g.m // 8), 1, 50, seed=9, index=0)
    G.apply_updates(b.edge_id, b.new_cap)
    gen.apply_batch(cap, b)
    want = oracle.maxflow_fifo(g.n, g.row_ptr, g.col, cap, g.s, g.t)
    assert G.flow_value() == want
    certify_gpu(G, g, cap, want)
    host = mf.bicsr_host(g.n, g.row_ptr, g.col, cap, g.s, g.t)
    out = G.export_graph()
    for k in ("arc_row", "head", "rev", "cap"):
        np.testing.assert_array_equal(out[k], host[k])
    # device buffers hold the same as host buffers
    r, e, h = G.export_state()
    A = len(r)
    dr = torch.zeros(A, dtype=torch.int32, device="cuda")
    de = torch.zeros(g.n, dtype=torch.int64, device="cuda")
    dh = torch.zeros(g.n, dtype=torch.int32, device="cuda")
    side = torch.zeros(g.n, dtype=torch.uint8, device="cuda")
    L, P = mf.lib(), lambda x: ctypes.c_void_p(x.data_ptr())
    assert L.mf_export_state(G._h, P(dr), P(de), P(dh), mf.MF_DEVICE_PTRS) == mf.MF_OK
    assert L.mf_min_cut(G._h, P(side), mf.MF_DEVICE_PTRS) == mf.MF_OK
    np.testing.assert_array_equal(dr.cpu().numpy(), r)
    np.testing.assert_array_equal(de.cpu().numpy(), e)
    np.testing.assert_array_equal(dh.cpu().numpy(), h)
    np.testing.assert_array_equal(side.cpu().numpy(), G.min_cut())
    # a checkpoint resumes in another instance, from host and from device buffers
    for arrays, flags in (((r, e, h), 0), ((dr, de, dh), mf.MF_DEVICE_PTRS)):
        H = mf.MaxFlowGraph(g.n, g.row_ptr, g.col, cap, g.s, g.t, mode=mode)
        ptr = [P(x) if flags else ctypes.c_void_p(x.ctypes.data) for x in arrays]
        assert L.mf_import_state(H._h, *ptr, flags) == mf.MF_OK
        assert H.flow_value() == want
        nxt, cap2 = gen.mixed_batch(cap, 100, 1, 50, seed=10, index=1), cap.copy()
        H.apply_updates(nxt.edge_id, nxt.new_cap)
        gen.apply_batch(cap2, nxt)
        assert H.flow_value() == oracle.maxflow_fifo(g.n, g.row_ptr, g.col, cap2, g.s, g.t)
        H.apply_updates(nxt.edge_id[:0], nxt.new_cap[:0], recompute=True)
        assert H.flow_value() == oracle.maxflow_fifo(g.n, g.row_ptr, g.col, cap2, g.s, g.t)
        H.close()
    G.close()
