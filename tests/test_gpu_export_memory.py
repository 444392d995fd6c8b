"""What exports of a renumbered graph hold on the device: nothing for host
buffers, one index of its arcs from the first export to device buffers on."""
import ctypes

import pytest

from workloads import generators as gen

pytestmark = pytest.mark.gpu


def test_host_exports_hold_nothing():
    import torch

    import paper_2511_05895_gb300 as mf
    L = mf.lib()

    def held(G):
        b = ctypes.c_int64(0)
        assert L.mf_device_bytes(G._h, ctypes.byref(b)) == mf.MF_OK
        return b.value

    g = gen.rmat(scale=12, seed=31)
    G = mf.MaxFlowGraph(g.n, g.row_ptr, g.col, g.cap, g.s, g.t)
    G.solve()
    start = held(G)
    G.export_graph()
    G.import_state(*G.export_state())
    G.min_cut()
    assert held(G) == start
    A = G.sizes()[2]
    r = torch.zeros(A, dtype=torch.int32, device="cuda")
    for _ in range(2):
        assert L.mf_export_state(G._h, ctypes.c_void_p(r.data_ptr()), None, None, mf.MF_DEVICE_PTRS) == mf.MF_OK
        assert held(G) == start + 4 * A
    G.close()
