"""Which graphs the library renumbers by degree: those where the vertices of more
than 64 entries, s and t aside, hold a quarter of all entries -- among them the
power-law and star graphs of test_gpu_renumbered.  (Seen from outside by the index
of its arcs that a renumbered graph holds after an export to device buffers.)"""
import ctypes

import numpy as np
import pytest

from tests.test_gpu_renumbered import GRAPHS
from workloads import generators as gen

pytestmark = pytest.mark.gpu


def _terminals_only():
    """Every vertex has an arc from s and to t: only those two have long rows."""
    n = 3000
    v = np.arange(2, n)
    rng = np.random.default_rng(2)
    tails = np.concatenate([np.zeros(n - 2, np.int64), v, rng.integers(2, n, 4 * n)])
    heads = np.concatenate([v, np.ones(n - 2, np.int64), rng.integers(2, n, 4 * n)])
    return gen.from_edges(n, tails, heads, rng.integers(1, 50, tails.size), 0, 1)


@pytest.mark.parametrize("make,renumbered", [*zip(GRAPHS, [True, True, True, False]), (_terminals_only, False)])
def test_rule(make, renumbered):
    import torch

    import paper_2511_05895_gb300 as mf
    g = make()
    tails = np.repeat(np.arange(g.n), np.diff(g.row_ptr))
    keep = tails != g.col
    deg = np.bincount(tails[keep], minlength=g.n) + np.bincount(g.col[keep], minlength=g.n)
    big = (deg > 64) & ~np.isin(np.arange(g.n), (g.s, g.t))
    assert (4 * deg[big].sum() >= deg.sum()) == renumbered
    G = mf.MaxFlowGraph(g.n, g.row_ptr, g.col, g.cap, g.s, g.t)
    G.solve()
    L, before, after = mf.lib(), ctypes.c_int64(0), ctypes.c_int64(0)
    r = torch.zeros(G.sizes()[2], dtype=torch.int32, device="cuda")
    assert L.mf_device_bytes(G._h, ctypes.byref(before)) == mf.MF_OK
    assert L.mf_export_state(G._h, ctypes.c_void_p(r.data_ptr()), None, None, mf.MF_DEVICE_PTRS) == mf.MF_OK
    assert L.mf_device_bytes(G._h, ctypes.byref(after)) == mf.MF_OK
    assert (after.value > before.value) == renumbered
    G.close()
