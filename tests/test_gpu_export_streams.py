"""Exports of a renumbered graph's state into device buffers: the first export
of a graph that lives on a stream of its own (torch's are non-blocking: they do
not wait for the legacy stream), with and without device memory for the index
that puts the arcs into the caller's order."""
import ctypes

import numpy as np
import pytest

from workloads import generators as gen

pytestmark = pytest.mark.gpu


def _to_device(mf, L, h, n, A, stream):
    import torch
    with torch.cuda.stream(stream):
        r = torch.full((A,), -1, dtype=torch.int32, device="cuda")
        e = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        d = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    stream.synchronize()
    P = lambda x: ctypes.c_void_p(x.data_ptr())
    assert L.mf_export_state(h, P(r), P(e), P(d), mf.MF_DEVICE_PTRS) == mf.MF_OK
    with torch.cuda.stream(stream):
        return [x.cpu().numpy() for x in (r, e, d)]


@pytest.mark.parametrize("refuse", [False, True])
def test_first_export_is_to_device_buffers(refuse):
    import torch

    import paper_2511_05895_gb300 as mf
    from paper_2511_05895_gb300 import _native as nat
    g = gen.rmat(scale=15, seed=91)
    L = mf.lib()
    off = {"refuse": False}
    dev = torch.cuda.current_device()
    alloc = nat.ALLOC_FN(lambda b, c: None if off["refuse"] else torch.cuda.caching_allocator_alloc(int(b), dev))
    free = nat.FREE_FN(lambda p, c: torch.cuda.caching_allocator_delete(int(p)))
    stream = torch.cuda.Stream()
    st = ctypes.c_void_p(stream.cuda_stream)
    host = []
    for _ in range(3):   # a fresh graph each time: its first export
        opt = nat.Options()
        L.mf_options_default(ctypes.byref(opt))
        opt.alloc, opt.free = alloc, free
        h = ctypes.c_void_p()
        arrays = [np.ascontiguousarray(x) for x in (g.row_ptr.astype(np.int64), g.col.astype(np.int32),
                                                    g.cap.astype(np.int32))]
        assert L.mf_create(g.n, len(arrays[1]), *[ctypes.c_void_p(x.ctypes.data) for x in arrays], g.s, g.t,
                           ctypes.byref(opt), st, ctypes.byref(h)) == mf.MF_OK
        try:
            A = ctypes.c_int64(0)
            assert L.mf_sizes(h, None, None, ctypes.byref(A)) == mf.MF_OK
            off["refuse"] = refuse
            assert L.mf_solve(h, st) == mf.MF_OK
            got = _to_device(mf, L, h, g.n, A.value, stream)
            host = [np.zeros(A.value, np.int32), np.zeros(g.n, np.int64), np.zeros(g.n, np.int32)]
            assert L.mf_export_state(h, *[ctypes.c_void_p(x.ctypes.data) for x in host], mf.MF_HOST_PTRS) == mf.MF_OK
            for a, b in zip(got, host):
                np.testing.assert_array_equal(a, b)
            for a, b in zip(_to_device(mf, L, h, g.n, A.value, stream), host):   # and a later one
                np.testing.assert_array_equal(a, b)
        finally:
            off["refuse"] = False
            L.mf_destroy(h)
    # the order is the caller's: the residual of every arc and its reverse add up to the capacities of the pair
    b = mf.bicsr_host(g.n, g.row_ptr, g.col, g.cap, g.s, g.t)
    r = host[0].astype(np.int64)
    np.testing.assert_array_equal(r + r[b["rev"]], b["cap"].astype(np.int64) + b["cap"][b["rev"]])
