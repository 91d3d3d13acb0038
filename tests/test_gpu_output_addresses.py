"""Outputs asked for as host memory at addresses of every kind, on the first
calls of a handle and on the later ones, which stage small outputs: pageable
and pinned memory, and device memory, which the copies take as well."""
import ctypes

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cc():
    from paper_1409_0035_gb300 import build
    build.build()
    import paper_1409_0035_gb300 as m
    return m


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("kind", ["pageable", "pinned", "device"])
def test_host_outputs_at_any_address(cc, kind, mixed):
    import torch
    n, s, d = synth.rmat_edges(8, 8, seed=1)
    g, _ = cc.cc_graph_from_edges(n, s, d)
    try:
        n = cc.cc_graph_info(g)[0]
        C = cc.cc_sample_choose(g, 8, 1)
        o = cc.cc_opts_default(8)
        want = cc.cc_estimate(g, C, o)
        total = torch.zeros(n, dtype=torch.int64)
        total = {"pageable": total, "pinned": total.pin_memory, "device": total.cuda}[kind]
        total = total if kind == "pageable" else total()
        pivot = np.zeros(n, np.int32)
        out = cc.cc_out()
        out.sample_sum = total.data_ptr()
        if mixed:
            out.pivot = pivot.ctypes.data
        for _ in range(5):
            total.zero_()
            pivot[:] = -1
            torch.cuda.synchronize()
            assert cc.lib().cc_estimate(g, C.ctypes.data_as(ctypes.c_void_p), 8, ctypes.byref(o),
                                        ctypes.byref(out)) == cc.CC_OK
            assert np.array_equal(total.cpu().numpy().astype(np.uint64), want["sum"])
            if mixed:
                assert np.array_equal(pivot, want["pivot"])
    finally:
        cc.cc_graph_free(g)
