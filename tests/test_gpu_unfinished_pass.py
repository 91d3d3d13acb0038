"""First passes that end before every node is reached -- a graph in parts, more
levels than the histogram first holds -- on memory that earlier graphs have
written: the kernels behind the pass read no index it has not set.  Integers
bit-exact."""
import numpy as np
import pytest

import synth
from oracle import oracle as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cc():
    from paper_1409_0035_gb300 import build
    build.build()
    import paper_1409_0035_gb300 as m
    return m


def used_memory(cc):
    """Buffers of the sizes a small handle takes, written and given back."""
    import torch
    t = [torch.full((size,), 0x7B7B7B7B, dtype=torch.int32, device="cuda")
         for size in (1 << 14, 1 << 16, 1 << 18, 1 << 20) for _ in range(16)]
    torch.cuda.synchronize()
    del t
    torch.cuda.empty_cache()
    for n, s, d in (synth.rmat_edges(12, 8, seed=3), synth.grid_edges(80, 60)):
        g, _ = cc.cc_graph_from_edges(n, s, d)
        cc.cc_estimate(g, cc.cc_sample_choose(g, 300, 1))
        cc.cc_graph_free(g)


@pytest.mark.parametrize("k", [1, 70])
@pytest.mark.parametrize("hybrid", [0, 1])
def test_more_levels_than_the_first_histogram(cc, k, hybrid):
    n, s, d = synth.path_edges(5000)
    used_memory(cc)
    g, _ = cc.cc_graph_from_edges(n, s, d)
    try:
        cc.cc_set_tuning(g, 14)  # the level-synchronous search
        C = cc.cc_sample_choose(g, k, 3)
        o = cc.cc_opts_default(k)
        o.want_hybrid = hybrid
        r = cc.cc_estimate(g, C, o)
    finally:
        cc.cc_graph_free(g)
    want = orc.estimate(orc.csr_from_edges(n, s, d), C, eps=(o.eps_num, o.eps_den))
    for key in ("sum", "pivot", "delta", "S_samp") + (("hyb",) if hybrid else ()):
        assert np.array_equal(r[key], want[key]), key


@pytest.mark.parametrize("k", [1, 70])
@pytest.mark.parametrize("call", ["plain", "hybrid", "sqerr", "adaptive"])
def test_graph_in_parts(cc, k, call):
    n, s, d = synth.rmat_edges(9, 8, seed=5)
    m, t, u = synth.cycle_edges(900)
    s, d = np.concatenate([s, t + n]), np.concatenate([d, u + n])
    used_memory(cc)
    g, _ = cc.cc_graph_from_edges(n + m, s.astype(np.uint32), d.astype(np.uint32),
                                  keep_component=False)
    try:
        C = cc.cc_sample_choose(g, k, 3)
        o = cc.cc_opts_default(k)
        o.want_hybrid = int(call != "plain")
        for _ in range(3):
            with pytest.raises(cc.CCError) as e:
                if call == "adaptive":
                    cc.cc_estimate_adaptive(g, C)
                else:
                    cc.cc_estimate(g, C, o, want_sqerr=call == "sqerr")
            assert e.value.code == cc.CC_ERR_DISCONNECTED
    finally:
        cc.cc_graph_free(g)
