"""What the bit planes leave on a handle: the captured estimate follows the
parameter that chooses them."""
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


def test_captured_estimate_follows_the_parameter(cc):
    n, s, d = synth.rmat_edges(12, 8, seed=9)
    g, _ = cc.cc_graph_from_edges(n, s, d)
    try:
        C = cc.cc_sample_choose(g, 100, 2)
        o = cc.cc_opts_default(100)
        o.eps_num, o.eps_den = 2, 3
        seen = []
        for one_pass in (1, 0, 1, 0):
            cc.cc_set_param(g, cc.CC_PARAM_HYBRID_ONE_PASS, one_pass)
            for call in range(4):
                r = cc.cc_estimate(g, C, o, want_sqerr=True)
                if call == 0:
                    first = r
                    assert not cc.cc_last_call_graph(g)
            assert cc.cc_last_call_graph(g)
            for key in r:
                assert np.array_equal(r[key], first[key]), key
            seen.append((cc.cc_last_call_timing(g)[3], r))
        assert seen[0][0] == seen[2][0] != seen[1][0] == seen[3][0]  # kernels of each form
        for _, r in seen[1:]:
            for key in r:
                assert np.array_equal(r[key], seen[0][1][key]), key
    finally:
        cc.cc_graph_free(g)
