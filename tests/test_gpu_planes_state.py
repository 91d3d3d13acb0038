"""What the bit planes leave on a handle: the captured estimate follows the
parameter that chooses them, graphs too deep for them do not keep their
memory, a server admits requests with them in the account."""
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


def comet(head, tail, directed):
    """A dense head with a tail of `tail` nodes; directed: arcs both ways in
    the tail, a cycle with chords in the head."""
    rng = np.random.default_rng(head + tail)
    ring = np.arange(head)
    s = np.concatenate([ring, rng.integers(0, head, 6 * head), np.arange(head - 1, head + tail - 1)])
    d = np.concatenate([(ring + 1) % head, rng.integers(0, head, 6 * head),
                        np.arange(head, head + tail)])
    if directed:
        t = np.arange(head - 1, head + tail - 1)
        s, d = np.concatenate([s, t + 1]), np.concatenate([d, t])
    return head + tail, s.astype(np.uint32), d.astype(np.uint32)


@pytest.mark.parametrize("directed", [False, True])
def test_planes_of_deep_graphs_are_given_back(cc, directed):
    """The planes of 1000 sources take 512 bytes a node and direction.  A graph
    of 60 levels cannot use them: its handle holds less than a shallow one's
    by more than half of that, other buffers (about 290 and, round trip, the
    distance rows) set aside."""
    import torch
    k, head = 1000, 150_000
    held = []
    for tail in (1, 60):
        n, s, d = comet(head, tail, directed)
        g, _ = cc.cc_graph_from_edges(n, s, d, directed=directed)
        try:
            C = cc.cc_sample_choose(g, k, 4)
            o = cc.cc_opts_default(k)
            o.roundtrip = int(directed)
            torch.cuda.synchronize()
            before = torch.cuda.mem_get_info()[0]
            ad = [cc.cc_estimate_adaptive(g, C, o) for _ in range(2)]
            torch.cuda.synchronize()
            held.append(before - torch.cuda.mem_get_info()[0])
            for key in ad[0]:
                assert np.array_equal(ad[0][key], ad[1][key]), key
        finally:
            cc.cc_graph_free(g)
    if directed:
        held[1] -= 2 * head * 1024 * 4  # the rows of all sources, both ways
    assert held[1] < held[0], held


def test_server_counts_the_planes(cc):
    """Two round-trip requests whose workspaces do not fit the budget together
    do not run together."""
    n, s, d = synth.watts_strogatz_edges(400_000, 10, 0.5, seed=6)
    s, d = np.concatenate([s, d]), np.concatenate([d, s])
    k = 1024
    g, _ = cc.cc_graph_from_edges(n, s, d, directed=True)
    try:
        srv = cc.cc_server_create([g], slots=2)
        try:
            rid = cc.cc_server_submit(srv, 0, 0, k, 1)
            assert cc.cc_server_wait(srv, rid, 60000) == cc.CC_OK
            one = cc.cc_server_cache_stats(srv)["resident_bytes"]
        finally:
            cc.cc_server_free(srv)
        srv = cc.cc_server_create([g], slots=2, hbm_budget=int(1.7 * one))
        try:
            ids = [cc.cc_server_submit(srv, 0, 0, k, 10 + i) for i in range(6)]
            for rid in ids:
                assert cc.cc_server_wait(srv, rid, 60000) == cc.CC_OK
            assert cc.cc_server_stats(srv)["peak_running"] == 1
            assert cc.cc_server_cache_stats(srv)["resident_bytes"] <= int(1.7 * one)
        finally:
            cc.cc_server_free(srv)
    finally:
        cc.cc_graph_free(g)
