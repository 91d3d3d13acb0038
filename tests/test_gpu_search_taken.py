"""Which search a call ran on, where the results alone cannot tell."""
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


def test_batch_plan_tells_members_on_tiles(cc):
    gens = [synth.grid_edges(300, 20), synth.rmat_edges(10, 8, seed=2), synth.grid_edges(64, 64)]
    handles, samples = [], []
    try:
        for n, s, d in gens:
            g, _ = cc.cc_graph_from_edges(n, s, d)
            handles.append(g)
            samples.append(cc.cc_sample_choose(g, 40, 5))
        b = cc.cc_batch_create(handles, samples, autotune=False)
        try:
            plans = [cc.cc_batch_plan(b, i) for i in range(3)]
        finally:
            cc.cc_batch_free(b)
    finally:
        for g in handles:
            cc.cc_graph_free(g)
    for i in (0, 2):
        assert (plans[i]["alpha"], plans[i]["team"], plans[i]["class_teams"]) == (0, 0, 1)
    assert plans[1]["alpha"] > 0


@pytest.mark.parametrize("tail,launches", [(1, 2), (60, 6)])
def test_round_trips_on_planes_or_rows(cc, tail, launches):
    """300 sources: one traversal each way into planes; a graph too deep for
    them takes three chunks each way."""
    rng = np.random.default_rng(tail)
    head = 600
    ring, t = np.arange(head), np.arange(head - 1, head + tail - 1)
    s = np.concatenate([ring, rng.integers(0, head, 6 * head), t, t + 1])
    d = np.concatenate([(ring + 1) % head, rng.integers(0, head, 6 * head), t + 1, t])
    g, _ = cc.cc_graph_from_edges(head + tail, s.astype(np.uint32), d.astype(np.uint32),
                                  directed=True)
    try:
        C = cc.cc_sample_choose(g, 300, 4)
        o = cc.cc_opts_default(300)
        o.roundtrip = 1
        for _ in range(2):
            cc.cc_estimate(g, C, o)
        assert cc.cc_last_call_timing(g)[0] == launches
    finally:
        cc.cc_graph_free(g)


def same(a, b):
    for key in a:
        assert np.array_equal(a[key], b[key]), key


def test_interleaved_tiles_serve_the_adaptive_hybrid_only(cc):
    """A random geometric graph of mean degree 4, whose tiles' borders are more
    than two sides long: one pass of 256 sources runs level by level, the
    adaptive hybrid, eight passes otherwise, on tiles."""
    n, s, d = synth.road_like_edges(8000, mean_degree=4.0, gen_degree=8.0, seed=4)[:3]
    g, _ = cc.cc_graph_from_edges(n, s, d)
    og = orc.csr_from_edges(n, s, d)
    try:
        C = cc.cc_sample_choose(g, 256, 3)
        deepest = int(orc.dist_table(og, C).max())
        r = cc.cc_estimate(g, C)
        assert cc.cc_last_pass_stats(g)["levels"] == deepest
        ad = cc.cc_estimate_adaptive(g, C)
        assert cc.cc_last_pass_stats(g)["levels"] < deepest
        same(r, cc.cc_estimate(g, C))
        assert cc.cc_last_pass_stats(g)["levels"] == deepest
        cc.cc_set_tuning(g, 4)
        same(r, cc.cc_estimate(g, C))
        same(ad, cc.cc_estimate_adaptive(g, C))
    finally:
        cc.cc_graph_free(g)


def test_interleaved_tiles_with_lengths(cc):
    """The same graph with arc lengths: 64 sources by the shortest-path rounds,
    250, of which those take four chunks, by tiles; the results are equal."""
    n, s, d, ln = synth.road_like_edges(8000, mean_degree=4.0, gen_degree=8.0, seed=4)
    g, _ = cc.cc_graph_from_edges(n, s, d, synth.edge_lengths_to_weights(ln))
    try:
        for k, rounds in ((64, True), (250, False), (64, True)):
            C = cc.cc_sample_choose(g, k, 3)
            o = cc.cc_opts_default(k)
            cc.cc_set_param(g, cc.CC_PARAM_SSSP_DELTA, 0)
            r = cc.cc_estimate(g, C, o)
            launches = cc.cc_last_call_timing(g)[0]
            levels = cc.cc_last_pass_stats(g)["levels"]
            cc.cc_set_param(g, cc.CC_PARAM_SSSP_DELTA, 4000)
            same(r, cc.cc_estimate(g, C, o))
            assert cc.cc_last_call_timing(g)[0] == (k + 63) // 64
            assert launches == 1
            if not rounds:  # a tile is crossed in a round, a bucket holds a few hops
                assert levels < cc.cc_last_pass_stats(g)["levels"]
            else:
                assert levels > 100
    finally:
        cc.cc_graph_free(g)


def test_shortcuts_leave_tiles_to_narrow_samples(cc):
    """A ring with 1 % of its edges rewired is 130 hops across 85 tiles of ten
    neighbours: 64 sources run on tiles, 2048 level by level."""
    n, s, d = synth.watts_strogatz_edges(20000, 4, 0.01, seed=2)
    g, _ = cc.cc_graph_from_edges(n, s, d)
    try:
        for k, tiles in ((64, True), (2048, False)):
            C = cc.cc_sample_choose(g, k, 3)
            cc.cc_set_tuning(g, 0)
            r = cc.cc_estimate(g, C)
            levels = cc.cc_last_pass_stats(g)["levels"]
            cc.cc_set_tuning(g, 14)
            same(r, cc.cc_estimate(g, C))
            other = cc.cc_last_pass_stats(g)["levels"]
            assert levels < other if tiles else levels == other
    finally:
        cc.cc_graph_free(g)
