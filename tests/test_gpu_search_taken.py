"""Which search a call ran on, where the results alone cannot tell."""
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
