"""Parity with the oracle where the traversal's rules change course: sample
widths of sixteen and thirty-two words (histogram by transposes and bit by
bit), graphs with fewer nodes than warps (a warp per light node) and just more
than a level's lists may hold before they are rebuilt, and hubs that complete
while other nodes go on.  Integers bit-exact; FP64 within 1e-12 relative (one
conversion and one division of the same integers on both sides)."""
import numpy as np
import pytest

import synth
from oracle import oracle as orc

pytestmark = pytest.mark.gpu
RTOL = 1e-12


@pytest.fixture(scope="module")
def cc():
    from paper_1409_0035_gb300 import build
    build.build()
    import paper_1409_0035_gb300 as m
    return m


def hubs_and_tail(n_leaf, tail):
    # two hubs sharing n_leaf leaves, a path hanging off one leaf
    leaf = np.arange(2, 2 + n_leaf)
    path = np.arange(2 + n_leaf, 2 + n_leaf + tail)
    s = np.concatenate([np.zeros(n_leaf), np.ones(n_leaf), [2], path[:-1]])
    d = np.concatenate([leaf, leaf, [path[0]], path[1:]])
    return 2 + n_leaf + tail, s.astype(np.uint32), d.astype(np.uint32)


CASES = {
    "rmat12-k700": (lambda: synth.rmat_edges(12, 8, seed=5), 700),
    "rmat12-k1024": (lambda: synth.rmat_edges(12, 8, seed=5), 1024),
    "rmat13-k2000": (lambda: synth.rmat_edges(13, 6, seed=6), 2000),
    "grid-k1100": (lambda: synth.grid_edges(60, 51), 1100),
    "ws45000-k300": (lambda: synth.watts_strogatz_edges(45000, 10, 0.05, seed=4), 300),
    "ws4850-k64": (lambda: synth.watts_strogatz_edges(4850, 8, 0.1, seed=2), 64),
    "hubs-k33": (lambda: hubs_and_tail(3000, 40), 33),
    "hubs-k130": (lambda: hubs_and_tail(700, 9), 130),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_estimate_at_the_edges(cc, name):
    make, k = CASES[name]
    n, s, d = make()
    g, _ = cc.cc_graph_from_edges(n, s, d)
    try:
        og = orc.csr_from_edges(n, s, d)
        C = cc.cc_sample_choose(g, k, 3)
        o = cc.cc_opts_default(k)
        for _ in range(3):  # direct, captured, replayed
            r = cc.cc_estimate(g, C, o)
    finally:
        cc.cc_graph_free(g)
    want = orc.estimate(og, C, eps=(o.eps_num, o.eps_den))
    for key in ("pivot", "delta", "sum", "S_samp", "delta_cc", "hyb"):
        assert np.array_equal(r[key], want[key]), key
    for key in ("s_hat", "closeness"):
        rel = np.abs(r[key] - want[key]) / np.abs(want[key])
        assert rel.max() <= RTOL, key


def ladder(n):
    # rungs every third step, every twentieth node with a few extra leaves:
    # rows of 2 to 7 entries around the four that are kept inline by node
    a = np.arange(n - 1)
    rung = np.arange(0, n, 3)
    hub = np.repeat(np.arange(0, n, 20), 4)
    leaf = 2 * n + np.arange(hub.size)
    s = np.concatenate([a, n + a, rung, hub])
    d = np.concatenate([a + 1, n + a + 1, n + rung, leaf])
    return 2 * n + hub.size, s.astype(np.uint32), d.astype(np.uint32)


@pytest.mark.parametrize("k", [1, 64, 65, 200, 500, 1000, 1500])
@pytest.mark.parametrize("name", ["ladder", "grid"])
def test_narrow_frontiers_at_every_width(cc, name, k):
    """Top-down levels of few bits per word at 1 to 32 words per node, rows on
    both sides of the inline limit."""
    n, s, d = ladder(900) if name == "ladder" else synth.grid_edges(59, 41)
    g, _ = cc.cc_graph_from_edges(n, s, d)
    try:
        og = orc.csr_from_edges(n, s, d)
        C = cc.cc_sample_choose(g, k, 9)
        o = cc.cc_opts_default(k)
        cc.cc_set_tuning(g, 1)  # top-down for as long as a frontier allows it
        r = cc.cc_estimate(g, C, o)
        stats = cc.cc_last_pass_stats(g)
    finally:
        cc.cc_graph_free(g)
    assert stats["td_levels"] > 0
    want = orc.estimate(og, C, eps=(o.eps_num, o.eps_den))
    for key in ("pivot", "delta", "sum", "S_samp", "delta_cc", "hyb"):
        assert np.array_equal(r[key], want[key]), key
