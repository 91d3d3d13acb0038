"""Graphs cut into tiles where the tiles cannot serve: more distances than
another search's histogram limit, memory too short to cut or to search them.  What the
level-synchronous search answered before stays answered."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
RTOL = 1e-12  # one conversion and one division of the same integers


@pytest.fixture(scope="module")
def cc():
    from paper_1409_0035_gb300 import build
    build.build()
    import paper_1409_0035_gb300 as m
    return m


def path_hybrid(n, C, v, eps):
    """Hybrid of node v of a path, C the sampled positions, from the
    definitions: (Hsum, Hnum, HCsum, LCsum, LCnum, estimate)."""
    d = np.abs(C.astype(np.int64) - v)
    i = int(d.argmin())
    p, t = int(C[i]), int(d[i]) * eps[1] // eps[0]
    num = tot = 0
    for side in (p, n - 1 - p):  # nodes beyond t on each side
        if side > t:
            num += side - t
            tot += (side * (side + 1) - t * (t + 1)) // 2
    dc = np.abs(C.astype(np.int64) - p)
    far = dc > t
    num -= int(far.sum())
    tot -= int(dc[far].sum())
    hc, lc, L = int(d[far].sum()), int(d[~far].sum()), int((~far).sum())
    est = ((tot + hc) * L + lc * (n - 1 - num - int(far.sum()))) / L
    return (tot, num, hc, lc, L), est


def test_more_distances_than_a_row_histogram(cc):
    """(D + 1) k counters of four bytes, over 4 GiB: a path of 1.1 million
    nodes and 1024 sources."""
    n, s, d = synth.path_edges(1_100_000)
    k = 1024
    g, _ = cc.cc_graph_from_edges(n, s, d)
    try:
        C = cc.cc_sample_choose(g, k, 2)
        o = cc.cc_opts_default(k)
        r = cc.cc_estimate(g, C, o)
        assert (int(r["delta_cc"].max()) + 1) * k * 4 > 4 << 30
        eps = [(1, 2), (1, 40)]
        ad = cc.cc_estimate_adaptive(g, C, o, eps)
    finally:
        cc.cc_graph_free(g)
    rng = np.random.default_rng(3)
    inC = np.zeros(n, bool)
    inC[C] = True
    for v in np.concatenate([[0, n - 1], rng.integers(0, n, 60)]):
        if inC[v]:
            continue
        dv = np.abs(C.astype(np.int64) - v)
        assert r["sum"][v] == dv.sum() and r["delta"][v] == dv.min() and r["pivot"][v] == dv.argmin()
        ints, est = path_hybrid(n, C, int(v), (o.eps_num, o.eps_den))
        assert tuple(int(x) for x in r["hyb"][v][:5]) == ints
        assert abs(r["s_hat"][3][v] - est) <= RTOL * est
        est = path_hybrid(n, C, int(v), eps[ad["choice"][v]])[1]
        assert abs(ad["s_hat"][v] - est) <= RTOL * est


class Short:
    """All device memory but `left` bytes taken, while it lives."""

    def __init__(self, left):
        import torch
        torch.cuda.empty_cache()
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        self.t = torch.empty(free - left, dtype=torch.uint8, device="cuda")

    def give_back(self):
        import torch
        self.t = None
        torch.cuda.empty_cache()


def test_no_memory_to_cut_tiles(cc):
    """From the memory that holds the graph and its tiles down to what does not
    hold the graph: in between the graph is there without tiles."""
    n, s, d = synth.grid_edges(2048, 1024)
    rounds = []
    for left in range(480, 160, -20):
        m = Short(left << 20)
        try:
            g, _ = cc.cc_graph_from_edges(n, s, d)
        except cc.CCError as e:
            assert e.code == cc.CC_ERR_OOM
            rounds.append(0)
            continue
        finally:
            m.give_back()
        try:
            C = np.array([0, 7777, n - 1], np.int32)
            r = cc.cc_estimate(g, C)
            x, y = np.arange(n) % 2048, np.arange(n) // 2048
            T = np.stack([np.abs(x - c % 2048) + np.abs(y - c // 2048) for c in C])
            assert np.array_equal(r["sum"], T.sum(0).astype(np.uint64))
            rounds.append(int(cc.cc_last_pass_stats(g)["levels"]))
        finally:
            cc.cc_graph_free(g)
    levels = 2048 + 1024 - 2
    assert rounds[0] > 0 and rounds[0] < levels  # tiles
    assert levels in rounds                      # none: a round per level
    at = rounds.index(levels)
    assert all(0 < x < levels for x in rounds[:at])


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("call", ["hybrid", "adaptive"])
def test_no_memory_to_search_tiles(cc, weighted, call):
    """The labels of an earlier call are held, the hybrid's tables do not fit
    beside them: the search that the tiles replace runs in their place."""
    n, s, d = synth.grid_edges(64, 3900)
    w = np.full(s.size, 1, np.uint32) if weighted else None
    k = 512
    g, _ = cc.cc_graph_from_edges(n, s, d, w)
    try:
        C = cc.cc_sample_choose(g, k, 2)
        o = cc.cc_opts_default(k)

        def run():
            if call == "adaptive":
                return cc.cc_estimate_adaptive(g, C, o)
            return cc.cc_estimate(g, C, o)

        o.want_hybrid = 0
        cc.cc_estimate(g, C, o)
        o.want_hybrid = 1
        m = Short(12 << 20)
        try:
            r = run()
        finally:
            m.give_back()
        want = run()
        assert cc.cc_last_pass_stats(g)["levels"] < 3000  # tiles again
    finally:
        cc.cc_graph_free(g)
    for key in want:
        assert np.array_equal(r[key], want[key]), key
