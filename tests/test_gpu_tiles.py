"""Estimates on graphs of narrow frontiers, whose search runs on tiles, against
the oracle and against the level-synchronous searches they replace (the
two-pass form on unit lengths, explicit buckets with arc lengths): grids,
paths, ladders, street lattices and road-like graphs, one source to several
words of them, tiles of one node to the largest, the error estimate and the
adaptive hybrid.  Integers bit-exact; FP64 within 1e-12 relative (one
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


def lattice(width, height, keep, seed, wmax):
    n, s, d = synth.grid_edges(width, height)
    rng = np.random.default_rng(seed)
    sel = rng.random(s.size) < keep
    s, d = s[sel], d[sel]
    return n, s, d, rng.integers(1, wmax + 1, s.size).astype(np.uint32)


def caterpillar(n):
    # a spine with two legs per node: rows of four, ids scrambled
    spine = np.arange(n - 1)
    legs = np.arange(n)
    s = np.concatenate([spine, legs, legs])
    d = np.concatenate([spine + 1, n + 2 * legs, n + 2 * legs + 1])
    p = np.random.default_rng(5).permutation(3 * n)
    return 3 * n, p[s].astype(np.uint32), p[d].astype(np.uint32), None


GRAPHS = {
    "grid": lambda: (*synth.grid_edges(70, 61), None),
    "strip": lambda: (*synth.grid_edges(3, 900), None),
    "path": lambda: (*synth.path_edges(6000), None),
    "caterpillar": lambda: caterpillar(700),
    "streets": lambda: lattice(64, 50, 0.7, 3, 1),
    "grid-w": lambda: lattice(40, 45, 1.0, 4, 9),
    "streets-w": lambda: lattice(75, 60, 0.68, 5, 1000),
    "streets-w1e6": lambda: lattice(50, 50, 0.75, 6, 1000000),
}


def off(cc, g, weighted):
    """Send the graph's estimates to the search without tiles."""
    if weighted:
        cc.cc_set_param(g, cc.CC_PARAM_SSSP_DELTA, 4000)
    else:
        cc.cc_set_param(g, cc.CC_PARAM_HYBRID_ONE_PASS, 0)


def same(r, want, keys):
    for key in keys:
        if r[key].dtype.kind == "f":
            assert (np.abs(r[key] - want[key]) <= RTOL * np.abs(want[key])).all(), key
        else:
            assert np.array_equal(r[key], want[key]), key


@pytest.mark.parametrize("k", [1, 31, 33, 64, 100, 260])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_tiles_match_oracle(cc, name, k):
    n, s, d, w = GRAPHS[name]()
    if name.startswith("streets") and w is not None and w.max() == 1:
        w = None
    g, _ = cc.cc_graph_from_edges(n, s, d, w)
    try:
        og = orc.csr_from_edges(n, s, d, w=w)
        C = cc.cc_sample_choose(g, k, 17)
        o = cc.cc_opts_default(k)
        try:
            for _ in range(2):
                r = cc.cc_estimate(g, C, o, want_sqerr=True)
        except cc.CCError as e:  # a histogram beyond the limit: refused either way
            off(cc, g, w is not None)
            with pytest.raises(cc.CCError) as other:
                cc.cc_estimate(g, C, o, want_sqerr=True)
            assert name == "streets-w1e6" and k >= 64
            assert e.code == other.value.code == cc.CC_ERR_TOO_LARGE
            return
        rounds = cc.cc_last_pass_stats(g)["levels"]
        off(cc, g, w is not None)
        r2 = cc.cc_estimate(g, C, o, want_sqerr=True)
        assert rounds < cc.cc_last_pass_stats(g)["levels"]  # the other search ran
    finally:
        cc.cc_graph_free(g)
    want = orc.estimate(og, C, eps=(o.eps_num, o.eps_den))
    same(r, want, ("pivot", "delta", "sum", "S_samp", "delta_cc", "hyb", "s_hat", "closeness"))
    for key in r:
        assert np.array_equal(r[key], r2[key]), key


@pytest.mark.parametrize("name", ["grid", "streets-w"])
def test_tiles_adaptive_and_options(cc, name):
    n, s, d, w = GRAPHS[name]()
    g, _ = cc.cc_graph_from_edges(n, s, d, w)
    try:
        C = cc.cc_sample_choose(g, 50, 2)
        first = cc.cc_estimate_adaptive(g, C)
        o = cc.cc_opts_default(50)
        o.want_hybrid = 0
        plain = cc.cc_estimate(g, C, o)
        o.want_hybrid, o.eps_num, o.eps_den = 1, 1, 1
        one = cc.cc_estimate(g, C, o)
        off(cc, g, w is not None)
        for key, x in cc.cc_estimate_adaptive(g, C).items():
            assert np.array_equal(first[key], x), key
        for key, x in cc.cc_estimate(g, C, o).items():
            assert np.array_equal(one[key], x), key
        o.want_hybrid = 0
        for key, x in cc.cc_estimate(g, C, o).items():
            assert np.array_equal(plain[key], x), key
    finally:
        cc.cc_graph_free(g)


def test_tiles_and_other_entry_points(cc):
    """Entry points that keep the shortest-path rounds run on a graph cut into
    tiles, before and after an estimate on the tiles."""
    n, s, d, w = lattice(40, 40, 0.8, 8, 50)
    og = orc.csr_from_edges(n, s, d, w=w)
    for first in (False, True):
        g, _ = cc.cc_graph_from_edges(n, s, d, w)
        try:
            if first:
                cc.cc_estimate(g, cc.cc_sample_choose(g, 20, 1))
            _, S = cc.cc_exact(g)
            assert np.array_equal(S, orc.exact_S(og))
            C = cc.cc_sample_choose(g, 64, 3)
            r = cc.cc_estimate(g, C)
            assert np.array_equal(r["S_samp"], S[C])
        finally:
            cc.cc_graph_free(g)


def test_lengths_near_the_limit(cc):
    """Distances up to 2^32 - 2 are answered; beyond, the call is refused as
    by the shortest-path rounds."""
    n = 1500
    _, s, d = synth.path_edges(n)
    for top, fits in ((2 ** 32 - 2, True), (2 ** 32 - 1, False)):
        w = np.full(n - 1, top // (n - 1), np.uint32)
        w[: top - int(w.sum())] += 1
        assert int(w.sum()) == top
        g, _ = cc.cc_graph_from_edges(n, s, d, w)
        try:
            o = cc.cc_opts_default(1)
            o.want_hybrid = 0  # no histogram of four thousand million distances
            got = []
            for explicit in (False, True):
                if explicit:
                    off(cc, g, True)
                try:
                    r = cc.cc_estimate(g, np.array([0], np.int32), o)
                    got.append(int(r["sum"][n - 1]))
                except cc.CCError as e:
                    got.append(e.code)
            assert got[0] == got[1]
            if fits:
                assert got[0] in (top, cc.CC_ERR_TOO_LARGE)
            else:
                assert got[0] == cc.CC_ERR_TOO_LARGE
        finally:
            cc.cc_graph_free(g)
