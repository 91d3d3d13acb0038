"""Estimates that take the distances as bit planes (round trips, the error
estimate, the adaptive hybrid, node weights) against the oracle, at one to
thirty-two words of sources and at depths around the 15 levels that the planes
hold, beyond which the other forms take over.  Integers bit-exact; FP64 within
1e-12 relative (one numerator, at most two roundings)."""
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


def close(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return (np.abs(a - b) <= RTOL * np.abs(b)).all()


@pytest.mark.parametrize("tail", [0, 10, 11, 12, 13, 40])
@pytest.mark.parametrize("directed", [False, True])
def test_depths_around_the_limit(cc, tail, directed):
    n, s, d = comet(600, tail, directed)
    k = 70
    g, _ = cc.cc_graph_from_edges(n, s, d, directed=directed)
    og = orc.csr_from_edges(n, s, d, directed=directed)
    try:
        C = cc.cc_sample_choose(g, k, 4)
        for eps in ((1, 8), (1, 2), (99, 100)):
            o = cc.cc_opts_default(k)
            o.eps_num, o.eps_den, o.roundtrip = *eps, int(directed)
            T = orc.dist_table(og, C, roundtrip=directed)
            want, se = orc.sqerr_from_table(T, C, eps)
            for _ in range(3):
                r = cc.cc_estimate(g, C, o, want_sqerr=True)
                assert np.array_equal(r["delta_cc"], T[:, C])
                assert np.array_equal(r["sum"], T.sum(0, dtype=np.uint64))
                assert np.array_equal(r["delta"], T.min(0))
                assert close(r["s_hat"][3], want) and close(r["sq_err"], se), eps
    finally:
        cc.cc_graph_free(g)


@pytest.mark.parametrize("k", [1, 64, 65, 200, 400, 700, 1100])
@pytest.mark.parametrize("directed", [False, True])
def test_every_width(cc, k, directed):
    n, s, d = synth.rmat_edges(12, 10, seed=21)
    g, _ = cc.cc_graph_from_edges(n, s, d, directed=directed)
    og = orc.csr_from_edges(n, s, d, directed=directed)
    try:
        C = cc.cc_sample_choose(g, k, 6)
        T = orc.dist_table(og, C, roundtrip=directed)
        o = cc.cc_opts_default(k)
        o.eps_num, o.eps_den, o.roundtrip = 2, 3, int(directed)
        r = cc.cc_estimate(g, C, o, want_sqerr=True)
        want, se = orc.sqerr_from_table(T, C, (2, 3))
        assert np.array_equal(r["sum"], T.sum(0, dtype=np.uint64))
        assert np.array_equal(r["pivot"], T.argmin(0))
        assert np.array_equal(r["S_samp"], T.sum(1, dtype=np.uint64))
        assert close(r["s_hat"][3], want) and close(r["sq_err"], se)
        ad = cc.cc_estimate_adaptive(g, C, o)
        best = None
        for e, eps in enumerate(cc.ADAPTIVE_EPS):
            h, q = orc.sqerr_from_table(T, C, eps)
            if best is None:
                best, err, ch = h.copy(), q.copy(), np.zeros(og.n, np.int32)
            else:
                less = q < err
                best[less], err[less], ch[less] = h[less], q[less], e
        ch[C] = -1
        assert np.array_equal(ad["choice"], ch)
        assert close(ad["s_hat"], best) and close(ad["sq_err"], err)
    finally:
        cc.cc_graph_free(g)


@pytest.mark.parametrize("k", [5, 100, 300])
@pytest.mark.parametrize("directed", [False, True])
def test_adaptive_eps_in_any_order(cc, k, directed):
    """More eps than a node's words, unsorted and repeated: the first of the
    smallest squared error."""
    n, s, d = synth.watts_strogatz_edges(900, 6, 0.3, seed=8)
    eps = [(1, 2), (1, 9), (9, 10), (1, 2), (1, 3), (3, 4), (1, 1), (2, 3), (1, 1000), (5, 7),
           (4, 9)]
    g, _ = cc.cc_graph_from_edges(n, s, d, directed=directed)
    og = orc.csr_from_edges(n, s, d, directed=directed)
    try:
        C = cc.cc_sample_choose(g, k, 2)
        T = orc.dist_table(og, C, roundtrip=directed)
        o = cc.cc_opts_default(k)
        o.roundtrip = int(directed)
        ad = cc.cc_estimate_adaptive(g, C, o, eps)
        hq = [orc.sqerr_from_table(T, C, e) for e in eps]
        at = np.argmin(np.stack([q for _, q in hq]), axis=0)
        other = np.setdiff1d(np.arange(og.n), C)
        got = ad["choice"][other]
        for v, e in zip(other, got):  # ties within rounding may fall to either
            assert e == at[v] or close(hq[e][1][v], hq[at[v]][1][v])
            assert close(ad["s_hat"][v], hq[e][0][v]) and close(ad["sq_err"][v], hq[e][1][v])
        assert (ad["choice"][C] == -1).all()
    finally:
        cc.cc_graph_free(g)


@pytest.mark.parametrize("k", [3, 64, 130, 300, 600])
@pytest.mark.parametrize("eps", [(1, 16), (1, 2), (9, 10)])
@pytest.mark.parametrize("directed", [False, True])
def test_node_weights(cc, k, eps, directed):
    n, s, d = synth.rmat_edges(11, 8, seed=23)
    g, _ = cc.cc_graph_from_edges(n, s, d, directed=directed)
    og = orc.csr_from_edges(n, s, d, directed=directed)
    try:
        rng = np.random.default_rng(k)
        beta = np.minimum(np.floor(rng.pareto(1.1, og.n) * 10), 1e6).astype(np.uint32)
        cc.cc_graph_set_node_weights(g, beta)
        C, tau = cc.cc_sample_varopt(g, k, 5)
        o = cc.cc_opts_default(k)
        o.eps_num, o.eps_den, o.roundtrip = *eps, int(directed)
        r = cc.cc_estimate_node_weighted(g, C, tau, o)
    finally:
        cc.cc_graph_free(g)
    T = orc.dist_table(og, C, roundtrip=directed).astype(object)
    b = beta.astype(object)
    tn, td = tau
    S = (T * b[None, :]).sum(1)
    assert [int(x) for x in r["S_sampled"]] == [int(x) for x in S]
    piv = orc.dist_table(og, C, roundtrip=directed).argmin(0)
    inC = np.zeros(og.n, bool)
    inC[C] = True
    mu = [max(tn, int(b[c]) * td) for c in C]
    for v in range(0, og.n, 7):
        if inC[v]:
            want = (S[list(C).index(v)],) * 2
            td_ = 1
        else:
            p, td_ = piv[v], td
            D = T[p, v]
            far = [T[p, c] * eps[0] > D * eps[1] for c in C]
            samp = sum(m * T[i, v] for i, m in enumerate(mu))
            hyb = sum((int(b[C[i]]) * td if far[i] else mu[i]) * T[i, v] for i in range(k))
            tail = sum(b[u] * T[p, u] for u in range(og.n)
                       if not inC[u] and T[p, u] * eps[0] > D * eps[1])
            want = (samp, hyb + td * tail)
        for e in range(2):
            assert abs(r["s_hat"][e][v] * td_ - want[e]) <= 1e-12 * want[e], (v, e)
