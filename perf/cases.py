"""Performance cases of the closeness library: the calls its users make, over
the graphs, sample sizes and options they make them with.

A case is a dict of plain values with a "kind" (which entry point) and a
"graph" (which family), both explained where they are listed.  prepare()
builds a graph from the seed and keeps its handle, sample and output buffers
as a program would; run() is one call through the public binding; exact()
recomputes the floating-point outputs from the definitions in 64 bits.
"""
import ctypes
import math
import random

import numpy as np
import torch

import paper_1409_0035_gb300 as cc

DEV = "cuda"


def listed():
    return [
        # One new estimate on a small social graph, sample drawn and results
        # taken as host arrays: what an interactive user or a service with
        # many small graphs calls; launches and copies count.
        dict(name="social12_new", kind="new", graph="rmat", scale=12, ef=8, k=64),
        # The all-nodes estimate of a large social or web graph, every
        # estimator, results left on the device for the program's next step.
        dict(name="social20", kind="estimate", graph="rmat", scale=20, ef=16, k=256),
        # A wide sample for accuracy on a medium graph (k of no round size,
        # sixteen words per node).
        dict(name="social18_wide", kind="estimate", graph="rmat", scale=18, ef=16, k=1000),
        # A mesh: thousands of small frontiers instead of a few large ones.
        dict(name="mesh1024", kind="estimate", graph="grid", width=1024, height=1024, k=256),
        # A small-world network (peer-to-peer or sensor overlay).
        dict(name="smallworld16", kind="estimate", graph="ws", n=65536, k=512),
        # A road network with arc lengths.
        dict(name="road500k", kind="estimate", graph="road", width=720, height=700, k=64),
        # Round-trip distances of a directed web graph.
        dict(name="roundtrip20", kind="estimate", graph="drmat", scale=20, ef=16, k=128),
        # Nodes of unequal importance (population, traffic): weighted sample
        # and both weighted estimates.
        dict(name="weighted18", kind="nodeweighted", graph="rmat", scale=18, ef=16, k=256),
        # Outbound centrality of a directed graph kept whole.
        dict(name="outbound18", kind="reach", graph="drmat", scale=18, ef=16, k=64),
        # The hybrid with its threshold chosen per node by estimated error.
        dict(name="adaptive18", kind="adaptive", graph="rmat", scale=18, ef=16, k=256),
        # Many small graphs of mixed families and sample sizes in one run.
        dict(name="batch12", kind="batch", graphs=12, plan=7),
        # From an edge list in host memory to host results: build, sample,
        # estimate, release.  Every program pays it once per graph.
        dict(name="ingest18", kind="ingest", graph="rmat", scale=18, ef=16, k=128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["new", "social", "mesh", "smallworld", "road", "roundtrip", "weighted",
                       "outbound", "adaptive", "batch", "ingest"])
    ef = rng.randint(8, 16)
    k = _log(rng, 16, 1024)
    if what == "new":
        return dict(kind="new", graph="rmat", scale=rng.randint(10, 14), ef=ef, k=min(k, 512))
    if what == "social":
        return dict(kind="estimate", graph="rmat", scale=rng.randint(12, 19), ef=ef, k=k)
    if what == "mesh":
        w, h = _log(rng, 64, 1000), _log(rng, 64, 1000)
        return dict(kind="estimate", graph="grid", width=w, height=h, k=min(k, 300))
    if what == "smallworld":
        return dict(kind="estimate", graph="ws", n=_log(rng, 4096, 131072), k=k)
    if what == "road":
        w, h = _log(rng, 64, 700), _log(rng, 64, 700)
        return dict(kind="estimate", graph="road", width=w, height=h, k=min(k, 128))
    if what == "roundtrip":
        return dict(kind="estimate", graph="drmat", scale=rng.randint(13, 19), ef=ef, k=min(k, 256))
    if what == "weighted":
        return dict(kind="nodeweighted", graph="rmat", scale=rng.randint(12, 18), ef=ef,
                    k=min(k, 512))
    if what == "outbound":
        return dict(kind="reach", graph="drmat", scale=rng.randint(12, 18), ef=ef,
                    k=_log(rng, 16, 128), inbound=rng.random() < 0.5)
    if what == "adaptive":
        return dict(kind="adaptive", graph="rmat", scale=rng.randint(12, 18), ef=ef,
                    k=min(k, 512))
    if what == "batch":
        return dict(kind="batch", graphs=rng.randint(4, 12), plan=rng.randrange(1 << 20))
    if rng.random() < 0.5:
        return dict(kind="ingest", graph="rmat", scale=rng.randint(12, 18), ef=ef, k=min(k, 256))
    return dict(kind="ingest", graph="road", width=_log(rng, 64, 400), height=_log(rng, 64, 400),
                k=min(k, 64))


# ------------------------------------------------------------------ inputs

def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + stream * 7919 + 12345) % (1 << 62))
    return g


def _edges(case, seed):
    """(n, src, dst, lengths or None) as device tensors.  Which edges an
    R-MAT or road graph has depends on the case alone, so that its largest
    component has one size; the seed gives the ids and the lengths."""
    fixed, g = _gen(1, 0), _gen(seed, 1)
    kind = case["graph"]
    if kind in ("rmat", "drmat"):
        # R-MAT with quadrants 0.57, 0.19, 0.19, 0.05 and scrambled ids
        n, m = 1 << case["scale"], case["ef"] << case["scale"]
        s = torch.zeros(m, dtype=torch.int64, device=DEV)
        d = torch.zeros(m, dtype=torch.int64, device=DEV)
        for _ in range(case["scale"]):
            u = torch.rand(m, device=DEV, generator=fixed)
            s.mul_(2).add_(u >= 0.76)
            d.mul_(2).add_(((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
        name = torch.randperm(n, device=DEV, generator=g)
        return n, name[s], name[d], None
    if kind == "grid":
        w, h = case["width"], case["height"]
        ids = torch.arange(w * h, device=DEV).reshape(h, w)
        return (w * h, torch.cat([ids[:, :-1].reshape(-1), ids[:-1].reshape(-1)]),
                torch.cat([ids[:, 1:].reshape(-1), ids[1:].reshape(-1)]), None)
    if kind == "ws":
        # ring of degree 10, 5 % of the edges rewired
        n = case["n"]
        u = torch.arange(n, device=DEV).repeat_interleave(5)
        v = (u + torch.arange(1, 6, device=DEV).repeat(n)) % n
        far = torch.randint(0, n, (5 * n,), device=DEV, generator=g)
        move = torch.rand(5 * n, device=DEV, generator=g) < 0.05
        return n, u, torch.where(move, far, v), None
    if kind == "road":
        # jittered street lattice with 35 % of its segments missing (mean
        # degree 2.6), lengths Euclidean
        w, h = case["width"], case["height"]
        ids = torch.arange(w * h, device=DEV).reshape(h, w)
        x = (ids % w).reshape(-1) + 0.8 * torch.rand(w * h, device=DEV, generator=g)
        y = (ids // w).reshape(-1) + 0.8 * torch.rand(w * h, device=DEV, generator=g)
        s = torch.cat([ids[:, :-1].reshape(-1), ids[:-1].reshape(-1)])
        d = torch.cat([ids[:, 1:].reshape(-1), ids[1:].reshape(-1)])
        keep = torch.rand(s.numel(), device=DEV, generator=fixed) < 0.65
        s, d = s[keep], d[keep]
        ln = torch.sqrt((x[s] - x[d]).double() ** 2 + (y[s] - y[d]).double() ** 2)
        return w * h, s, d, (1000.0 * ln).round().long() + 1
    raise ValueError(kind)


def _u32(t):
    return None if t is None else t.to(torch.int32).cpu().numpy().view(np.uint32)


def _host_edges(case, seed):
    n, s, d, w = _edges(case, seed)
    return n, _u32(s), _u32(d), _u32(w)


def _node_weights(n, seed):
    u = torch.rand(n, device=DEV, generator=_gen(seed, 2), dtype=torch.float64)
    x = (1.0 - u) ** (-1.0 / 1.2) - 1.0
    return torch.clamp(torch.floor(10 * x) + 1, max=1e6).long()


def _batch_members(case):
    """(graph case, k) of each member: half R-MAT, a quarter grids, a quarter
    Watts-Strogatz."""
    r = random.Random(case["plan"])
    out = []
    for i in range(case["graphs"]):
        k = r.choice([16, 64, 256, 512])
        if i % 4 < 2:
            c = dict(graph="rmat", scale=r.randint(10, 15), ef=r.randint(8, 16))
        elif i % 4 == 2:
            side = r.randint(64, 200)
            c = dict(graph="grid", width=side, height=side)
        else:
            c = dict(graph="ws", n=1 << r.randint(12, 14))
        out.append((c, k))
    return out


class State:
    """Handles and buffers of one prepared case; frees what it holds."""

    def __init__(self, case, seed):
        self.case, self.seed, self.handles, self.batch = case, int(seed), [], None

    def build(self, case, seed, keep=True):
        n, s, d, w = _host_edges(case, seed)
        g, _ = cc.cc_graph_from_edges(n, s, d, w, directed=case["graph"] == "drmat",
                                      keep_component=keep)
        self.handles.append(g)
        return g

    def __del__(self):
        if cc is None:
            return
        if self.batch is not None:
            cc.cc_batch_free(self.batch)
        for g in self.handles:
            cc.cc_graph_free(g)


def _device_out(n):
    t = dict(s_hat=torch.zeros((4, n), dtype=torch.float64, device=DEV),
             closeness=torch.zeros((4, n), dtype=torch.float64, device=DEV),
             pivot=torch.zeros(n, dtype=torch.int32, device=DEV),
             delta=torch.zeros(n, dtype=torch.int32, device=DEV),
             sum=torch.zeros(n, dtype=torch.int64, device=DEV))
    o = cc.cc_out()
    for e in range(4):
        o.s_hat[e] = t["s_hat"][e].data_ptr()
        o.closeness[e] = t["closeness"][e].data_ptr()
    o.pivot, o.delta, o.sample_sum = (t[x].data_ptr() for x in ("pivot", "delta", "sum"))
    return t, o


def prepare(case, seed):
    kind = case["kind"]
    s = State(case, seed)
    if kind == "ingest":
        s.edges = _host_edges(case, seed)
        return s
    if kind == "batch":
        s.ks, samples, s.outs = [], [], []
        for i, (c, k) in enumerate(_batch_members(case)):
            g = s.build(c, seed * 64 + i)
            n = cc.cc_graph_info(g)[0]
            k = min(k, n)
            samples.append(cc.cc_sample_choose(g, k, seed + i))
            s.outs.append(_device_out(n))
        s.batch = cc.cc_batch_create(s.handles, samples, autotune=False)
        return s
    g = s.g = s.build(case, seed, keep=kind != "reach")
    n = cc.cc_graph_info(g)[0]
    k = s.k = min(case["k"], n)
    if kind in ("new", "reach"):
        return s
    if kind == "nodeweighted":
        cc.cc_graph_set_node_weights(g, _u32(_node_weights(n, seed)))
        s.sample, s.tau = cc.cc_sample_varopt(g, k, seed)
        s.out = dict(s_hat=torch.zeros((2, n), dtype=torch.float64, device=DEV),
                     closeness=torch.zeros((2, n), dtype=torch.float64, device=DEV))
        s.cout = cc.cc_wout()
        for e in range(2):
            s.cout.s_hat[e] = s.out["s_hat"][e].data_ptr()
            s.cout.closeness[e] = s.out["closeness"][e].data_ptr()
        s.opts = cc.cc_opts_default(k)
        s.opts.device_outputs = 1
        return s
    s.sample = cc.cc_sample_choose(g, k, seed)
    s.opts = cc.cc_opts_default(k)
    if kind == "estimate":
        s.opts.device_outputs = 1
        s.opts.roundtrip = int(case["graph"] == "drmat")
        s.out, s.cout = _device_out(n)
    return s


def run(s):
    kind = s.case["kind"]
    if kind == "estimate":
        cc.cc_estimate(s.g, s.sample, s.opts, out=s.cout)
        return s.out
    if kind == "new":
        return cc.cc_estimate(s.g, cc.cc_sample_choose(s.g, s.k, s.seed))
    if kind == "nodeweighted":
        cc.cc_estimate_node_weighted(s.g, s.sample, s.tau, s.opts, out=s.cout)
        return s.out
    if kind == "reach":
        return cc.cc_reach_estimate(s.g, s.k, s.seed, inbound=s.case.get("inbound", False))
    if kind == "adaptive":
        return cc.cc_estimate_adaptive(s.g, s.sample, s.opts)
    if kind == "batch":
        cc.cc_batch_run(s.batch)
        for i, (_, o) in enumerate(s.outs):
            rc = cc.lib().cc_batch_result(s.batch, i, ctypes.byref(o), 1)
            if rc != cc.CC_OK:
                raise cc.CCError(rc, "cc_batch_result")
        return [t for t, _ in s.outs]
    n, src, dst, w = s.edges
    g, old = cc.cc_graph_from_edges(n, src, dst, w)
    try:
        k = min(s.case["k"], cc.cc_graph_info(g)[0])
        r = cc.cc_estimate(g, cc.cc_sample_choose(g, k, s.seed))
    finally:
        cc.cc_graph_free(g)
    r["old_id"] = old
    return r


# ------------------------------------------------------------------ work

def _size(c):
    """(nodes, edges) given, before duplicates and small components go."""
    if c["graph"] in ("rmat", "drmat"):
        return 1 << c["scale"], c["ef"] << c["scale"]
    if c["graph"] == "ws":
        return c["n"], 5 * c["n"]
    n = c["width"] * c["height"]
    return n, int(2 * n * (0.65 if c["graph"] == "road" else 1.0))


def work(case):
    """Bytes of a pass: the graph's rows once (both directions of an
    undirected edge, both graphs of a round trip) and every output once."""
    if case["kind"] == "batch":
        parts = [dict(c, kind="estimate", k=k) for c, k in _batch_members(case)]
        return {"bytes": sum(work(p)["bytes"] for p in parts), "flops": 0}
    n, m = _size(case)
    arcs = m if case["kind"] == "reach" else 2 * m
    csr = 8.0 * n + (8.0 if case["graph"] == "road" else 4.0) * arcs
    out = {"estimate": 80, "new": 128, "ingest": 132, "nodeweighted": 36, "reach": 36,
           "adaptive": 28}[case["kind"]] * float(n)
    if case["kind"] == "new":
        out += 4.0 * case["k"] ** 2
    if case["kind"] == "ingest":
        out += 4.0 * case["k"] ** 2 + (12.0 if case["graph"] == "road" else 8.0) * m
    return {"bytes": csr + out, "flops": 0}


# ------------------------------------------------------------------ exact

_MASK = (1 << 64) - 1


def _keys(seed, lo, hi):
    """splitmix64 outputs number lo .. hi-1 of stream `seed`."""
    c = np.arange(lo, hi, dtype=np.uint64)
    with np.errstate(over="ignore"):
        z = np.uint64(seed & _MASK) + (c + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _bottom_k(n, k, seed):
    order = np.argsort(_keys(seed, 0, n), kind="stable")
    return torch.from_numpy(order[:k].astype(np.int64)).to(DEV)


def _reach(n, src, dst, start):
    seen = torch.zeros(n, dtype=torch.bool, device=DEV)
    seen[start] = True
    while True:
        before = int(seen.sum())
        seen[dst[seen[src]]] = True
        if int(seen.sum()) == before:
            return seen


def _simple_graph(case, seed):
    """(n, src, dst, lengths) of the arcs of the largest component: loops
    dropped, parallel arcs merged at their smallest length, ids renumbered
    in order."""
    n, s, d, w = _edges(case, seed)
    directed = case["graph"] == "drmat"
    if not directed:
        s, d = torch.cat([s, d]), torch.cat([d, s])
        w = None if w is None else torch.cat([w, w])
    ok = s != d
    key = s[ok] * n + d[ok]
    uniq, inv = torch.unique(key, return_inverse=True)
    if w is not None:
        w = torch.full_like(uniq, 1 << 40).scatter_reduce(0, inv, w[ok], "amin")
    s, d = uniq // n, uniq % n
    if directed:
        deg = torch.bincount(s, minlength=n) * torch.bincount(d, minlength=n)
        p = int(deg.argmax())
        keep = _reach(n, s, d, p) & _reach(n, d, s, p)
    else:
        lab = torch.arange(n, device=DEV)
        while True:
            new = lab.scatter_reduce(0, d, lab[s], "amin")
            new = new[new]
            if torch.equal(new, lab):
                break
            lab = new
        keep = lab == torch.bincount(lab, minlength=n).argmax()
    ids = torch.cumsum(keep, 0) - 1
    arc = keep[s] & keep[d]
    return int(keep.sum()), ids[s[arc]], ids[d[arc]], None if w is None else w[arc]


def _bfs(n, s, d, sample):
    """Hop distances from each sampled node, n x k int32."""
    rows = torch.bincount(d, minlength=n)
    crow = torch.cat([rows.new_zeros(1), rows.cumsum(0)])
    order = torch.argsort(d, stable=True)
    A = torch.sparse_csr_tensor(crow, s[order], torch.ones(s.numel(), device=DEV), (n, n))
    D = torch.full((n, sample.numel()), -1, dtype=torch.int32, device=DEV)
    for lo in range(0, sample.numel(), 128):
        sub = sample[lo:lo + 128]
        part = D[:, lo:lo + 128]
        X = torch.zeros((n, sub.numel()), device=DEV)
        X[sub, torch.arange(sub.numel(), device=DEV)] = 1.0
        part[X > 0] = 0
        level = 0
        while True:
            level += 1
            new = ((A @ X) > 0) & (part < 0)
            if not bool(new.any()):
                break
            part[new] = level
            X = new.float()
    return D


def _bellman_ford(n, s, d, w, sample):
    """Shortest-path distances on a graph of small degree, n x k int32."""
    deg = torch.bincount(d, minlength=n)
    order = torch.argsort(d, stable=True)
    start = deg.cumsum(0) - deg
    slot = torch.arange(s.numel(), device=DEV) - start[d[order]]
    K = int(deg.max())
    nb = torch.arange(n, device=DEV).repeat(K, 1)
    ln = torch.zeros((K, n, 1), dtype=torch.int32, device=DEV)
    nb[slot, d[order]] = s[order]
    ln[slot, d[order], 0] = w[order].int()
    D = torch.full((n, sample.numel()), 1 << 30, dtype=torch.int32, device=DEV)
    D[sample, torch.arange(sample.numel(), device=DEV)] = 0
    r = 0
    while True:
        new = D
        for q in range(K):
            new = torch.minimum(new, D[nb[q]] + ln[q])
        r += 1
        if r % 16 == 0 and torch.equal(new, D):
            return D
        D = new


def _distances(case, seed, sample_of):
    """(n, sample, n x k int32 distances)."""
    if case["graph"] == "grid":
        w, n = case["width"], case["width"] * case["height"]
        sample = sample_of(n)
        v = torch.arange(n, device=DEV)[:, None]
        D = (v % w - sample % w).abs() + (v // w - sample // w).abs()
        return n, sample, D.int()
    n, s, d, w = _simple_graph(case, seed)
    sample = sample_of(n)
    if case["graph"] == "road":
        return n, sample, _bellman_ford(n, s, d, w, sample)
    D = _bfs(n, s, d, sample)
    if case["graph"] == "drmat":
        D += _bfs(n, d, s, sample)
    return n, sample, D


def _pivots(D):
    k = D.shape[1]
    i = torch.arange(k, device=DEV)
    best = torch.cat([(D[lo:lo + 65536].long() * k + i).amin(1)
                      for lo in range(0, D.shape[0], 65536)])
    return best % k, best // k


def _tails(D, sample, pivot, thr, weight=None):
    """Per node: how many unsampled nodes (or their weight) lie farther than
    thr from its pivot, and the sum of their (weighted) distances."""
    n, k = D.shape
    un = torch.ones(n, dtype=torch.bool, device=DEV)
    un[sample] = False
    num = torch.zeros(n, dtype=torch.int64, device=DEV)
    tot = torch.zeros(n, dtype=torch.int64, device=DEV)
    mass = None if weight is None else weight[un]
    by = torch.argsort(pivot, stable=True)
    cut = torch.cat([pivot.new_zeros(1), torch.bincount(pivot, minlength=k).cumsum(0)]).tolist()
    for i in range(k):
        v = by[cut[i]:cut[i + 1]]
        x, order = torch.sort(D[un, i].long())
        m = torch.ones_like(x) if mass is None else mass[order]
        cn = torch.cat([x.new_zeros(1), m.cumsum(0)])
        cs = torch.cat([x.new_zeros(1), (m * x).cumsum(0)])
        at = torch.searchsorted(x, thr[v], right=True)
        num[v] = cn[-1] - cn[at]
        tot[v] = cs[-1] - cs[at]
    return num, tot


def _hybrid(D, sample, S, pivot, delta, a, b, sq=False):
    """Estimate (and its error estimate) of the hybrid for eps = a / b."""
    n, k = D.shape
    thr = delta * b // a
    Hnum, Hsum = _tails(D, sample, pivot, thr)
    C = D[sample].long()  # row p: distances between sampled nodes
    C = C.T.contiguous()
    est = torch.empty(n, dtype=torch.float64, device=DEV)
    err = torch.zeros(n, dtype=torch.float64, device=DEV)
    if sq:
        far = C.clone()
        far.fill_diagonal_(-1)
        istar = (far * k + (k - 1 - torch.arange(k, device=DEV))).argmax(1)
    for lo in range(0, n, 65536):
        hi = min(n, lo + 65536)
        d, p, t = D[lo:hi].long(), pivot[lo:hi], thr[lo:hi]
        near = C[p] <= t[:, None]
        L = near.sum(1)
        LCsum = (d * near).sum(1)
        HCsum = d.sum(1) - LCsum
        rest = (n - 1) - Hnum[lo:hi] - (k - L)
        est[lo:hi] = ((Hsum[lo:hi] + HCsum) * L + LCsum * rest).double() / L.double()
        if sq:
            LCsq = (d * d * near).sum(1)
            Ld = L.double()
            t1 = ((LCsq * L - LCsum * LCsum) * rest).double() / (Ld * Ld * Ld)
            e = d - C[p]
            e2 = ((e * e) * ~near).sum(1)
            one = e.gather(1, istar[p][:, None])[:, 0]
            H = Hnum[lo:hi]
            t2 = torch.where(L < k, (e2 * H).double() / (k - L).clamp(min=1).double(),
                             (one * one * H).double())
            err[lo:hi] = t1 + t2
    est[sample] = S.double()
    err[sample] = 0.0
    return est, err


def _estimates(case, seed, sample_seed):
    n, sample, D = _distances(case, seed, lambda nn: _bottom_k(nn, min(case["k"], nn),
                                                               sample_seed))
    k = sample.numel()
    pivot, delta = _pivots(D)
    total = torch.cat([D[lo:lo + 65536].long().sum(1) for lo in range(0, n, 65536)])
    S = torch.stack([D[:, i].long().sum() for i in range(k)])
    est = torch.empty((4, n), dtype=torch.float64, device=DEV)
    est[0] = ((n - 1) * total).double() / k
    est[1] = S[pivot].double()
    est[2] = (S[pivot] + (n - 1) * delta).double()
    est[:3, sample] = S.double()
    est[3] = _hybrid(D, sample, S, pivot, delta, 1, max(1, int(math.floor(math.sqrt(k) + 0.5))))[0]
    return dict(s_hat=est, closeness=(n - 1) / est)


def _adaptive(case, seed):
    n, sample, D = _distances(case, seed, lambda nn: _bottom_k(nn, min(case["k"], nn), seed))
    pivot, delta = _pivots(D)
    S = torch.stack([D[:, i].long().sum() for i in range(sample.numel())])
    best = err = None
    for a, b in ((1, 1000), (1, 40), (1, 20), (1, 10), (1, 5), (1, 2), (99, 100)):
        e, q = _hybrid(D, sample, S, pivot, delta, a, b, sq=True)
        if best is None:
            best, err = e, q
        else:
            less = q < err
            best, err = torch.where(less, e, best), torch.where(less, q, err)
    return dict(s_hat=best, closeness=(n - 1) / best, sq_err=err)


def _systematic(beta, k, seed):
    """(sample, tn, td): systematic draw of k nodes with probabilities
    min(1, beta td / tn) along the splitmix64 order."""
    n = beta.size
    w = np.sort(beta)[::-1].astype(np.int64)
    rest = int(w.sum())
    for h in range(k):
        if int(w[h]) * (k - h) < rest:
            break
        rest -= int(w[h])
    tn, td = rest, k - h
    order = np.argsort(_keys(seed, 0, n), kind="stable")
    x = beta[order].astype(np.int64) * td
    sure = x >= tn
    end = np.cumsum(np.where(sure, 0, x))
    begin = end - np.where(sure, 0, x)
    u = (int(_keys(seed, n, n + 1)[0]) * tn) >> 64

    def below(y):
        return np.maximum(0, (y - u + tn - 1) // tn)

    return order[sure | (below(end) > below(begin))], tn, td


def _node_weighted(case, seed):
    n, s, d, _ = _simple_graph(case, seed)
    k = min(case["k"], n)
    beta = _node_weights(n, seed)
    ids, tn, td = _systematic(beta.cpu().numpy(), k, seed)
    sample = torch.from_numpy(ids).to(DEV)
    D = _bfs(n, s, d, sample)
    pivot, delta = _pivots(D)
    thr = delta * max(1, int(math.floor(math.sqrt(k) + 0.5)))
    _, Hsum = _tails(D, sample, pivot, thr, beta)
    C = D[sample].long().T.contiguous()
    bs = beta[sample]
    mu = torch.clamp(bs * td, min=tn)
    S = torch.stack([(D[:, i].long() * beta).sum() for i in range(k)])
    est = torch.empty((2, n), dtype=torch.float64, device=DEV)
    for lo in range(0, n, 65536):
        hi = min(n, lo + 65536)
        dd, p, t = D[lo:hi].long(), pivot[lo:hi], thr[lo:hi]
        near = C[p] <= t[:, None]
        est[0, lo:hi] = (dd * mu).sum(1).double() / td
        num = (dd * torch.where(near, mu, bs * td)).sum(1) + Hsum[lo:hi] * td
        est[1, lo:hi] = num.double() / td
    est[:, sample] = S.double()
    return dict(s_hat=est, closeness=(beta.sum() - beta).double() / est)


def exact(case, seed):
    """Floating-point outputs of run() from the definitions; None for whole
    numbers and for the reachability samples of a whole directed graph,
    whose plain computation is quadratic."""
    kind = case["kind"]
    if kind == "reach":
        return None
    if kind == "adaptive":
        return dict(_adaptive(case, seed), choice=None)
    if kind == "nodeweighted":
        return _node_weighted(case, seed)
    whole = dict(pivot=None, delta=None, sum=None)
    if kind == "batch":
        return [dict(_estimates(dict(c, k=k), seed * 64 + i, seed + i), **whole)
                for i, (c, k) in enumerate(_batch_members(case))]
    r = dict(_estimates(case, seed, seed), **whole)
    if kind in ("new", "ingest"):
        r.update(hyb=None, S_samp=None, delta_cc=None)
    if kind == "ingest":
        r["old_id"] = None
    return r
