// Outbound / inbound estimates of general directed graphs (section 6.2,
// Algorithm 4): for every node v, the k nodes of smallest rank (a seeded
// random order) among those v reaches (outbound) or that reach v (inbound),
// their distances, and the rank position of the k-th.
//
// One persistent cooperative launch walks the order in groups of 64 W
// sources whose search can still reach a node that takes samples.  Each
// group is a bit-packed multi-source BFS on the search graph (G^T for
// outbound, G for inbound: bit i leaves the group's i-th source), recording
// the level at which each bit first reaches each node; then every node it
// touched accepts its lowest-rank bits (its own excluded) until it holds k
// samples.  Bits are ranks, so the accepted ones are exactly the next samples
// in rank order.
//
// Levels 1 to 15, which bring most bits on graphs of small diameter, are kept
// as four bit planes: plane p of a node's words holds the bits whose level has
// bit p set, and accepted distances are population counts.  The bits of later
// levels have none set; their levels are stored one by one in lev.  Planes are
// zeroed by the first level that needs them and zero again when a group ends.
//
// Pruning: a node x saturated at the start of a group -- k + 1 sources
// other than x have reached it, or k have and x's own position is past --
// holds k + 1 nodes of smaller rank than every source still to come among
// x and its reachability set; every node that reaches x through x holds k
// of them other than itself, so x is neither entered nor expanded.  Nodes
// that saturate during a group still propagate that group's bits: extra
// bits only reach nodes that really reach the source, and each node keeps
// its lowest ranks, so the samples equal those of the sequential procedure
// with this pruning, and the first-arrival levels are exact distances
// (every node on a shortest path from v to an accepted source is
// unsaturated).  Algorithm 4 prunes at k nodes other than x, which can stop
// a search at a node whose k samples include v and leave v a sample short;
// the rule above keeps the stated aim, a uniform sample of size k of every
// reachability set.
//
// With arc lengths (section 6.2 runs Dijkstra) each (node, source) slot
// holds a tentative distance instead of a level: a round relaxes every
// source whose distance at a frontier node dropped into its neighbours
// (atomicMin), the nodes that improved form the next frontier, and the
// rounds end when nothing improves -- label-correcting search, exact on the
// unsaturated nodes by the same argument.  The slots of a node return to
// infinity when it takes its samples.
//
// Every wait is the bounded grid barrier (CC_ERR_TIMEOUT on expiry).
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <type_traits>

#include "barrier.cuh"
#include "nodew.h"
#include "reach.h"

namespace ccg {

namespace {

constexpr int kRT = 256;
// Positions of the order tested for useful sources at once.
constexpr int kMaxWin = 131072;
// Arcs beyond which a source is taken without a proof that it is useful.
constexpr int kTestArcs = 1024;

struct RState {
    unsigned qlen[2], blen[2];  // frontier queue: small nodes, parts of big ones
    unsigned tlen[2];
    unsigned long long levels, groups;
    uint8_t flags[2][kMaxWin / 8];  // useful positions of a window, by parity
};

// x is saturated for the sources from position base on (see above): k others
// have reached it and either another one has or its own position is past.
__device__ __forceinline__ bool saturated(const ReachJob &J, int32_t x, uint32_t base)
{
    return base >= J.satpos[x];
}

// Mark the useful sources among positions [pos, hi): unsaturated nodes with
// an unsaturated neighbour on the search graph.  The search of any other
// source touches no node but its own, whose own bit does not count, so it is
// dropped (saturation only grows: it stays useless).  Eight positions per
// warp, four lanes each over the first 64 arcs, the whole warp over a longer
// row of saturated neighbours.
__device__ void mark_useful(const ReachJob &J, int64_t pos, int64_t hi, uint8_t *flags,
                            int64_t gw, int64_t nwarps, int lane)
{
    const uint32_t base = (uint32_t)pos;
    const int64_t nbytes = (hi - pos + 31) / 32 * 4;
    const int sub = lane >> 2, t = lane & 3;
    for (int64_t wi = gw; wi < nbytes; wi += nwarps) {
        const int64_t p = pos + wi * 8 + sub;
        int64_t b = 0, e = 0;
        if (p < hi) {
            const int32_t s = J.order[p];
            if (!saturated(J, s, base)) {
                b = J.rp[s];
                e = J.rp[s + 1];
            }
        }
        bool found = false;
        int64_t x = b + t;
        for (int step = 0; step < 4; ++step, x += 16) {
            int32_t c[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) c[q] = !found && x + 4 * q < e ? J.col[x + 4 * q] : -1;
            bool f = false;
#pragma unroll
            for (int q = 0; q < 4; ++q) f |= c[q] >= 0 && !saturated(J, c[q], base);
            const unsigned m = __ballot_sync(0xFFFFFFFFu, f);
            found = found || ((m >> (4 * sub)) & 15u) != 0u;
            if (__all_sync(0xFFFFFFFFu, found || x - t + 16 >= e)) break;
        }
        unsigned rest = __ballot_sync(0xFFFFFFFFu, t == 0 && !found && e > b + 64);
        unsigned got = 0;
        while (rest) {
            const int l0 = __ffs(rest) - 1;
            rest &= rest - 1;
            const int64_t bb = __shfl_sync(0xFFFFFFFFu, b, l0) + 64;
            const int64_t ee = __shfl_sync(0xFFFFFFFFu, e, l0);
            bool any = ee - bb > kTestArcs;
            for (int64_t y = bb; y < ee && !any; y += 256) {
                int32_t c[8];
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    c[q] = y + lane + 32 * q < ee ? J.col[y + lane + 32 * q] : -1;
                bool f = false;
#pragma unroll
                for (int q = 0; q < 8; ++q) f |= c[q] >= 0 && !saturated(J, c[q], base);
                any = __any_sync(0xFFFFFFFFu, f);
            }
            if (any) got |= 1u << l0;
        }
        const unsigned m = __ballot_sync(0xFFFFFFFFu, t == 0 && found) | got;  // bits 0, 4, ..
        if (lane == 0) {
            unsigned byte = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) byte |= ((m >> (4 * q)) & 1u) << q;
            flags[wi] = (uint8_t)byte;
        }
    }
}

// The first G marked positions (offsets from the window's start, ascending)
// into s_src, by every CTA alike; returns how many the window marks.
__device__ int pick_sources(const uint8_t *flags, int64_t len, int G, int *s_src)
{
    __shared__ int s_w[kRT / 32];
    const int nwords = (int)((len + 31) / 32);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int kPer = kMaxWin / 32 / kRT;  // words per thread
    uint32_t m[kPer];
    int c = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int i = (int)threadIdx.x * kPer + j;
        m[j] = i < nwords ? __ldcg(reinterpret_cast<const uint32_t *>(flags) + i) : 0u;
        c += __popc(m[j]);
    }
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    __syncthreads();  // s_w and s_src of the group before are no longer read
    if (lane == 31) s_w[wid] = incl;
    __syncthreads();
    int at = incl - c, total = 0;
    for (int w = 0; w < kRT / 32; ++w) {
        if (w < wid) at += s_w[w];
        total += s_w[w];
    }
#pragma unroll
    for (int j = 0; j < kPer; ++j)
        for (uint32_t b = m[j]; b && at < G; b &= b - 1, ++at)
            s_src[at] = ((int)threadIdx.x * kPer + j) * 32 + __ffs(b) - 1;
    __syncthreads();
    return total;
}

// What bounds a pass: the first group or two, which reach most nodes -- the
// chain of L2 reads per arc, one row of W words each -- and for the rest the
// grid barriers of the groups (five or more each), since most nodes are
// saturated by then and almost all sources useless.  Directed R-MAT 18 kept
// whole, k = 64, 262,144 nodes:
// - a group takes the next 64 W *useful* sources of the order, however far
//   apart: 21.5 -> 7.2 ms;
// - W lanes carry one arc's words (a coalesced row instead of W reads a lane),
//   long rows are queued in parts so that no warp and no round of the grid
//   waits for a hub, and the queues are appended to once a warp: 7.2 -> 1.7
//   ms (reading nxt as well, to save the atomics of bits that another arc
//   brought, cost 3 %);
// - the window of positions tested follows the density of useful sources, so
//   that a late group sweeps most of what is left: 12 groups -> 4.
template <bool LEN>
__global__ void __launch_bounds__(kRT, 4) k_reach(ReachJob J, RState *rs)
{
    constexpr unsigned FULL = 0xFFFFFFFFu;
    const unsigned nb = gridDim.x;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t nthr = (int64_t)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    const int64_t gw = tid >> 5, nwarps = nthr >> 5;
    const int W = J.W, G = 64 * W;
    // lane groups of W lanes: one node's words
    const int gq = lane & (W - 1), g0 = lane & ~(W - 1), NPW = 32 / W;
    const unsigned gm = ((1u << W) - 1u) << g0;
    volatile unsigned *qlen = rs->qlen, *blen = rs->blen, *tlen = rs->tlen;
    __shared__ int s_src[64 * kReachMaxW];
    __shared__ int32_t s_arc[kRT / 32][32];
    int32_t *const arcs = s_arc[threadIdx.x >> 5];
    const int64_t plane = J.n * W;
    unsigned epoch = 0;
    int wpar = 0, par = 0, zeroed = 0;
    int64_t win = 2 * G, next = 0;
    // Append the node of every lane with `want`: all lanes of the warp call.
    auto degree = [&](int32_t v) { return J.rp[v + 1] - J.rp[v]; };
    auto push = [&](int which, int32_t v, int64_t deg, bool want) {
        const unsigned small = __ballot_sync(FULL, want && deg <= kReachBigDeg);
        if (small) {
            unsigned at = 0;
            if (lane == 0) at = atomicAdd((unsigned *)&qlen[which], __popc(small));
            at = __shfl_sync(FULL, at, 0) + __popc(small & ((1u << lane) - 1u));
            if (small >> lane & 1u) J.Q[which][at] = v;
        }
        if (want && deg > kReachBigDeg) {
            const unsigned parts = (unsigned)((deg + kReachBigDeg - 1) / kReachBigDeg);
            const unsigned at = atomicAdd((unsigned *)&blen[which], parts);
            for (unsigned p = 0; p < parts; ++p)
                J.QB[which][at + p] = (uint64_t)p << 32 | (uint32_t)v;
        }
    };
    for (int64_t pos = 0; pos < J.n; pos = next, wpar ^= 1) {
        const int64_t hi = pos + win < J.n ? pos + win : J.n;
        const uint32_t base = (uint32_t)pos;
        mark_useful(J, pos, hi, rs->flags[wpar], gw, nwarps, lane);
        if (!grid_sync(J.ctl, blockIdx.x, nb, J.timeout_ns)) return;
        const int found = pick_sources(rs->flags[wpar], hi - pos, G, s_src);
        const int gs = found < G ? found : G;
        next = found > G ? pos + s_src[G - 1] + 1 : hi;
        // the next window, in whole words: what this group consumed, times
        // more the fewer of its sources were useful
        win = (next - pos) * (4 * found >= G ? 2 : 16 * found >= G ? 4 : 16);
        win = win < 2 * G ? 2 * G : win > kMaxWin ? kMaxWin : (win + 31) & ~31ll;
        if (gs == 0) continue;
        int cur = 0;
        // sources of the group (distinct nodes: one thread each)
        for (int64_t i0 = gw * 32; i0 < gs; i0 += nwarps * 32) {
            const int64_t i = i0 + lane;
            const bool ok = i < gs;
            const int32_t s = ok ? J.order[pos + s_src[i]] : 0;
            if (ok) {
                const uint64_t bit = 1ull << (i & 63);
                J.vis[(int64_t)s * W + (i >> 6)] = bit;
                J.F[(int64_t)s * W + (i >> 6)] = bit;
                if (LEN) J.lev[(int64_t)s * G + i] = 0;
                J.TL[i] = s;
            }
            push(0, s, degree(s), ok);
        }
        if (tid == 0) tlen[par] = (unsigned)gs;
        if (!grid_sync(J.ctl, blockIdx.x, nb, J.timeout_ns)) return;
        uint32_t level = 0;
        for (;;) {
            const unsigned qn = qlen[cur], bn = blen[cur];
            if (qn + bn == 0) break;
            ++level;
            ++epoch;
            const int nxq = cur ^ 1;
            // a plane this level is the first of the call to write (after the
            // barrier below)
            if (!LEN && zeroed < kReachPlanes && level >> zeroed) {
                for (int64_t i = tid; i < plane; i += nthr) J.planes[zeroed * plane + i] = 0;
                ++zeroed;
            }
            // Expand arcs [lo, end) of node u in steps (all lanes together).
            auto expand = [&](int32_t u, int64_t lo, int64_t end, int64_t step) {
                const uint64_t Fw = J.F[(int64_t)u * W + gq];
                const unsigned words = LEN ? __ballot_sync(FULL, Fw != 0 && lane < W) : 0;
                for (int64_t e0 = lo; e0 < end; e0 += step) {
                    const int64_t e = e0 + lane;
                    int32_t w = -1;
                    if (e < end) {
                        w = J.col[e];
                        if (saturated(J, w, base)) w = -1;
                    }
                    const unsigned act = __ballot_sync(FULL, w >= 0);
                    if (!act) continue;
                    if (LEN) {
                        // a lane per arc: relax every changed source of u into w
                        bool any = false;
                        const uint64_t len = w >= 0 ? J.w[e] : 0;
                        for (unsigned m = words; m; m &= m - 1) {
                            const int q = __ffs(m) - 1;
                            const uint64_t fq = __shfl_sync(FULL, Fw, q);
                            if (w < 0) continue;
                            uint64_t nbits = 0;
                            for (uint64_t x = fq; x; x &= x - 1) {
                                const int i = q * 64 + (__ffsll((long long)x) - 1);
                                const uint64_t cand =
                                    (uint64_t)__ldcg(&J.lev[(int64_t)u * G + i]) + len;
                                if (cand >= (uint64_t)kInf) continue;
                                const uint32_t old =
                                    atomicMin(&J.lev[(int64_t)w * G + i], (uint32_t)cand);
                                if (cand < old) nbits |= 1ull << (i & 63);
                            }
                            if (nbits) {
                                atomicOr((unsigned long long *)&J.nxt[(int64_t)w * W + q],
                                         (unsigned long long)nbits);
                                any = true;
                            }
                        }
                        push(nxq, w, w >= 0 ? degree(w) : 0,
                             any && atomicExch(&J.qstamp[w], epoch) != epoch);
                        continue;
                    }
                    // W lanes per arc, over the unsaturated targets
                    const int na = __popc(act);
                    __syncwarp();
                    if (w >= 0) arcs[__popc(act & ((1u << lane) - 1u))] = w;
                    __syncwarp();
                    int a0 = 0;
                    // U rows of words in flight per lane group
                    auto round = [&](auto rows) {
                        constexpr int U = decltype(rows)::value;
                        int32_t t[U];
                        uint64_t have[U];
#pragma unroll
                        for (int q = 0; q < U; ++q) {
                            const int i = a0 + q * NPW + lane / W;
                            t[q] = i < na ? arcs[i] : -1;
                            have[q] = ~0ull;
                        }
#pragma unroll
                        for (int q = 0; q < U; ++q)
                            if (t[q] >= 0 && Fw) have[q] = J.vis[(int64_t)t[q] * W + gq];
                        // step q's touched nodes go to the lanes gq == q (32
                        // arcs are at most W steps)
                        int32_t got = -1;
#pragma unroll
                        for (int q = 0; q < U; ++q) {
                            const uint64_t nbits = Fw & ~have[q];
                            if (nbits)
                                atomicOr((unsigned long long *)&J.nxt[(int64_t)t[q] * W + gq],
                                         (unsigned long long)nbits);
                            const unsigned m = __ballot_sync(FULL, nbits != 0);
                            if (gq == q && (m & gm)) got = t[q];
                        }
                        a0 += U * NPW;
                        if (!__any_sync(FULL, got >= 0)) return;
                        const int64_t deg = got >= 0 ? degree(got) : 0;
                        push(nxq, got, deg,
                             got >= 0 && atomicExch(&J.qstamp[got], epoch) != epoch);
                    };
                    // (steps without arcs are not free: short rows at eight
                    // took a directed grid from 33 to 38 ms, and skipping each
                    // of the eight by a branch R-MAT 18 from 1.72 to 1.93)
                    while (a0 < na) {
                        if (na - a0 <= NPW) round(std::integral_constant<int, 1>());
                        else if (na - a0 <= 4 * NPW) round(std::integral_constant<int, 4>());
                        else round(std::integral_constant<int, 8>());
                    }
                }
            };
            // A warp per small node or part of a big row, or several warps
            // each while there are fewer of them than warps.
            const unsigned items = qn + bn;
            const unsigned fit = (unsigned)nwarps / items;
            const unsigned S = fit < 1 ? 1 : fit > kReachBigDeg / 32 ? kReachBigDeg / 32 : fit;
            for (int64_t i = gw; i < (int64_t)items * S; i += nwarps) {
                const unsigned it = S > 1 ? (unsigned)i % items : (unsigned)i;
                const unsigned sl = S > 1 ? (unsigned)i / items : 0;
                int32_t u;
                int64_t lo, end;
                if (it < bn) {
                    const uint64_t x = J.QB[cur][it];
                    u = (int32_t)(uint32_t)x;
                    lo = J.rp[u] + (int64_t)(x >> 32) * kReachBigDeg;
                    end = J.rp[u + 1];
                    end = end < lo + kReachBigDeg ? end : lo + kReachBigDeg;
                } else {
                    u = J.Q[cur][it - bn];
                    lo = J.rp[u];
                    end = J.rp[u + 1];
                }
                expand(u, lo + sl * 32, end, S * 32);
            }
            if (!grid_sync(J.ctl, blockIdx.x, nb, J.timeout_ns)) return;
            // the next frontier: new bits (with arc lengths: the sources whose
            // distance dropped), their levels, first touches; W lanes a node
            const int64_t qn2 = qlen[nxq], all2 = qn2 + blen[nxq];
            for (int64_t i0 = gw * NPW; i0 < all2; i0 += nwarps * NPW) {
                const int64_t i = i0 + lane / W;
                bool ok = i < all2;
                int32_t w = 0;
                if (ok && i < qn2) {
                    w = J.Q[nxq][i];
                } else if (ok) {
                    const uint64_t x = J.QB[nxq][i - qn2];
                    w = (int32_t)(uint32_t)x;
                    ok = x >> 32 == 0;  // once, not for every part of the row
                }
                const int64_t at = (int64_t)w * W + gq;
                const uint64_t old = ok ? J.vis[at] : 0, nx = ok ? J.nxt[at] : 0;
                const uint64_t nbits = LEN ? nx : nx & ~old;
                const unsigned seen = __ballot_sync(FULL, old != 0) & gm;
                const unsigned f = __ballot_sync(FULL, ok && !seen && gq == 0);
                if (f) {
                    unsigned to = 0;
                    if (lane == 0) to = atomicAdd((unsigned *)&tlen[par], __popc(f));
                    to = __shfl_sync(FULL, to, 0) + __popc(f & ((1u << lane) - 1u));
                    if (f >> lane & 1u) J.TL[to] = w;
                }
                if (!ok) continue;
                if (nx) J.nxt[at] = 0;
                if (nbits & ~old) J.vis[at] = old | nbits;
                J.F[at] = nbits;
                if (!LEN && level >= 1u << kReachPlanes)
                    for (uint64_t x = nbits; x; x &= x - 1)
                        J.lev[(int64_t)w * G + gq * 64 + (__ffsll((long long)x) - 1)] = level;
                else if (!LEN && nbits)
                    for (uint32_t l = level; l; l &= l - 1)
                        atomicOr((unsigned long long *)&J.planes[(__ffs((int)l) - 1) * plane + at],
                                 (unsigned long long)nbits);
            }
            if (tid == 0) {
                qlen[cur] = 0;
                blen[cur] = 0;
                rs->levels += 1;
            }
            cur = nxq;
            if (!grid_sync(J.ctl, blockIdx.x, nb, J.timeout_ns)) return;
        }
        // acceptance: each touched node takes its lowest-rank bits, W lanes a
        // node, a lane a word
        const unsigned tn = tlen[par];
        for (int64_t i0 = gw * NPW; i0 < tn; i0 += nwarps * NPW) {
            const int64_t i = i0 + lane / W;
            const bool ok = i < tn;
            const int32_t v = ok ? J.TL[i] : 0;
            const int64_t at = (int64_t)v * W + gq;
            const int64_t rv = J.rank[v];
            const int c0 = J.cnt[v];
            const uint64_t reached = ok ? J.vis[at] : 0;
            uint64_t bits = reached;
            if (ok && rv >= pos && rv < next) {  // its own search, if it ran
                int lo = 0, up = gs;
                while (lo < up) {
                    const int mid = (lo + up) >> 1;
                    if (s_src[mid] < (int)(rv - pos)) lo = mid + 1;
                    else up = mid;
                }
                if (lo < gs && s_src[lo] == (int)(rv - pos) && (lo >> 6) == gq)
                    bits &= ~(1ull << (lo & 63));
            }
            const int pc = __popcll(bits);
            int incl = pc;
            for (int o = 1; o < W; o <<= 1) {
                const int y = __shfl_up_sync(FULL, incl, o, W);
                if (gq >= o) incl += y;
            }
            const int first = c0 + incl - pc;  // samples before this word's
            const int total = c0 + __shfl_sync(FULL, incl, g0 + W - 1);
            int take = J.k - first;
            take = take < 0 ? 0 : take > pc ? pc : take;
            uint64_t rest = bits;
            for (int a = 0; a < take; ++a) rest &= rest - 1;
            const uint64_t acc = bits ^ rest;  // the lowest `take` bits
            if (take > 0 && first + take == J.k) {
                const int64_t p = pos + s_src[gq * 64 + 63 - __clzll((long long)acc)];
                J.T[v] = rv < p ? p : p + 1;  // 1-based, v not counted
            }
            unsigned long long ds = 0;
            uint64_t one = acc;  // levels read one by one
            if (!LEN && reached) {
                uint64_t pl[kReachPlanes];
#pragma unroll
                for (int p = 0; p < kReachPlanes; ++p)
                    pl[p] = level >> p ? J.planes[p * plane + at] : 0;
#pragma unroll
                for (int p = 0; p < kReachPlanes; ++p) {
                    ds += (unsigned long long)__popcll(acc & pl[p]) << p;
                    one &= ~pl[p];
                    if (pl[p]) J.planes[p * plane + at] = 0;
                }
            }
            for (uint64_t x = one; x; x &= x - 1)
                ds += __ldcg(&J.lev[(int64_t)v * G + gq * 64 + (__ffsll((long long)x) - 1)]);
            for (int o = 1; o < W; o <<= 1) ds += __shfl_xor_sync(FULL, ds, o);
            if (!ok) continue;
            if (reached) J.vis[at] = 0;
            J.F[at] = 0;
            if (LEN)  // tentative distances start at infinity in every group
                for (uint64_t y = reached; y; y &= y - 1)
                    J.lev[(int64_t)v * G + gq * 64 + (__ffsll((long long)y) - 1)] = kInf;
            if (gq == 0) {
                const int c = total < J.k ? total : J.k;
                J.cnt[v] = c;
                J.dsum[v] += ds;
                // a (k+1)-th source reached it: saturated from now on; k: once
                // its own position is past
                if (c == J.k) J.satpos[v] = total > J.k ? 0u : (uint32_t)rv + 1u;
            }
        }
        if (tid == 0) {
            tlen[par ^ 1] = 0;  // the next group's touched list
            rs->groups += 1;
        }
        if (!grid_sync(J.ctl, blockIdx.x, nb, J.timeout_ns)) return;
        par ^= 1;
    }
}

__global__ void k_rank_of(const uint32_t *order, int64_t n, int32_t *order32, int32_t *rank)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t v = order[p];
        order32[p] = (int32_t)v;
        rank[v] = (int32_t)p;
    }
}

__global__ void k_reach_final(int64_t n, int k, const int32_t *cnt, const uint64_t *dsum,
                              const int64_t *T, double *avg, double *rhat)
{
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int c = cnt[v];
        if (avg) avg[v] = c ? (double)dsum[v] / (double)c : 0.0;
        if (rhat) {
            double r = (double)c;
            if (c >= k)
                r = k == 1 ? 1.0
                           : 1.0 + (double)((uint64_t)(k - 1) * (uint64_t)(n - 2)) /
                                       (double)(T[v] - 1);
            rhat[v] = r;
        }
    }
}

int grid_of(int64_t n)
{
    return (int)std::min<int64_t>(std::max<int64_t>(1, (n + 255) / 256), 152 * 16);
}

#define R_CK(x)                                  \
    do {                                         \
        const cudaError_t e_ = (x);              \
        if (e_ != cudaSuccess) {                 \
            note_cuda_error(e_, __FILE__, __LINE__); \
            cudaGetLastError();                  \
            return CC_ERR_CUDA;                  \
        }                                        \
    } while (0)
#define R_RC(x)                      \
    do {                             \
        int r_ = (x);                \
        if (r_ != CC_OK) return r_;  \
    } while (0)

}  // namespace

int reach_order(int64_t n, uint64_t seed, uint64_t *keys, uint32_t *vals, uint64_t *tk,
                uint32_t *tv, int32_t *order, int32_t *rank, cudaStream_t st)
{
    bool in_tmp = false;
    R_RC(random_order(n, seed, keys, vals, tk, tv, &in_tmp, st));
    k_rank_of<<<grid_of(n), 256, 0, st>>>(in_tmp ? tv : vals, n, order, rank);
    R_CK(cudaGetLastError());
    return CC_OK;
}

int reach_run(const ReachJob &job, cudaStream_t st, ReachStats *stats)
{
    int dev = 0, sms = 0, per = 0;
    const void *kernel = job.w ? (const void *)k_reach<true> : (const void *)k_reach<false>;
    R_CK(cudaGetDevice(&dev));
    R_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    R_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, kRT, 0));
    if (per < 1) return CC_ERR_CUDA;
    int grid = sms * std::min(per, 4);
    RState *rs = nullptr;
    R_CK(cudaMallocAsync((void **)&rs, sizeof(RState), st));
    int rc = CC_OK;
    if (cudaMemsetAsync(rs, 0, sizeof(RState), st) != cudaSuccess ||
        cudaMemsetAsync(job.ctl, 0, sizeof(Ctl), st) != cudaSuccess) {
        rc = CC_ERR_CUDA;
    } else {
        ReachJob j = job;
        void *args[] = {(void *)&j, (void *)&rs};
        if (cudaLaunchCooperativeKernel(kernel, grid, kRT, args, 0, st) !=
            cudaSuccess)
            rc = CC_ERR_CUDA;
    }
    unsigned long long h[2] = {0, 0};  // levels, groups
    Ctl c{};
    if (rc == CC_OK && (cudaMemcpyAsync(h, &rs->levels, sizeof(h), cudaMemcpyDeviceToHost, st) !=
                            cudaSuccess ||
                        cudaMemcpyAsync(&c, job.ctl, sizeof(c), cudaMemcpyDeviceToHost, st) !=
                            cudaSuccess ||
                        cudaStreamSynchronize(st) != cudaSuccess))
        rc = CC_ERR_CUDA;
    cudaFreeAsync(rs, st);
    if (rc != CC_OK) {
        cudaGetLastError();
        return rc;
    }
    if (stats) {
        stats->levels = (int64_t)h[0];
        stats->groups = (int64_t)h[1];
        stats->grid = grid;
    }
    return c.err < 0 ? c.err : CC_OK;
}

void reach_finalize(int64_t n, int k, const int32_t *cnt, const uint64_t *dsum,
                    const int64_t *T, double *avg, double *rhat, cudaStream_t st)
{
    k_reach_final<<<grid_of(n), 256, 0, st>>>(n, k, cnt, dsum, T, avg, rhat);
}

}  // namespace ccg
