// Outbound / inbound estimates of general directed graphs (section 6.2,
// Algorithm 4): for every node v, the k nodes of smallest rank (a seeded
// random order) among those v reaches (outbound) or that reach v (inbound),
// their distances, and the rank position of the k-th.
//
// One persistent cooperative launch walks the order in groups of 64 W
// sources whose search can still reach a node that takes samples.  Each group is a bit-packed multi-source BFS on the search graph
// (G^T for outbound, G for inbound: bit i leaves the group's i-th source),
// recording the level at which each bit first reaches each node; then every
// node it touched accepts its lowest-rank bits (its own excluded) until it
// holds k samples.  Bits are ranks, so the accepted ones are exactly the
// next samples in rank order.
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

#include "barrier.cuh"
#include "nodew.h"
#include "reach.h"

namespace ccg {

namespace {

constexpr int kRT = 256;
// Positions of the order tested for useful sources at once.
constexpr int kMaxWin = 32768;
// Arcs beyond which a source is taken without a proof that it is useful.
constexpr int kTestArcs = 4096;

struct RState {
    unsigned qlen[2], blen[2];  // frontier queue: small nodes, big ones
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
            for (int64_t y = bb; y < ee && !any; y += 128) {
                int32_t c[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    c[q] = y + lane + 32 * q < ee ? J.col[y + lane + 32 * q] : -1;
                bool f = false;
#pragma unroll
                for (int q = 0; q < 4; ++q) f |= c[q] >= 0 && !saturated(J, c[q], base);
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

// What bounds a pass: the grid barriers of its groups (five or more each)
// and, after the first few groups, nothing else -- most nodes are saturated,
// and of 512 consecutive sources almost all are useless.  So a group takes
// the next 64 W *useful* sources of the order, however far apart (directed
// R-MAT 18 kept whole, k = 64, 262,144 nodes: 21.5 -> 8.0 ms).
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
    const unsigned gm = W == 32 ? FULL : ((1u << W) - 1u) << g0;
    volatile unsigned *qlen = rs->qlen, *blen = rs->blen, *tlen = rs->tlen;
    __shared__ int s_src[64 * kReachMaxW];
    unsigned epoch = 0;
    int wpar = 0, par = 0;
    int64_t win = 2 * G, next = 0;
    auto queue = [&](int which, int32_t v) {
        if (J.rp[v + 1] - J.rp[v] > kReachBigDeg)
            J.QB[which][atomicAdd((unsigned *)&blen[which], 1u)] = v;
        else
            J.Q[which][atomicAdd((unsigned *)&qlen[which], 1u)] = v;
    };
    for (int64_t pos = 0; pos < J.n; pos = next, wpar ^= 1) {
        const int64_t hi = pos + win < J.n ? pos + win : J.n;
        const uint32_t base = (uint32_t)pos;
        mark_useful(J, pos, hi, rs->flags[wpar], gw, nwarps, lane);
        if (!grid_sync(J.ctl, blockIdx.x, nb, J.timeout_ns)) return;
        const int found = pick_sources(rs->flags[wpar], hi - pos, G, s_src);
        const int gs = found < G ? found : G;
        next = found > G ? pos + s_src[G - 1] + 1 : hi;
        // the next window: twice what this group consumed, in whole words
        win = ((2 * (next - pos) + 31) & ~31ll);
        win = win < 2 * G ? 2 * G : win > kMaxWin ? kMaxWin : win;
        if (gs == 0) continue;
        int cur = 0;
        // sources of the group (distinct nodes: one thread each)
        for (int64_t i = tid; i < gs; i += nthr) {
            const int32_t s = J.order[pos + s_src[i]];
            const uint64_t bit = 1ull << (i & 63);
            J.vis[(int64_t)s * W + (i >> 6)] = bit;
            J.F[(int64_t)s * W + (i >> 6)] = bit;
            J.lev[(int64_t)s * G + i] = 0;
            queue(0, s);
            J.TL[i] = s;
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
            // Expand arcs x0, x0 + step, ... of node u, a lane per arc (all
            // lanes of the warp together).
            auto expand = [&](int32_t u, int64_t x0, int64_t step) {
                const uint64_t Fw = lane < W ? J.F[(int64_t)u * W + lane] : 0;
                const unsigned words = __ballot_sync(FULL, Fw != 0);
                const int64_t end = J.rp[u + 1];
                for (int64_t e0 = J.rp[u] + x0; e0 < end; e0 += step) {
                    const int64_t e = e0 + lane;
                    int32_t w = 0;
                    bool ok = e < end;
                    if (ok) {
                        w = J.col[e];
                        ok = !saturated(J, w, base);
                    }
                    if (!__any_sync(FULL, ok)) continue;
                    bool any = false;
                    const uint64_t len = J.w && ok ? J.w[e] : 0;
                    for (unsigned m = words; m; m &= m - 1) {
                        const int q = __ffs(m) - 1;
                        const uint64_t fq = __shfl_sync(FULL, Fw, q);
                        if (!ok) continue;
                        uint64_t nbits = 0;
                        if (J.w) {
                            // arc lengths: relax every changed source of u into w
                            for (uint64_t x = fq; x; x &= x - 1) {
                                const int i = q * 64 + (__ffsll((long long)x) - 1);
                                const uint64_t cand =
                                    (uint64_t)__ldcg(&J.lev[(int64_t)u * G + i]) + len;
                                if (cand >= (uint64_t)kInf) continue;
                                const uint32_t old =
                                    atomicMin(&J.lev[(int64_t)w * G + i], (uint32_t)cand);
                                if (cand < old) nbits |= 1ull << (i & 63);
                            }
                        } else {
                            nbits = fq & ~J.vis[(int64_t)w * W + q];
                        }
                        if (nbits) {
                            atomicOr((unsigned long long *)&J.nxt[(int64_t)w * W + q],
                                     (unsigned long long)nbits);
                            any = true;
                        }
                    }
                    if (any && atomicExch(&J.qstamp[w], epoch) != epoch) queue(nxq, w);
                }
            };
            // Small nodes: a warp each, or several warps each while there
            // are fewer nodes than warps.
            const int64_t S = qn > 0 && qn < nwarps ? nwarps / qn : 1;
            for (int64_t i = gw; i < (int64_t)qn * S; i += nwarps)
                expand(J.Q[cur][i % qn], i / qn * 32, S * 32);
            for (unsigned i = 0; i < bn; ++i) expand(J.QB[cur][i], gw * 32, nwarps * 32);
            if (!grid_sync(J.ctl, blockIdx.x, nb, J.timeout_ns)) return;
            // the next frontier: new bits (with arc lengths: the sources whose
            // distance dropped), their levels, first touches; W lanes a node
            const int64_t qn2 = qlen[nxq], all2 = qn2 + blen[nxq];
            for (int64_t i0 = gw * NPW; i0 < all2; i0 += nwarps * NPW) {
                const int64_t i = i0 + lane / W;
                const bool ok = i < all2;
                const int32_t w = ok ? (i < qn2 ? J.Q[nxq][i] : J.QB[nxq][i - qn2]) : 0;
                const int64_t at = (int64_t)w * W + gq;
                const uint64_t old = ok ? J.vis[at] : 0, nx = ok ? J.nxt[at] : 0;
                const uint64_t nbits = J.w ? nx : nx & ~old;
                const bool fresh = (__ballot_sync(FULL, old != 0) & gm) == 0;
                if (!ok) continue;
                if (nx) J.nxt[at] = 0;
                if (nbits & ~old) J.vis[at] = old | nbits;
                J.F[at] = nbits;
                if (!J.w)
                    for (uint64_t x = nbits; x; x &= x - 1)
                        J.lev[(int64_t)w * G + gq * 64 + (__ffsll((long long)x) - 1)] = level;
                if (fresh && gq == 0) J.TL[atomicAdd((unsigned *)&tlen[par], 1u)] = w;
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
            unsigned long long ds = 0;
            uint64_t x = bits;
            for (int a = 0; a < take; ++a, x &= x - 1) {
                const int bit = gq * 64 + (__ffsll((long long)x) - 1);
                ds += __ldcg(&J.lev[(int64_t)v * G + bit]);
                if (first + a + 1 == J.k) {
                    const int64_t p = pos + s_src[bit];
                    J.T[v] = rv < p ? p : p + 1;  // 1-based, v not counted
                }
            }
            for (int o = 1; o < W; o <<= 1) ds += __shfl_xor_sync(FULL, ds, o);
            if (!ok) continue;
            if (reached) J.vis[at] = 0;
            J.F[at] = 0;
            if (J.w)  // tentative distances start at infinity in every group
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
    R_CK(cudaGetDevice(&dev));
    R_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    R_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_reach, kRT, 0));
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
        if (cudaLaunchCooperativeKernel((const void *)k_reach, grid, kRT, args, 0, st) !=
            cudaSuccess)
            rc = CC_ERR_CUDA;
    }
    RState h{};
    Ctl c{};
    if (rc == CC_OK && (cudaMemcpyAsync(&h, rs, sizeof(h), cudaMemcpyDeviceToHost, st) !=
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
        stats->levels = (int64_t)h.levels;
        stats->groups = (int64_t)h.groups;
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
