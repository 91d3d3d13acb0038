// Shortest paths from k sources on graphs of narrow frontiers (grids, road
// networks: rows of few entries, thousands of hops across), tile by tile.
//
// A level-synchronous search pays its grid barriers and a chain of dependent
// memory accesses per level -- about 15 us of a level on a GB300 whatever the
// frontier holds, thousands of times.  Here the nodes are cut once into tiles
// of up to 512 neighbouring ones, and a round takes every (tile, source) pair
// whose labels were lowered from outside: a warp loads the source's labels of
// the tile into shared memory, corrects labels there until none drops
// (shared-memory latency in place of the L2's, no barrier), writes back what
// dropped and lowers the labels across the tile's border, which makes those
// pairs the next round's.  A round moves every search front on by a tile, so
// the grid barrier is passed once per ~20 hops.  Labels only fall and every
// drop is carried on, so the labels end at the exact distances, with unit or
// 32-bit arc lengths, whatever the order (sections 3 and 7: the distances of
// k Dijkstra or breadth-first searches).
//
// Every wait is the bounded grid barrier (CC_ERR_TIMEOUT on expiry).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "barrier.cuh"
#include "graph_gpu.h"
#include "per_device.h"
#include "tiles.h"

namespace ccg {

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int kT = 256;
constexpr uint16_t kNoArc = 0xFFFF, kLongRow = 0xFFFE;
// Breadth-first growth of the clusters: hops per pass, passes.
constexpr int kGrowHops = 32;
constexpr int kGrowPasses = 8;
// Graphs are taken when at most a fifth of the arcs leave their tile and a
// tile has at most ten neighbouring ones on average: a grid has 7 % and
// about 6, a graph with a few random long links has a hundred, and its
// labels would be lowered over and over through them.
constexpr double kMaxCut = 0.2, kMaxNeighbours = 10.0;

int grid_of(int64_t n)
{
    return (int)std::min<int64_t>(std::max<int64_t>(1, (n + kT - 1) / kT), 152 * 16);
}

#define T_CK(x)                                      \
    do {                                             \
        const cudaError_t e_ = (x);                  \
        if (e_ != cudaSuccess) {                     \
            note_cuda_error(e_, __FILE__, __LINE__); \
            cudaGetLastError();                      \
            return CC_ERR_CUDA;                      \
        }                                            \
    } while (0)
#define T_RC(x)                     \
    do {                            \
        int r_ = (x);               \
        if (r_ != CC_OK) return r_; \
    } while (0)
#define STRIDED(i, n)                                                                   \
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (n);               \
    i += (int64_t)gridDim.x * blockDim.x

struct Buf {
    void *p = nullptr;
    Buf() = default;
    Buf(const Buf &) = delete;
    Buf &operator=(const Buf &) = delete;
    ~Buf() { if (p) cudaFree(p); }
    int alloc(size_t bytes)
    {
        if (cudaMalloc(&p, bytes ? bytes : 16) == cudaSuccess) return CC_OK;
        cudaGetLastError();
        p = nullptr;
        return CC_ERR_OOM;
    }
    template <class T> T *as() const { return static_cast<T *>(p); }
    template <class T> T *take()
    {
        T *t = static_cast<T *>(p);
        p = nullptr;
        return t;
    }
};

// ---- cutting the graph ----------------------------------------------------

// Clusters: unlabelled nodes picked at random (one in half a tile's capacity) and the
// nodes nearest to them in hops (ties to the smallest centre), pass by pass.
// stamp = the step a node was labelled at (kInf: not yet); a step only reads
// labels of earlier steps, so the result does not depend on timing.
__global__ void k_centres(int64_t n, unsigned mean, uint64_t seed, uint32_t step, int32_t *lab,
                          uint32_t *stamp)
{
    for (STRIDED(v, n))
        if (stamp[v] == kInf && splitmix64_out(seed, (uint64_t)v) < ~0ull / mean) {
            lab[v] = (int32_t)v;
            stamp[v] = step;
        }
}

__global__ void k_grow(int64_t n, const int64_t *rp, const int32_t *col, uint32_t step,
                       int32_t *lab, uint32_t *stamp, unsigned *left)
{
    unsigned open = 0;
    for (STRIDED(v, n)) {
        if (stamp[v] != kInf) continue;
        int32_t best = 0x7FFFFFFF;
        for (int64_t e = rp[v]; e < rp[v + 1]; ++e) {
            const int32_t u = col[e];
            if (stamp[u] < step) best = min(best, lab[u]);
        }
        if (best != 0x7FFFFFFF) {
            lab[v] = best;
            stamp[v] = step;
        } else {
            open += 1;
        }
    }
    if (left && open) atomicAdd(left, open);
}

// Sort keys; nodes no centre reached keep their neighbourhood in id order.
// hops += the nodes' hops to their centres.
__global__ void k_keys(int64_t n, const int32_t *lab, const uint32_t *stamp, uint64_t *keys,
                       uint32_t *vals, unsigned long long *hops)
{
    unsigned long long h = 0;
    for (STRIDED(v, n)) {
        const uint32_t s = stamp[v];
        keys[v] = s != kInf ? (uint64_t)lab[v] : (uint64_t)(v & ~255ll);
        vals[v] = (uint32_t)v;
        h += s != kInf ? s % (kGrowHops + 1) : kGrowHops;
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) h += __shfl_xor_sync(FULL, h, o);
    if ((threadIdx.x & 31) == 0 && h) atomicAdd(hops, h);
}

__global__ void k_cluster_starts(int64_t n, const uint64_t *keys, uint64_t *flag)
{
    for (STRIDED(i, n)) flag[i] = i == 0 || keys[i] != keys[i - 1];
}

// first[c] = sorted position of cluster c's first node (idx: exclusive scan
// of the start flags).
__global__ void k_cluster_first(int64_t n, const uint64_t *keys, const uint64_t *idx,
                                int32_t *first)
{
    for (STRIDED(i, n))
        if (i == 0 || keys[i] != keys[i - 1]) first[idx[i]] = (int32_t)i;
}

// A cluster of more than a tile's capacity is chopped into tiles of that many.
__global__ void k_tile_starts(int64_t n, const uint64_t *keys, const uint64_t *idx,
                              const int32_t *first, int cap, uint64_t *flag)
{
    for (STRIDED(i, n)) {
        const bool head = i == 0 || keys[i] != keys[i - 1];
        const int64_t c = (int64_t)idx[i] - (head ? 0 : 1);
        flag[i] = (i - first[c]) % cap == 0;
    }
}

__global__ void k_tile_first(int64_t n, const uint64_t *flag, const uint64_t *tidx, int32_t *tfirst,
                             int64_t tiles)
{
    for (STRIDED(i, n))
        if (flag[i]) tfirst[tidx[i]] = (int32_t)i;
    if (blockIdx.x == 0 && threadIdx.x == 0) tfirst[tiles] = (int32_t)n;
}

__global__ void k_tile_words(int64_t tiles, const int32_t *tfirst, uint64_t *words)
{
    for (STRIDED(t, tiles)) words[t] = (uint64_t)(tfirst[t + 1] - tfirst[t] + 31) / 32;
}

__global__ void k_tile_slots(int64_t tiles, const int32_t *tfirst, const uint64_t *wstart,
                             const uint32_t *sorted, int64_t words, int32_t *tb,
                             int32_t *word_tile, int32_t *perm, int32_t *iperm)
{
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int32_t b = tfirst[t], sz = tfirst[t + 1] - b, s0 = (int32_t)wstart[t] * 32;
        const int nw = (sz + 31) / 32;
        if (threadIdx.x == 0) tb[t] = s0;
        for (int i = threadIdx.x; i < nw; i += blockDim.x) word_tile[wstart[t] + i] = (int32_t)t;
        for (int i = threadIdx.x; i < nw * 32; i += blockDim.x) {
            const int32_t v = i < sz ? (int32_t)sorted[b + i] : -1;
            perm[s0 + i] = v;
            if (v >= 0) iperm[v] = s0 + i;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) tb[tiles] = (int32_t)words * 32;
}

// Arcs inside and leaving the tile per slot (entry `slots` stays 0).
__global__ void k_tile_degrees(int64_t slots, const int32_t *perm, const int32_t *iperm,
                               const int32_t *word_tile, const int64_t *rp, const int32_t *col,
                               uint64_t *in, uint64_t *ex)
{
    for (STRIDED(s, slots + 1)) {
        const int32_t v = s < slots ? perm[s] : -1;
        unsigned a = 0, b = 0;
        if (v >= 0)
            for (int64_t e = rp[v]; e < rp[v + 1]; ++e) {
                if (word_tile[iperm[col[e]] >> 5] == word_tile[s >> 5]) ++a;
                else ++b;
            }
        in[s] = a;
        ex[s] = b;
    }
}

__global__ void k_tile_arcs(int64_t slots, const int32_t *perm, const int32_t *iperm,
                            const int32_t *word_tile, const int32_t *tb, const int64_t *rp,
                            const int32_t *col, const uint32_t *w, const uint64_t *ioff,
                            const uint64_t *eoff, uint32_t *irp, uint32_t *erp, uint16_t *icol,
                            int32_t *ecol, uint16_t *etail, uint32_t *iw, uint32_t *ew,
                            ushort4 *icol4, uint4 *iw4)
{
    for (STRIDED(s, slots + 1)) {
        uint32_t a = (uint32_t)ioff[s], b = (uint32_t)eoff[s];
        irp[s] = a;
        erp[s] = b;
        if (s == slots) continue;
        const int32_t v = perm[s], t = word_tile[s >> 5];
        uint16_t c[4] = {kNoArc, kNoArc, kNoArc, kNoArc};
        uint32_t l[4] = {0u, 0u, 0u, 0u};
        int m = 0;
        for (int64_t e = v < 0 ? 0 : rp[v], end = v < 0 ? 0 : rp[v + 1]; e < end; ++e) {
            const int32_t h = iperm[col[e]];
            if (word_tile[h >> 5] == t) {
                icol[a] = (uint16_t)(h - tb[t]);
                if (w) iw[a] = w[e];
                if (m < 4) {
                    c[m] = (uint16_t)(h - tb[t]);
                    l[m] = w ? w[e] : 1u;
                }
                ++m;
                ++a;
            } else {
                ecol[b] = h;
                etail[b] = (uint16_t)(s - tb[t]);
                if (w) ew[b] = w[e];
                ++b;
            }
        }
        if (m > 4) c[0] = kLongRow;
        icol4[s] = make_ushort4(c[0], m > 4 ? kNoArc : c[1], m > 4 ? kNoArc : c[2],
                                m > 4 ? kNoArc : c[3]);
        if (iw4) iw4[s] = make_uint4(l[0], l[1], l[2], l[3]);
    }
}

// stats[1] = neighbouring tiles summed over the tiles (an arc counts when no
// earlier one of the tile's leads to the same tile; beyond 2048 leaving arcs
// every one counts).
__global__ void k_tile_stats(int64_t tiles, const int32_t *tb, const int32_t *word_tile,
                             const uint32_t *erp, const int32_t *ecol,
                             unsigned long long *stats)
{
    __shared__ int32_t s_t[2048];
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const uint32_t b = erp[tb[t]], e = erp[tb[t + 1]], m = e - b;
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < m && i < 2048u; i += blockDim.x)
            s_t[i] = word_tile[ecol[b + i] >> 5];
        __syncthreads();
        unsigned fresh = 0;
        for (uint32_t i = threadIdx.x; i < m; i += blockDim.x) {
            bool seen = false;
            if (i < 2048u)
                for (uint32_t j = 0; j < i && !seen; ++j) seen = s_t[j] == s_t[i];
            fresh += !seen;
        }
        if (fresh) atomicAdd(&stats[1], (unsigned long long)fresh);
    }
}

// Breadth-first depth of the tile graph from tile 0, on one CTA (depth, q0,
// q1: tiles entries each, depth at -1): *out = the deepest level.
__global__ void __launch_bounds__(1024)
k_tile_depth(const int32_t *tb, const int32_t *word_tile, const uint32_t *erp,
             const int32_t *ecol, int32_t *depth, int32_t *q0, int32_t *q1,
             unsigned long long *out)
{
    __shared__ unsigned s_n[2];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        depth[0] = 0;
        q0[0] = 0;
        s_n[0] = 1;
        s_n[1] = 0;
    }
    __syncthreads();
    int level = 0;
    for (;; ++level) {
        const unsigned n = s_n[level & 1];
        int32_t *const q = level & 1 ? q1 : q0, *const nq = level & 1 ? q0 : q1;
        for (unsigned i = wid; i < n; i += 32) {
            const int32_t t = q[i];
            const uint32_t e = erp[tb[t + 1]];
            for (uint32_t x = erp[tb[t]] + lane; x < e; x += 32) {
                const int32_t h = word_tile[ecol[x] >> 5];
                if (depth[h] < 0 && atomicCAS(&depth[h], -1, level + 1) == -1)
                    nq[atomicAdd(&s_n[(level + 1) & 1], 1u)] = h;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) s_n[level & 1] = 0;
        __syncthreads();
        if (s_n[(level + 1) & 1] == 0) break;
    }
    if (threadIdx.x == 0) *out = (unsigned long long)level;
}

// ---- the search -----------------------------------------------------------

// Threads of a CTA of the search: a unit of the road-like lattice keeps two to
// four warps busy (64 sources), one of the grid six (256 sources); 256 / 128
// / 64 threads: grid 17.6 / 17.8 / 22.4 ms, road-like 13.2 / 10.4 / 12.2 ms.
template <bool WT>
constexpr int kTileThreads = WT ? 128 : 256;
constexpr int kPair = 2;       // sources a warp takes together
constexpr int kList = 192;     // labels to carry on that a list holds

// A warp's labels of its tile for two sources side by side (entry = half x
// kCap + slot), which of them changed, and two lists of labels to carry
// on, used in turns.
template <bool WT>
struct TileWarp {
    static constexpr int kCap = tile_cap(WT);
    uint32_t d[kPair * kCap];
    uint32_t chg[32];
    uint16_t list[2][kList];
};

// A CTA's tile: inline rows, the first kExt leaving arcs.
constexpr int kExt = 256;
template <bool WT>
struct TileShared {
    TileWarp<WT> warp[kTileThreads<WT> / 32];
    uint4 w4[WT ? tile_cap(WT) : 1];
    ushort4 c4[tile_cap(WT)];
    int32_t ecol[kExt];
    uint32_t ew[WT ? kExt : 1];
    uint16_t etail[kExt];
    int32_t s0, nw, ext;
    uint32_t e0;
};

// A tile and up to two sources (src[1] = -1: one) on one warp: a front inside
// a tile is a dozen nodes wide, and two fill a warp's lanes better than one.
// Labels above T are lowered but not carried on: they stay dirty for the next
// round (with arc lengths, whose labels would otherwise run ahead of the
// shortest paths and be carried on again and again).  pend: smallest label
// left dirty anywhere.  Latency is what bounds it, so the arcs are read from
// shared memory and everything a step can have in flight is: the labels with
// the dirty words, a node's four arcs, the border's minima.
template <bool WT>
__device__ __forceinline__ void tile_sources(const TileJob &J, const TileShared<WT> &C,
                                             TileWarp<WT> &S, int t, const int (&src)[kPair],
                                             uint32_t T, int par,
                                             const Stage &stage, int32_t *Qn, unsigned *qlen,
                                             uint32_t stamp, unsigned *s_pend,
                                             unsigned long long &relax)
{
    constexpr int kCap = TileWarp<WT>::kCap, kWords = kCap / 32;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const int64_t slots = J.g.slots, words = slots >> 5;
    uint32_t *const d = S.d, *const chg = S.chg;
    const int32_t s0 = C.s0;
    const int nw = C.nw, ext = C.ext;
    // The dirty words: lanes 0 .. kWords - 1 the first source's, the next
    // kWords the second's.
    const int hq = lane < kWords ? lane : lane - kWords;
    const int hs = lane < kWords ? src[0] : lane < kPair * kWords ? src[1] : -1;
    uint32_t *const dw = J.dirty[par] + (int64_t)hs * words + (s0 >> 5) + hq;
    const bool mine = hs >= 0 && hq < nw;
    const uint32_t a = mine ? __ldcg(dw) : 0u;
    constexpr int kLoads = (kCap + 127) / 128;
#pragma unroll
    for (int h = 0; h < kPair; ++h) {
        uint4 x[kLoads];
#pragma unroll
        for (int q = 0; q < kLoads; ++q) {
            const int i = 4 * lane + 128 * q;
            if (src[h] >= 0 && i < 32 * nw)
                x[q] = __ldcg(reinterpret_cast<const uint4 *>(J.dist + src[h] * slots + s0 + i));
        }
#pragma unroll
        for (int q = 0; q < kLoads; ++q) {
            const int i = 4 * lane + 128 * q;
            if (src[h] >= 0 && i < 32 * nw)
                *reinterpret_cast<uint4 *>(d + h * kCap + i) = x[q];
        }
    }
    if (a) *dw = 0u;
    chg[lane] = a;
    int n = __popc(a);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, n, o);
        if (lane >= o) n += y;
    }
    int at = n - __popc(a);
    n = __shfl_sync(FULL, n, 31);
    // A list that would not fit is replaced by a sweep over every slot.
    bool sweep = n > kList;
    int cur = 0;
    if (!sweep)
        for (uint32_t b = a; b; b &= b - 1) S.list[0][at++] = (uint16_t)(32 * lane + __ffs(b) - 1);
    __syncwarp();
    while (n) {
        const int todo = sweep ? kPair * 32 * nw : n;
        int cn = 0;
        for (int j0 = 0; j0 < todo; j0 += 32) {
            const int j = j0 + lane;
            int u = 0;
            bool on = j < todo;
            if (on) {
                if (!sweep) u = S.list[cur][j];
                else if (j < 32 * nw) u = j;
                else u = kCap + j - 32 * nw, on = src[1] >= 0;
            }
            const uint32_t du = on ? d[u] : kInf;
            const int hb = u >= kCap ? kCap : 0;
            uint32_t x = 0, e = 0;  // rows of more than four arcs: the rest of the row
            ushort4 c = make_ushort4(kNoArc, kNoArc, kNoArc, kNoArc);
            uint4 w = make_uint4(1u, 1u, 1u, 1u);
            if (du <= T && du != kInf) {
                c = C.c4[u - hb];
                if (WT) w = C.w4[u - hb];
                if (c.x == kLongRow) {
                    x = J.g.irp[s0 + u - hb];
                    e = J.g.irp[s0 + u - hb + 1];
                    c.x = kNoArc;
                }
            }
            const unsigned more = __reduce_max_sync(FULL, (e - x + 3) / 4);
            for (unsigned r = 0;; ++r) {
                int v[4] = {c.x, c.y, c.z, c.w};
                const uint32_t len[4] = {w.x, w.y, w.z, w.w};
                uint32_t nd[4];
                bool imp[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    nd[q] = du + (WT ? len[q] : 1u);
                    imp[q] = v[q] != kNoArc;
                    if (WT && imp[q] && (nd[q] < du || nd[q] == kInf)) {
                        J.ctl->band_ovf = 1;
                        imp[q] = false;
                    }
                    v[q] += hb;
                    if (imp[q]) imp[q] = nd[q] < d[v[q]];
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (imp[q]) imp[q] = nd[q] < atomicMin(&d[v[q]], nd[q]);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const unsigned m = __ballot_sync(FULL, imp[q]);
                    if (imp[q]) {
                        const int p = cn + __popc(m & below);
                        if (p < kList) S.list[cur ^ 1][p] = (uint16_t)v[q];
                        atomicOr(&chg[v[q] >> 5], 1u << (v[q] & 31));
                    }
                    cn += __popc(m);
                }
                if (r == more) break;
                // the next four of a long row
                c.x = x < e ? J.g.icol[x] : kNoArc;
                c.y = x + 1 < e ? J.g.icol[x + 1] : kNoArc;
                c.z = x + 2 < e ? J.g.icol[x + 2] : kNoArc;
                c.w = x + 3 < e ? J.g.icol[x + 3] : kNoArc;
                if (WT) {
                    w.x = x < e ? J.g.iw[x] : 0u;
                    w.y = x + 1 < e ? J.g.iw[x + 1] : 0u;
                    w.z = x + 2 < e ? J.g.iw[x + 2] : 0u;
                    w.w = x + 3 < e ? J.g.iw[x + 3] : 0u;
                }
                x = x + 4 < e ? x + 4 : e;
            }
        }
        if (lane == 0) relax += (unsigned)n;
        __syncwarp();
        n = cn;
        sweep = cn > kList;
        cur ^= 1;
    }
    // What dropped goes back (another tile may have lowered a border label
    // meanwhile: a minimum, not a store); what is above T stays dirty.
    uint32_t pend = kInf;
    unsigned defer = 0;  // bit h: source h has labels left
#pragma unroll
    for (int h = 0; h < kPair; ++h) {
        if (src[h] < 0) continue;
        uint32_t *const dist = J.dist + src[h] * slots + s0;
        for (int q = 0; q < nw; ++q) {
            const uint32_t cw = chg[h * kWords + q];
            if (cw == 0u) continue;
            bool later = false;
            if ((cw >> lane) & 1u) {
                const uint32_t du = d[h * kCap + 32 * q + lane];
                atomicMin(dist + 32 * q + lane, du);
                if (WT && du > T) {
                    later = true;
                    pend = min(pend, du);
                }
            }
            if (WT) {
                const unsigned m = __ballot_sync(FULL, later);
                if (m) {
                    defer |= 1u << h;
                    if (lane == 0)
                        atomicOr(J.dirty[par ^ 1] + src[h] * words + (s0 >> 5) + q, m);
                }
            }
        }
    }
    auto queue_unit = [&](int tt, int s, uint32_t before) {
        if (before) return;
        const int32_t unit = tt * J.ku + (s >> 5) / J.uw;
        if (atomicExch(J.stamp + unit, stamp) != stamp) stage_push(stage, unit, Qn, qlen);
    };
    auto activate = [&](int tt, int s) {
        return atomicOr(J.act[par ^ 1] + (int64_t)tt * J.kw + (s >> 5), 1u << (s & 31));
    };
    if (WT && lane < kPair && ((defer >> lane) & 1u)) {
        const int s = lane == 0 ? src[0] : src[1];
        queue_unit(t, s, activate(t, s));
    }
    // ... and across the border, a lane per leaving arc, two arcs and both
    // sources at a time.
    for (int x0 = 0; x0 < ext; x0 += 64) {
        uint32_t nd[4], old[4];
        int32_t v[2];
        bool go[4];
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            const int x = x0 + 32 * y + lane;
            const bool in = x < ext;
            int u = 0;
            uint32_t len = 1u;
            v[y] = 0;
            if (in && x < kExt) {
                u = C.etail[x];
                v[y] = C.ecol[x];
                if (WT) len = C.ew[x];
            } else if (in) {
                u = J.g.etail[C.e0 + x];
                v[y] = J.g.ecol[C.e0 + x];
                if (WT) len = J.g.ew[C.e0 + x];
            }
#pragma unroll
            for (int h = 0; h < kPair; ++h) {
                const int q = 2 * y + h;
                go[q] = in && src[h] >= 0 &&
                        ((chg[h * kWords + (u >> 5)] >> (u & 31)) & 1u) != 0u;
                const uint32_t du = go[q] ? d[h * kCap + u] : 0u;
                nd[q] = du + len;
                if (WT && go[q]) {
                    if (du > T) go[q] = false;
                    else if (nd[q] < du || nd[q] == kInf) {
                        J.ctl->band_ovf = 1;
                        go[q] = false;
                    }
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            old[q] = 0u;
            if (go[q]) old[q] = atomicMin(J.dist + src[q & 1] * slots + v[q >> 1], nd[q]);
        }
        uint32_t before[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            go[q] = go[q] && nd[q] < old[q];
            before[q] = 1u;
            if (go[q]) {
                const int s = src[q & 1];
                const int32_t vv = v[q >> 1];
                pend = min(pend, nd[q]);
                atomicOr(J.dirty[par ^ 1] + s * words + (vv >> 5), 1u << (vv & 31));
                before[q] = activate(J.g.word_tile[vv >> 5], s);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (go[q]) queue_unit(J.g.word_tile[v[q >> 1] >> 5], src[q & 1], before[q]);
    }
    if (WT) {
        pend = __reduce_min_sync(FULL, pend);
        if (lane == 0 && pend != kInf) atomicMin(s_pend, pend);
    }
    __syncwarp();
}

// Units of a round (a tile, up to 32 uw sources) go to the CTAs: the first
// ones dealt out, the rest taken from a counter.  A CTA loads the tile's arcs
// once and its warps take the unit's active sources two by two.
template <bool WT>
__global__ void __launch_bounds__(kTileThreads<WT>, WT ? 6 : 4) k_tiles(TileJob J)
{
    constexpr int kTT = kTileThreads<WT>;
    extern __shared__ __align__(16) unsigned char s_raw[];
    TileShared<WT> &Cs = *reinterpret_cast<TileShared<WT> *>(s_raw);
    TileWarp<WT> &S = Cs.warp[threadIdx.x >> 5];
    __shared__ int32_t s_buf[kStage];
    __shared__ unsigned s_cnt, s_base, s_pend, s_pop, s_next, s_mask[kUnitWords];
    const Stage stage{s_buf, &s_cnt, &s_base};
    const int lane = threadIdx.x & 31;
    const int64_t gthreads = (int64_t)gridDim.x * kTT;
    const int64_t gtid = (int64_t)blockIdx.x * kTT + threadIdx.x;
    const int64_t slots = J.g.slots, words = slots >> 5;
    Ctl *ctl = J.ctl;
    if (threadIdx.x == 0) s_cnt = 0;
    {
        const uint4 inf = make_uint4(kInf, kInf, kInf, kInf);
        uint4 *d4 = reinterpret_cast<uint4 *>(J.dist);
        for (int64_t i = gtid; i < J.k * (slots >> 2); i += gthreads) d4[i] = inf;
        for (int64_t i = gtid; i < J.k * words; i += gthreads) {
            J.dirty[0][i] = 0u;
            J.dirty[1][i] = 0u;
        }
        for (int64_t i = gtid; i < (int64_t)J.g.tiles * J.kw; i += gthreads) {
            J.act[0][i] = 0u;
            J.act[1][i] = 0u;
        }
        for (int64_t i = gtid; i < (int64_t)J.g.tiles * J.ku; i += gthreads) J.stamp[i] = 0u;
    }
    if (!grid_sync(ctl, blockIdx.x, gridDim.x, J.timeout_ns)) return;
    for (int64_t i = gtid; i < J.k; i += gthreads) {
        const int32_t s = J.g.iperm[J.sources[i]];
        J.dist[i * slots + s] = 0u;
        atomicOr(J.dirty[0] + i * words + (s >> 5), 1u << (s & 31));
        const int32_t t = J.g.word_tile[s >> 5];
        atomicOr(J.act[0] + (int64_t)t * J.kw + (i >> 5), 1u << (i & 31));
        const int32_t unit = t * J.ku + (int32_t)(i >> 5) / J.uw;
        if (atomicExch(J.stamp + unit, 1u) != 1u)  // queued for round 0
            J.Q[0][atomicAdd(&ctl->lev[0].qlen, 1u)] = unit;
    }
    if (!grid_sync(ctl, blockIdx.x, gridDim.x, J.timeout_ns)) return;
    unsigned long long relax = 0;
    uint32_t T = WT ? 0u : kInf;
    int r = 0;
    for (;; ++r) {
        const int par = r & 1;
        LevelCtl *C = &ctl->lev[r & 3];
        const unsigned qn = ((volatile LevelCtl *)C)->qlen;
        if (qn == 0) break;
        if (WT) {  // T moves on by delta, and to the smallest label at least
            const uint32_t pend = r ? ~((volatile LevelCtl *)C)->mlen : 0u;
            const uint32_t from = pend > T ? pend : T;
            T = from + J.delta < from ? kInf : from + J.delta;
        }
        if (gtid == 0) {  // round r + 2's counters
            ctl->lev[(r + 2) & 3].qlen = 0;
            ctl->lev[(r + 2) & 3].hnext = 0;
            ctl->lev[(r + 2) & 3].mlen = 0;  // the complement of its smallest label
        }
        if (threadIdx.x == 0) s_pend = kInf;
        __syncthreads();
        int32_t *Qn = J.Q[par ^ 1];
        unsigned *qlen = &ctl->lev[(r + 1) & 3].qlen;
        for (unsigned p = blockIdx.x; p < qn;) {
            const unsigned unit = (unsigned)__ldcg(J.Q[par] + p);
            const int t = (int)(unit / (unsigned)J.ku), w0 = (int)(unit % (unsigned)J.ku) * J.uw;
            if (threadIdx.x == 0) {
                s_next = 0u;
                s_pop = qn > gridDim.x ? gridDim.x + atomicAdd(&C->hnext, 1u) : qn;
            }
            if (threadIdx.x < kUnitWords) {
                const int w = w0 + (int)threadIdx.x;
                unsigned m = 0u;
                if ((int)threadIdx.x < J.uw && w < J.kw) {
                    uint32_t *act = J.act[par] + (int64_t)t * J.kw + w;
                    m = __ldcg(act);
                    if (m) *act = 0u;
                }
                s_mask[threadIdx.x] = m;
            }
            const int32_t s0 = J.g.tb[t], size = J.g.tb[t + 1] - s0;
            const uint32_t e0 = J.g.erp[s0];
            const int ext = (int)(J.g.erp[s0 + size] - e0);
            if (threadIdx.x == 0) {
                Cs.s0 = s0;
                Cs.nw = size >> 5;
                Cs.ext = ext;
                Cs.e0 = e0;
            }
            for (int i = threadIdx.x; i < size; i += kTT) {
                Cs.c4[i] = J.g.icol4[s0 + i];
                if (WT) Cs.w4[i] = J.g.iw4[s0 + i];
            }
            for (int i = threadIdx.x; i < ext && i < kExt; i += kTT) {
                Cs.etail[i] = J.g.etail[e0 + i];
                Cs.ecol[i] = J.g.ecol[e0 + i];
                if (WT) Cs.ew[i] = J.g.ew[e0 + i];
            }
            __syncthreads();
            for (;;) {
                unsigned q = 0;
                if (lane == 0) q = atomicAdd(&s_next, (unsigned)kPair);
                q = __shfl_sync(FULL, q, 0);
                // active sources number q and q + 1
                int src[kPair] = {-1, -1};
                int w = 0;
                unsigned m = s_mask[0];
#pragma unroll
                for (int h = 0; h < kPair; ++h) {
                    while (q >= (unsigned)__popc(m) && w < kUnitWords - 1) {
                        q -= __popc(m);
                        m = s_mask[++w];
                    }
                    if (q >= (unsigned)__popc(m)) break;
                    for (; q; --q) m &= m - 1;
                    src[h] = (w0 + w) * 32 + __ffs(m) - 1;
                    m &= m - 1;
                }
                if (src[0] < 0) break;
                tile_sources<WT>(J, Cs, S, t, src, T, par, stage, Qn, qlen, (uint32_t)r + 2u,
                                 &s_pend, relax);
            }
            p = s_pop;
            __syncthreads();
        }
        stage_flush(stage, Qn, qlen);
        if (WT && threadIdx.x == 0 && s_pend != kInf)
            atomicMax(&ctl->lev[(r + 1) & 3].mlen, ~s_pend);
        if (!grid_sync(ctl, blockIdx.x, gridDim.x, J.timeout_ns)) return;
    }
    if (lane == 0 && relax) atomicAdd(&ctl->words, relax);
    if (gtid == 0) ctl->levels = r;
}

// ---- reductions -----------------------------------------------------------

// Sums, and the nearest sampled node (ties to the smallest index), a thread
// per slot: consecutive threads read consecutive labels of each source.
__global__ void k_tr_nodes(TileReduce R)
{
    const int64_t slots = R.g.slots;
    for (STRIDED(s, slots)) {
        const int32_t v = R.g.perm[s];
        if (v < 0) continue;
        unsigned long long sum = 0, sq = 0;
        uint32_t best = kInf;
        int bi = 0;
        const uint32_t *p = R.dist + s;
#pragma unroll 8
        for (int i = 0; i < R.k; ++i) {
            const uint64_t d = p[(int64_t)i * slots];
            sum += d;
            sq += d * d;
            if (d < best) {
                best = (uint32_t)d;
                bi = i;
            }
        }
        R.sum2[2 * (int64_t)v] = sum;
        R.sum2[2 * (int64_t)v + 1] = sq;
        R.pivot[v] = bi;
        R.delta[v] = best;
    }
}

// Per source: exact S, the largest distance, whether a node was not reached.
constexpr int kSeg = 8192;  // slots per CTA
constexpr int kWarps = kT / 32;

__global__ void k_tr_sources(TileReduce R)
{
    const int i = blockIdx.y;
    const int64_t b = (int64_t)blockIdx.x * kSeg, e = min(R.g.slots, b + kSeg);
    const uint32_t *d = R.dist + (int64_t)i * R.g.slots;
    unsigned long long sum = 0;
    uint32_t mx = 0;
    bool bad = false;
    for (int64_t s = b + threadIdx.x; s < e; s += kT) {
        if (R.g.perm[s] < 0) continue;
        const uint32_t x = d[s];
        bad |= x == kInf;
        sum += x;
        mx = max(mx, x);
    }
    __shared__ unsigned long long s_sum[kWarps];
    __shared__ uint32_t s_max[kWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(FULL, sum, o);
    mx = __reduce_max_sync(FULL, mx);
    if (lane == 0) {
        s_sum[wid] = sum;
        s_max[wid] = mx;
    }
    if (__syncthreads_or(bad)) {
        if (threadIdx.x == 0) atomicExch(R.err, CC_ERR_DISCONNECTED);
        return;
    }
    if (threadIdx.x == 0) {
        for (int w = 1; w < kWarps; ++w) {
            sum += s_sum[w];
            mx = max(mx, s_max[w]);
        }
        atomicAdd(&R.S_samp[i], sum);
        atomicMax(R.dmax, (unsigned long long)mx);
    }
}

__global__ void k_tr_dcc(TileReduce R)
{
    for (STRIDED(q, (int64_t)R.k * R.k)) {
        const int64_t i = q / R.k, j = q % R.k;
        R.dcc[q] = R.dist[i * R.g.slots + R.g.iperm[R.sources[j]]];
    }
}

// Distance histogram of each source over all nodes; a CTA's slots count in
// shared memory while the distances are few (kSmemHist).
constexpr int kSmemHist = 8192;

__global__ void k_tr_hist(TileReduce R, int local)
{
    extern __shared__ unsigned s_h[];
    const int i = blockIdx.y;
    const int64_t b = (int64_t)blockIdx.x * kSeg, e = min(R.g.slots, b + kSeg);
    const uint32_t *d = R.dist + (int64_t)i * R.g.slots;
    uint32_t *h = R.hist + (int64_t)i * R.hs;
    if (local) {
        for (int x = threadIdx.x; x <= (int)R.D; x += kT) s_h[x] = 0u;
        __syncthreads();
    }
    for (int64_t s = b + threadIdx.x; s < e; s += kT) {
        if (R.g.perm[s] < 0) continue;
        atomicAdd(local ? &s_h[d[s]] : &h[d[s]], 1u);
    }
    if (local) {
        __syncthreads();
        for (int x = threadIdx.x; x <= (int)R.D; x += kT)
            if (s_h[x]) atomicAdd(&h[x], s_h[x]);
    }
}

// The sampled nodes leave the histogram (it counts V \ C).
__global__ void k_tr_unhist(TileReduce R)
{
    for (STRIDED(q, (int64_t)R.k * R.k))
        atomicSub(&R.hist[q / R.k * R.hs + R.dcc[q]], 1u);
}

// Counts and distance sums of each block of 64 distances.
__global__ void k_tr_blocks(TileReduce R)
{
    const int64_t nb = R.hs / 64;
    for (STRIDED(q, (int64_t)R.k * nb)) {
        const int64_t i = q / nb, b = q % nb;
        const uint4 *h = reinterpret_cast<const uint4 *>(R.hist + i * R.hs + 64 * b);
        unsigned long long cn = 0, cs = 0;
#pragma unroll
        for (int x = 0; x < 16; ++x) {
            const uint4 c = h[x];
            const unsigned t = c.x + c.y + c.z + c.w;
            cn += t;
            cs += (unsigned long long)(64 * b + 4 * x) * t + c.y + 2ull * c.z + 3ull * c.w;
        }
        R.TN[i * (nb + 1) + b] = cn;
        R.TS[i * (nb + 1) + b] = cs;
    }
}

// Their suffix sums, a CTA per source: entry b = the blocks from b on.
__global__ void __launch_bounds__(1024) k_tr_suffix(TileReduce R)
{
    __shared__ unsigned long long s_n[32], s_s[32];
    const int64_t nb = R.hs / 64;
    uint64_t *N = R.TN + (int64_t)blockIdx.x * (nb + 1), *Ss = R.TS + (int64_t)blockIdx.x * (nb + 1);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    unsigned long long cn = 0, cs = 0;
    if (tid == 0) N[nb] = Ss[nb] = 0;
    for (int64_t top = nb - 1; top >= 0; top -= 1024) {
        const int64_t b = top - tid;
        unsigned long long x = b >= 0 ? N[b] : 0, y = b >= 0 ? Ss[b] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long p = __shfl_up_sync(FULL, x, o), q = __shfl_up_sync(FULL, y, o);
            if (lane >= o) {
                x += p;
                y += q;
            }
        }
        __syncthreads();
        if (lane == 31) {
            s_n[wid] = x;
            s_s[wid] = y;
        }
        __syncthreads();
        for (int w = 0; w < wid; ++w) {
            x += s_n[w];
            y += s_s[w];
        }
        if (b >= 0) {
            N[b] = cn + x;
            Ss[b] = cs + y;
        }
        for (int w = 0; w < 32; ++w) {
            cn += s_n[w];
            cs += s_s[w];
        }
    }
}

// H statistics of every unsampled node: the blocks beyond its threshold's and
// the rest of that block.
__global__ void k_tr_tail(TileReduce R)
{
    const int64_t nb = R.hs / 64;
    for (STRIDED(s, R.g.slots)) {
        const int32_t v = R.g.perm[s];
        if (v < 0 || R.sidx[v] >= 0) continue;
        const uint64_t thr = R.hp[v].thr;
        if (thr >= (uint64_t)R.D) continue;  // both zero already
        const int p = R.pivot[v];
        const int64_t t = (int64_t)thr, b = t / 64;
        unsigned long long cn = R.TN[p * (nb + 1) + b + 1], cs = R.TS[p * (nb + 1) + b + 1];
        const uint32_t *h = R.hist + p * R.hs;
        for (int64_t x = t + 1; x < 64 * (b + 1); ++x) {
            const unsigned c = h[x];
            cn += c;
            cs += (unsigned long long)x * c;
        }
        R.hp[v].Hnum = cn;
        R.hp[v].Hsum = cs;
    }
}

// Sums over L(v) n C of the nodes whose L(v) misses a sampled node, and the
// inputs of the error estimate (see k_reduce2).
__global__ void k_tr_lc(TileReduce R)
{
    const int64_t slots = R.g.slots;
    for (STRIDED(s, slots)) {
        const int32_t v = R.g.perm[s];
        if (v < 0 || R.sidx[v] >= 0) continue;
        const uint8_t f = R.sqflag ? R.sqflag[v] : 0;
        const bool part = (R.hp[v].LCnum & kPartialBit) != 0;
        const uint32_t *p = R.dist + s;
        if (f & 2) R.fdist[v] = p[(int64_t)R.istar[R.pivot[v]] * slots];
        if (!part && !(f & 1)) continue;
        unsigned long long a = 0, b = 0;
        uint64_t lo = 0, hi = 0;
        const uint32_t *row = R.dcc + (int64_t)R.pivot[v] * R.k;
        for (int w = 0; w < R.W; ++w) {
            const uint64_t m = R.Lmask[(int64_t)v * R.W + w];
            const int i1 = min(R.k, 64 * w + 64);
#pragma unroll 4
            for (int i = 64 * w; i < i1; ++i) {
                const uint64_t d = p[(int64_t)i * slots];
                if ((m >> (i & 63)) & 1ull) {
                    a += d;
                    b += d * d;
                } else if (f & 1) {
                    const int64_t e = (int64_t)d - (int64_t)row[i];
                    const uint64_t x = (uint64_t)(e * e);
                    lo += x;
                    hi += lo < x;
                }
            }
        }
        R.lc2[2 * (int64_t)v] = a;
        R.lc2[2 * (int64_t)v + 1] = b;
        if (f & 1) {
            R.hcse[2 * (int64_t)v] = lo;
            R.hcse[2 * (int64_t)v + 1] = hi;
        }
    }
}

}  // namespace

int tiles_build(int64_t n, int64_t arcs, const int64_t *rp, const int32_t *col,
                const uint32_t *w, TileGraph &out, TileShape &shape, bool *ok, cudaStream_t st)
{
    *ok = false;
    const int cap = tile_cap(w != nullptr);
    Buf lab, stamp, left, k0, v0, k1, v1, flag, idx, first, tfirst, stats;
    T_RC(lab.alloc(n * 4));
    T_RC(stamp.alloc(n * 4));
    T_RC(left.alloc(16));
    const int g = grid_of(n);
    T_CK(cudaMemsetAsync(stamp.p, 0xFF, n * 4, st));
    uint32_t step = 0;
    for (int pass = 0; pass < kGrowPasses; ++pass) {
        k_centres<<<g, kT, 0, st>>>(n, (unsigned)(cap / 2), 0x7f4a7c15ull + pass, step++,
                                    lab.as<int32_t>(), stamp.as<uint32_t>());
        unsigned open = 0;
        T_CK(cudaMemsetAsync(left.p, 0, 4, st));
        for (int h = 0; h < kGrowHops; ++h)
            k_grow<<<g, kT, 0, st>>>(n, rp, col, step++, lab.as<int32_t>(), stamp.as<uint32_t>(),
                                     h == kGrowHops - 1 ? left.as<unsigned>() : nullptr);
        T_CK(cudaMemcpyAsync(&open, left.p, 4, cudaMemcpyDeviceToHost, st));
        T_CK(cudaStreamSynchronize(st));
        if (open == 0) break;
    }
    // Nodes sorted by cluster, tiles of at most cap of them.
    T_RC(k0.alloc(n * 8));
    T_RC(v0.alloc(n * 4));
    T_RC(k1.alloc(n * 8));
    T_RC(v1.alloc(n * 4));
    T_RC(flag.alloc((n + 1) * 8));
    T_RC(idx.alloc((n + 1) * 8));
    T_RC(first.alloc((n + 1) * 4));
    T_RC(tfirst.alloc((n + 1) * 4));
    T_RC(stats.alloc(32));
    T_CK(cudaMemsetAsync(stats.p, 0, 32, st));
    k_keys<<<g, kT, 0, st>>>(n, lab.as<int32_t>(), stamp.as<uint32_t>(), k0.as<uint64_t>(),
                             v0.as<uint32_t>(), stats.as<unsigned long long>() + 2);
    int bits = 1;
    while ((1ll << bits) < n) ++bits;
    bool in_tmp = false;
    T_RC(device_radix_sort(k0.as<uint64_t>(), v0.as<uint32_t>(), n, bits, k1.as<uint64_t>(),
                           v1.as<uint32_t>(), st, &in_tmp));
    const uint64_t *keys = in_tmp ? k1.as<uint64_t>() : k0.as<uint64_t>();
    const uint32_t *sorted = in_tmp ? v1.as<uint32_t>() : v0.as<uint32_t>();
    uint64_t clusters = 0, tiles = 0, words = 0;
    k_cluster_starts<<<g, kT, 0, st>>>(n, keys, flag.as<uint64_t>());
    T_RC(device_scan_u64(flag.as<uint64_t>(), idx.as<uint64_t>(), n, &clusters, st));
    k_cluster_first<<<g, kT, 0, st>>>(n, keys, idx.as<uint64_t>(), first.as<int32_t>());
    k_tile_starts<<<g, kT, 0, st>>>(n, keys, idx.as<uint64_t>(), first.as<int32_t>(), cap,
                                    flag.as<uint64_t>());
    T_RC(device_scan_u64(flag.as<uint64_t>(), idx.as<uint64_t>(), n, &tiles, st));
    k_tile_first<<<g, kT, 0, st>>>(n, flag.as<uint64_t>(), idx.as<uint64_t>(),
                                   tfirst.as<int32_t>(), (int64_t)tiles);
    k_tile_words<<<grid_of((int64_t)tiles), kT, 0, st>>>((int64_t)tiles, tfirst.as<int32_t>(),
                                                         flag.as<uint64_t>());
    T_RC(device_scan_u64(flag.as<uint64_t>(), idx.as<uint64_t>(), (int64_t)tiles, &words, st));
    const int64_t slots = (int64_t)words * 32;
    Buf perm, iperm, tb, wt, irp, erp, icol, ecol, etail, iw, ew, icol4, iw4, din, dex;
    if (slots > 0x7FFFFFE0LL) return CC_OK;
    T_RC(perm.alloc(slots * 4));
    T_RC(iperm.alloc(n * 4));
    T_RC(tb.alloc((tiles + 1) * 4));
    T_RC(wt.alloc(words * 4));
    k_tile_slots<<<(int)std::min<uint64_t>(tiles, 152 * 16), 128, 0, st>>>(
        (int64_t)tiles, tfirst.as<int32_t>(), idx.as<uint64_t>(), sorted, (int64_t)words,
        tb.as<int32_t>(), wt.as<int32_t>(), perm.as<int32_t>(), iperm.as<int32_t>());
    T_RC(din.alloc((slots + 1) * 8));
    T_RC(dex.alloc((slots + 1) * 8));
    const int gs = grid_of(slots + 1);
    k_tile_degrees<<<gs, kT, 0, st>>>(slots, perm.as<int32_t>(), iperm.as<int32_t>(),
                                      wt.as<int32_t>(), rp, col, din.as<uint64_t>(),
                                      dex.as<uint64_t>());
    uint64_t in = 0, ex = 0;
    T_RC(device_scan_u64(din.as<uint64_t>(), din.as<uint64_t>(), slots + 1, &in, st));
    T_RC(device_scan_u64(dex.as<uint64_t>(), dex.as<uint64_t>(), slots + 1, &ex, st));
    if ((double)ex > kMaxCut * (double)arcs) return CC_OK;
    T_RC(irp.alloc((slots + 1) * 4));
    T_RC(erp.alloc((slots + 1) * 4));
    T_RC(icol.alloc(in * 2));
    T_RC(ecol.alloc(ex * 4));
    T_RC(etail.alloc(ex * 2));
    T_RC(icol4.alloc(slots * 8));
    if (w) T_RC(iw4.alloc(slots * 16));
    if (w) {
        T_RC(iw.alloc(in * 4));
        T_RC(ew.alloc(ex * 4));
    }
    k_tile_arcs<<<gs, kT, 0, st>>>(slots, perm.as<int32_t>(), iperm.as<int32_t>(),
                                   wt.as<int32_t>(), tb.as<int32_t>(), rp, col, w,
                                   din.as<uint64_t>(), dex.as<uint64_t>(), irp.as<uint32_t>(),
                                   erp.as<uint32_t>(), icol.as<uint16_t>(), ecol.as<int32_t>(),
                                   etail.as<uint16_t>(), iw.as<uint32_t>(), ew.as<uint32_t>(),
                                   icol4.as<ushort4>(), iw4.as<uint4>());
    k_tile_stats<<<(int)std::min<uint64_t>(tiles, 152 * 8), 128, 0, st>>>(
        (int64_t)tiles, tb.as<int32_t>(), wt.as<int32_t>(), erp.as<uint32_t>(),
        ecol.as<int32_t>(), stats.as<unsigned long long>());
    T_CK(cudaMemsetAsync(lab.p, 0xFF, tiles * 4, st));
    k_tile_depth<<<1, 1024, 0, st>>>(tb.as<int32_t>(), wt.as<int32_t>(), erp.as<uint32_t>(),
                                     ecol.as<int32_t>(), lab.as<int32_t>(), first.as<int32_t>(),
                                     tfirst.as<int32_t>(), stats.as<unsigned long long>() + 3);
    unsigned long long h[4];
    T_CK(cudaMemcpyAsync(h, stats.p, 32, cudaMemcpyDeviceToHost, st));
    T_CK(cudaStreamSynchronize(st));
    T_CK(cudaGetLastError());
    if ((double)h[1] > kMaxNeighbours * (double)tiles)
        return CC_OK;
    // Arc lengths: tiles of few neighbours with long borders interleave, and
    // shortest paths cross the same border again and again (random geometric
    // graphs thinned to degree 2.2 to 4: 2.2 to 3.2 neighbours, 0.9 to 1.9
    // sides of arcs to each, five to seven rounds per tile across; 464 K nodes,
    // k = 64: tiles 77 ms, buckets 47).  Street lattices have 4 to 6 neighbours
    // or borders of 0.2 to 0.4 sides, two and a half rounds (478 K: 9.4
    // against 35 ms).  tiles_pay decides on the others by the call.
    // (Below 64 tiles most lie at the rim and have few neighbours anyway.)
    if (w && tiles >= 64 && (double)h[1] < 4.0 * (double)tiles &&
        (double)ex > 0.5 * std::sqrt((double)n / (double)tiles) * (double)h[1])
        return CC_OK;
    out.n = n;
    out.slots = slots;
    out.tiles = (int32_t)tiles;
    // a tile is about two mean radii across
    out.levels = 2.0 * (double)h[2] / (double)n * (double)h[3];
    shape.depth = (double)h[3];
    shape.neighbours = (double)h[1] / (double)tiles;
    shape.border = (double)ex / (double)std::max(1ull, h[1]) /
                   std::sqrt((double)n / (double)tiles);
    out.perm = perm.take<int32_t>();
    out.iperm = iperm.take<int32_t>();
    out.tb = tb.take<int32_t>();
    out.word_tile = wt.take<int32_t>();
    out.irp = irp.take<uint32_t>();
    out.erp = erp.take<uint32_t>();
    out.icol = icol.take<uint16_t>();
    out.ecol = ecol.take<int32_t>();
    out.etail = etail.take<uint16_t>();
    out.icol4 = icol4.take<ushort4>();
    out.iw4 = iw4.take<uint4>();
    out.iw = iw.take<uint32_t>();
    out.ew = ew.take<uint32_t>();
    *ok = true;
    return CC_OK;
}

void tiles_free(TileGraph &g)
{
    void *p[] = {g.perm, g.iperm, g.tb, g.word_tile, g.irp, g.erp, g.icol, g.ecol, g.etail, g.iw, g.ew, g.icol4, g.iw4};
    for (void *x : p)
        if (x) cudaFree(x);
    g = TileGraph{};
}

// Tiles whose borders to each neighbour are longer than a side interleave:
// fronts cross them to and fro, 5 to 10 levels a round in place of 16 to 32,
// and once there are enough tiles to fill the GPU a label costs five times as
// much (120 to 200 ns a tile and source, elsewhere 14 to 35).  Tiles against
// the other search on thinned random geometric graphs:
// - one bit-packed pass: 60 K nodes of degree 2.6 (2.5 neighbours, 1.5 sides)
//   k = 64 13.4 / 13.7 ms, k = 256 22 / 16, k = 1024 55 / 21; of degree 4 (5.6,
//   1.6) k = 8 8.3 / 5.7, k = 256 19 / 6.6;
// - two passes (the error estimate): degree 2.6 k = 128 18 / 37, degree 4 k = 8
//   8.4 / 11.9; from four on (the adaptive hybrid) tiles were ahead
//   everywhere, 64 / 76 ms at the least;
// - few tiles run side by side at any k: degree 2.6, 14 K nodes k = 256 5.8 /
//   10.2, 18 K (2.5 sides) k = 128 9.3 / 10.5, but 7 K (3.3 sides) 7.3 / 5.4;
// - with arc lengths the other search takes 64 sources at a time: degree 4,
//   60 K nodes k = 64 11.9 / 7.5, k = 200 17 / 26, 16 K 11.0 / 3.1, 12.6 / 11.2.
// Shortcuts (more tiles than three times the square of the tiles across)
// leave few levels: 200 K-node rings, 0.5 % rewired, k = 64 3.0 / 4.6 ms, k =
// 256 10.0 / 6.0; 20 K nodes, 1 %, k = 512 2.0 / 2.5, k = 2048 5.7 / 3.3.
// Lattices with or without gaps, mazes, honeycombs and trees (borders of 0.1 to
// 0.9 sides, below 64 tiles, most of them at the rim, up to 1.4) gain 1.2 to 16
// times from k = 1 to 2048; so do strips a tile or two wide (0.6 to 1.03), told
// by the levels for their tiles (30 x 2000, 11: k = 2048 20 / 62 ms).
bool tiles_pay(const TileGraph &g, const TileShape &s, int64_t k, int passes)
{
    if (s.border > (g.tiles < 64 ? 1.7 : 1.0) && g.levels < 8.0 * (double)g.tiles) {
        const bool thin = s.neighbours < 2.7 &&
                          (s.border < 1.6 || (g.tiles < 128 && s.border < 2.5));
        if (g.iw) return thin || k > 192;
        if (passes >= 4) return true;
        if (thin) return k <= 64 * passes || g.tiles * k <= 24576 * passes;
        return k <= 32 * (passes - 1);
    }
    if (!g.iw && (double)g.tiles > 3.0 * s.depth * s.depth)
        return (double)g.tiles * (double)k <= 1000.0 * passes * g.levels;
    return true;
}

int tile_unit_words(const TileGraph &g, int k)
{
    const int64_t kw = (k + 31) / 32;
    return (int)std::max<int64_t>(1, std::min<int64_t>({kw, kUnitWords, g.tiles * kw / 1216}));
}

int launch_tiles(const TileJob &job, cudaStream_t st)
{
    // The shared memory opted into is a device's, like the residency.
    static PerDevice<Residency> residency[2];
    const int q = job.g.iw ? 1 : 0;
    const void *fn = q ? (const void *)k_tiles<true> : (const void *)k_tiles<false>;
    const size_t smem = q ? sizeof(TileShared<true>) : sizeof(TileShared<false>);
    const int threads = q ? kTileThreads<true> : kTileThreads<false>;
    int dev = 0;
    T_CK(cudaGetDevice(&dev));
    Residency fit;
    T_RC(residency[q].get(dev, &fit, [&](Residency &r) -> int {
        T_CK(cudaDeviceGetAttribute(&r.sms, cudaDevAttrMultiProcessorCount, dev));
        T_CK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        T_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r.per_sm, fn, threads, smem));
        return r.per_sm < 1 ? CC_ERR_CUDA : CC_OK;
    }));
    TileJob j = job;
    void *args[] = {&j};
    T_CK(cudaLaunchCooperativeKernel(fn, dim3(fit.per_sm * fit.sms), dim3(threads), args, smem, st));
    return CC_OK;
}

void run_tiles_reduce1(const TileReduce &r, cudaStream_t st)
{
    k_tr_nodes<<<grid_of(r.g.slots), kT, 0, st>>>(r);
    const dim3 seg((unsigned)((r.g.slots + kSeg - 1) / kSeg), (unsigned)r.k);
    k_tr_sources<<<seg, kT, 0, st>>>(r);
    k_tr_dcc<<<grid_of((int64_t)r.k * r.k), kT, 0, st>>>(r);
}

void run_tiles_reduce2(const TileReduce &r, cudaStream_t st)
{
    const dim3 seg((unsigned)((r.g.slots + kSeg - 1) / kSeg), (unsigned)r.k);
    const bool local = r.D < kSmemHist;
    k_tr_hist<<<seg, kT, local ? (size_t)(r.D + 1) * 4 : 0, st>>>(r, local);
    k_tr_unhist<<<grid_of((int64_t)r.k * r.k), kT, 0, st>>>(r);
    k_tr_blocks<<<grid_of((int64_t)r.k * (r.hs / 64)), kT, 0, st>>>(r);
    k_tr_suffix<<<r.k, 1024, 0, st>>>(r);
    k_tr_tail<<<grid_of(r.g.slots), kT, 0, st>>>(r);
    k_tr_lc<<<grid_of(r.g.slots), kT, 0, st>>>(r);
}

}  // namespace ccg
