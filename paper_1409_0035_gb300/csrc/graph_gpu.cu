// Graph to CSR on the device (undirected graphs): the preprocessing step
// that section 7 counts in its times.
//
//   1. edges as 64-bit keys (smaller end << b | larger end), b = ceil(log2
//      n); self-loops get the largest key and sort last;
//   2. stable LSD radix sort of the keys, lengths carried along if given;
//   3. parallel edges merged keeping the smallest length (first of each run,
//      compacted tile by tile);
//   4. connected components by lock-free union-find over the merged edges
//      (roots hooked under the smaller root with atomicCAS), so a component's
//      label is its smallest node id; the largest component wins, ties to
//      the smallest label; kept nodes renumbered in increasing original id
//      (exclusive scan);
//   5. the edges sorted the other way round (by the larger end alone: the
//      sort is stable);
//   6. a kept node's row is its edges as the larger end, then those as the
//      smaller end: both runs ascend and the first lies below the second.
// Half the keys of a sort of both arcs of every edge, and no pass over rows.
#include <algorithm>
#include <cstdint>
#include <vector>

#include "cc_internal.h"
#include "graph_gpu.h"

namespace ccg {

namespace {

constexpr int kThreads = 256;
constexpr int kItems = 8;                  // keys per thread per sort tile
constexpr int kTile = kThreads * kItems;   // 2048 keys per tile
constexpr int kRadix = 256;

// ---------------------------------------------------------------- scan

// Exclusive scan of uint64 values in tiles of kThreads*4: per-tile sums,
// scan of the sums (recursively), then the in-tile scan plus offset.
__global__ void k_tile_sums(const uint64_t *in, int64_t n, uint64_t *sums)
{
    __shared__ uint64_t s[kThreads];
    const int64_t base = (int64_t)blockIdx.x * kThreads * 4;
    uint64_t t = 0;
    for (int j = 0; j < 4; ++j) {
        const int64_t i = base + (int64_t)j * kThreads + threadIdx.x;
        if (i < n) t += in[i];
    }
    s[threadIdx.x] = t;
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) sums[blockIdx.x] = s[0];
}

__global__ void k_tile_scan(const uint64_t *in, int64_t n, const uint64_t *offs,
                            uint64_t *out)
{
    __shared__ uint64_t s[kThreads * 4];
    const int64_t base = (int64_t)blockIdx.x * kThreads * 4;
    for (int j = 0; j < 4; ++j) {
        const int64_t i = base + (int64_t)j * kThreads + threadIdx.x;
        s[j * kThreads + threadIdx.x] = i < n ? in[i] : 0;
    }
    __syncthreads();
    // each thread scans 4 consecutive values, then a Hillis-Steele scan of
    // the thread totals
    uint64_t v[4], tot = 0;
    for (int j = 0; j < 4; ++j) {
        v[j] = s[threadIdx.x * 4 + j];
        tot += v[j];
    }
    __shared__ uint64_t t[kThreads];
    t[threadIdx.x] = tot;
    __syncthreads();
    for (int o = 1; o < kThreads; o <<= 1) {
        const uint64_t a = threadIdx.x >= o ? t[threadIdx.x - o] : 0;
        __syncthreads();
        t[threadIdx.x] += a;
        __syncthreads();
    }
    uint64_t run = t[threadIdx.x] - tot + offs[blockIdx.x];
    __syncthreads();
    for (int j = 0; j < 4; ++j) {
        s[threadIdx.x * 4 + j] = run;
        run += v[j];
    }
    __syncthreads();
    for (int j = 0; j < 4; ++j) {
        const int64_t i = base + (int64_t)j * kThreads + threadIdx.x;
        if (i < n) out[i] = s[j * kThreads + threadIdx.x];
    }
}

// Exclusive scan in place of nb sums by one CTA, four a thread and step;
// *total = their sum.
__global__ void __launch_bounds__(1024) k_scan_sums(uint64_t *sums, int64_t nb, uint64_t *total)
{
    __shared__ uint64_t s_w[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t run = 0;
    for (int64_t b0 = 0; b0 < nb; b0 += 4096) {
        const int64_t b = b0 + 4 * (int64_t)threadIdx.x;
        uint64_t v[4], t = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            v[j] = b + j < nb ? sums[b + j] : 0;
            t += v[j];
        }
        uint64_t incl = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += y;
        }
        __syncthreads();
        if (lane == 31) s_w[wid] = incl;
        __syncthreads();
        uint64_t at = run + incl - t;
        for (int w = 0; w < 32; ++w) {
            if (w < wid) at += s_w[w];
            run += s_w[w];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (b + j < nb) sums[b + j] = at;
            at += v[j];
        }
    }
    if (threadIdx.x == 0) *total = run;
}

// ---------------------------------------------------------------- sort
//
// Stable LSD radix sort, 8 bits a round: digit counts per tile, a scan of
// each digit's counts over the tiles, and a scatter that first orders its
// tile in shared memory, so that keys of one digit leave in runs.  Bound by
// the 16 (24 with values) bytes a key moves per round; ranking warp by warp
// (a match of the digits per 32 keys, no block barrier inside a tile) and
// scattering from shared memory took the five rounds over 8.4 M keys of an
// R-MAT 18 (five over both arcs with values, 0.96 ms) to 0.40 ms (eight over the
// edges alone).

__global__ void __launch_bounds__(kThreads)
k_digit_hist(const uint64_t *keys, int64_t n, int shift, int nbits, uint32_t *counts, int ntiles)
{
    __shared__ uint32_t h[kRadix];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kTile;
    const uint64_t mask = (1ull << nbits) - 1;
    uint64_t k[kItems];
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
        const int64_t i = base + (int64_t)j * kThreads + threadIdx.x;
        k[j] = i < n ? keys[i] : 0;
    }
#pragma unroll
    for (int j = 0; j < kItems; ++j)
        if (base + (int64_t)j * kThreads + threadIdx.x < n)
            atomicAdd(&h[(k[j] >> shift) & mask], 1u);
    __syncthreads();
    counts[(int64_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// Exclusive scan of x over the CTA's 256 threads (s_w: 8 entries); returns
// the total in *total.
__device__ __forceinline__ uint32_t block_scan256(uint32_t x, uint32_t *s_w, uint32_t *total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    __syncthreads();
    if (lane == 31) s_w[wid] = incl;
    __syncthreads();
    uint32_t at = incl - x, t = 0;
    for (int w = 0; w < kThreads / 32; ++w) {
        if (w < wid) at += s_w[w];
        t += s_w[w];
    }
    *total = t;
    return at;
}

// counts[d][0 .. ntiles) -> exclusive prefix sums, tot[d] = the digit's total
// (a CTA per digit; a digit has fewer than 2^32 keys).
__global__ void __launch_bounds__(kThreads) k_digit_rows(uint32_t *counts, int ntiles,
                                                         uint32_t *tot)
{
    __shared__ uint32_t s_w[kThreads / 32];
    uint32_t *row = counts + (int64_t)blockIdx.x * ntiles;
    uint32_t run = 0;
    for (int t0 = 0; t0 < ntiles; t0 += kThreads) {
        const int t = t0 + threadIdx.x;
        uint32_t all;
        const uint32_t at = block_scan256(t < ntiles ? row[t] : 0u, s_w, &all);
        if (t < ntiles) row[t] = run + at;
        run += all;
    }
    if (threadIdx.x == 0) tot[blockIdx.x] = run;
}

template <bool VALS>
__global__ void __launch_bounds__(kThreads)
k_digit_scatter(const uint64_t *keys, const uint32_t *vals, int64_t n, int shift, int nbits,
                const uint32_t *counts, const uint32_t *tot, int ntiles, uint64_t *okeys,
                uint32_t *ovals)
{
    constexpr int kWarps = kThreads / 32;
    __shared__ uint32_t s_cnt[kWarps][kRadix];
    __shared__ uint64_t s_key[kTile];
    __shared__ uint32_t s_val[VALS ? kTile : 1];
    __shared__ uint32_t s_start[kRadix], s_w[kWarps];
    __shared__ int64_t s_off[kRadix];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int w = 0; w < kWarps; ++w) s_cnt[w][tid] = 0;
    // where the digit's keys begin: those of smaller digits, then of earlier
    // tiles
    uint32_t all;
    const int64_t dbase = block_scan256(tot[tid], s_w, &all);
    const int64_t gbase = dbase + counts[(int64_t)tid * ntiles + blockIdx.x];
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kTile;
    const int size = (int)min((int64_t)kTile, n - base);
    const uint64_t mask = (1ull << nbits) - 1;
    uint64_t key[kItems];
    uint32_t val[kItems];
    uint16_t rank[kItems];
    // a warp's keys are consecutive: kItems x 32 of the tile
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
        const int x = wid * 32 * kItems + 32 * j + lane;
        key[j] = x < size ? keys[base + x] : 0;
        if (VALS) val[j] = x < size ? vals[base + x] : 0;
    }
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
        const int x = wid * 32 * kItems + 32 * j + lane;
        const int d = x < size ? (int)((key[j] >> shift) & mask) : kRadix;
        const unsigned peers = __match_any_sync(0xFFFFFFFFu, d);
        const int before = __popc(peers & ((1u << lane) - 1u));
        const uint32_t at = d < kRadix ? s_cnt[wid][d] : 0u;
        __syncwarp();
        if (d < kRadix && before == 0) s_cnt[wid][d] = at + __popc(peers);
        __syncwarp();
        rank[j] = (uint16_t)(at + before);
    }
    __syncthreads();
    uint32_t acc = 0;  // thread = digit: earlier warps' keys of it
    for (int w = 0; w < kWarps; ++w) {
        const uint32_t c = s_cnt[w][tid];
        s_cnt[w][tid] = acc;
        acc += c;
    }
    s_start[tid] = block_scan256(acc, s_w, &all);
    s_off[tid] = gbase - (int64_t)s_start[tid];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
        const int x = wid * 32 * kItems + 32 * j + lane;
        if (x >= size) continue;
        const int d = (int)((key[j] >> shift) & mask);
        const uint32_t p = s_start[d] + s_cnt[wid][d] + rank[j];
        s_key[p] = key[j];
        if (VALS) s_val[p] = val[j];
    }
    __syncthreads();
    for (int x = tid; x < size; x += kThreads) {
        const uint64_t k = s_key[x];
        const int64_t to = s_off[(k >> shift) & mask] + x;
        okeys[to] = k;
        if (VALS) ovals[to] = s_val[x];
    }
}

// ---------------------------------------------------------------- arcs

// Arc keys (tail << b | head) of directed input with their lengths; flags: the
// arcs to keep (no self-loops).
__global__ void k_make_arcs(const uint32_t *src, const uint32_t *dst, const uint32_t *w,
                            int64_t m, int64_t n, int b, uint64_t *keys, uint32_t *vals,
                            uint64_t *flags, int *err)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t u = src[e], v = dst[e];
        const uint32_t ww = w ? w[e] : 1u;
        if ((int64_t)u >= n || (int64_t)v >= n) atomicExch(err, CC_ERR_GRAPH);
        if (ww == 0) atomicExch(err, CC_ERR_ARG);
        keys[e] = (u << b) | v;
        vals[e] = ww;
        flags[e] = u != v && (int64_t)u < n && (int64_t)v < n;
    }
}

__global__ void k_compact(const uint64_t *keys, const uint32_t *vals, const uint64_t *flags,
                          const uint64_t *pos, int64_t n, uint64_t *okeys, uint32_t *ovals)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        if (flags[i]) {
            okeys[pos[i]] = keys[i];
            ovals[pos[i]] = vals[i];
        }
}

// flags[i] = 1 for the first arc of each run of equal keys; mins[run start]
// = the smallest length of the run.
__global__ void k_first_of_run(const uint64_t *keys, int64_t n, uint64_t *flags)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        flags[i] = (i == 0 || keys[i] != keys[i - 1]) ? 1 : 0;
}

__global__ void k_run_min(const uint64_t *keys, uint32_t *vals, const uint64_t *flags,
                          int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (!flags[i]) continue;
        uint32_t mn = vals[i];
        for (int64_t j = i + 1; j < n && keys[j] == keys[i]; ++j) mn = min(mn, vals[j]);
        vals[i] = mn;
    }
}

// Row offsets from keys sorted by tail: rp[u] = first arc with tail >= u.
__global__ void k_row_ptr(const uint64_t *keys, int64_t a, int64_t n, int b, int64_t *rp)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= a;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t cur = i < a ? (int64_t)(keys[i] >> b) : n;
        const int64_t prev = i > 0 ? (int64_t)(keys[i - 1] >> b) : -1;
        for (int64_t u = prev + 1; u <= cur; ++u) rp[u] = i;
    }
}

__global__ void k_heads(const uint64_t *keys, int64_t a, int b, int32_t *col)
{
    const uint64_t mask = (1ull << b) - 1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a;
         i += (int64_t)gridDim.x * blockDim.x)
        col[i] = (int32_t)(keys[i] & mask);
}

// ---------------------------------------------------------------- components

__device__ __forceinline__ int32_t find_root(int32_t *parent, int32_t x)
{
    int32_t p = parent[x];
    while (p != x) {
        const int32_t g = parent[p];
        if (g != p) parent[x] = g;  // path halving (benign race)
        x = p;
        p = g;
    }
    return x;
}

__global__ void k_iota32(int32_t *p, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        p[i] = (int32_t)i;
}

// Union of the endpoints of every arc u -> v with u < v.
// A warp per node, a lane per arc (hub rows no longer run on one thread).
__global__ void k_hook(const int64_t *rp, const int32_t *col, int64_t n, int32_t *parent)
{
    const int lane = threadIdx.x & 31;
    for (int64_t u = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; u < n;
         u += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        for (int64_t e = rp[u] + lane; e < rp[u + 1]; e += 32) {
            const int32_t v = col[e];
            if (v <= u) continue;
            int32_t a = find_root(parent, (int32_t)u), b = find_root(parent, v);
            while (a != b) {
                if (a < b) { const int32_t t = a; a = b; b = t; }  // hook larger under smaller
                const int32_t old = atomicCAS(&parent[a], a, b);
                if (old == a) break;
                a = find_root(parent, old);
                b = find_root(parent, b);
            }
        }
    }
}

// ------------------------------------------------ undirected input, edge-wise

constexpr int kEdgeTile = kThreads * 8;

struct BuildInfo {
    int err;
    unsigned long long loops;           // self-loops dropped
    unsigned long long m;               // edges given
    uint64_t edges, nodes, arcs;        // merged edges; kept nodes; their arcs
    unsigned long long best;            // largest component: size << 32 | ~root
};

// Keys (smaller << b | larger); loops, and ends out of range, get the key of
// a loop at the largest id there is room for, which sorts last.
__global__ void k_pack_edges(const uint32_t *src, const uint32_t *dst, const uint32_t *w,
                             int64_t m, int64_t n, int b, uint64_t *keys, uint32_t *vals,
                             BuildInfo *info)
{
    unsigned long long loops = 0;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t u = src[e], v = dst[e];
        const bool out = (int64_t)u >= n || (int64_t)v >= n;
        if (out) atomicExch(&info->err, CC_ERR_GRAPH);
        if (w) {
            if (w[e] == 0) atomicExch(&info->err, CC_ERR_ARG);
            vals[e] = w[e];
        }
        const bool loop = out || u == v;
        loops += loop;
        keys[e] = loop ? (1ull << (2 * b)) - 1 : u < v ? (u << b) | v : (v << b) | u;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) loops += __shfl_xor_sync(0xFFFFFFFFu, loops, o);
    if ((threadIdx.x & 31) == 0 && loops) atomicAdd(&info->loops, loops);
    if (blockIdx.x == 0 && threadIdx.x == 0) info->m = (unsigned long long)m;
}

// First edges of runs of equal keys per tile (eight consecutive a thread).
__device__ __forceinline__ unsigned run_heads(const uint64_t *keys, int64_t i0, int64_t n)
{
    unsigned heads = 0;
    uint64_t last = i0 > 0 && i0 < n ? keys[i0 - 1] : ~0ull;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (i0 + j >= n) break;
        const uint64_t k = keys[i0 + j];
        if (k != last) heads |= 1u << j;
        last = k;
    }
    return heads;
}

__global__ void __launch_bounds__(kThreads) k_runs_count(const uint64_t *keys,
                                                         const BuildInfo *info, uint64_t *tiles)
{
    __shared__ uint32_t s_w[kThreads / 32];
    const int64_t n = (int64_t)(info->m - info->loops);
    const int64_t i0 = (int64_t)blockIdx.x * kEdgeTile + 8 * (int64_t)threadIdx.x;
    uint32_t all;
    block_scan256(__popc(run_heads(keys, i0, n)), s_w, &all);
    if (threadIdx.x == 0) tiles[blockIdx.x] = all;
}

__global__ void __launch_bounds__(kThreads)
k_runs_write(const uint64_t *keys, const uint32_t *vals, const BuildInfo *info,
             const uint64_t *tiles, uint64_t *okeys, uint32_t *ovals)
{
    __shared__ uint32_t s_w[kThreads / 32];
    const int64_t n = (int64_t)(info->m - info->loops);
    const int64_t i0 = (int64_t)blockIdx.x * kEdgeTile + 8 * (int64_t)threadIdx.x;
    const unsigned heads = run_heads(keys, i0, n);
    uint32_t all;
    uint64_t at = tiles[blockIdx.x] + block_scan256(__popc(heads), s_w, &all);
    for (unsigned h = heads; h; h &= h - 1, ++at) {
        const int64_t i = i0 + __ffs(h) - 1;
        const uint64_t k = keys[i];
        okeys[at] = k;
        if (vals) {
            uint32_t mn = vals[i];
            for (int64_t x = i + 1; x < n && keys[x] == k; ++x) mn = min(mn, vals[x]);
            ovals[at] = mn;
        }
    }
}

// Union of the ends of the merged edges: which = 0 each smaller end's first
// edge, 1 its second, 2 the others.
__global__ void k_link(const uint64_t *keys, const BuildInfo *info, int b, int which,
                       int32_t *parent)
{
    const int64_t A = (int64_t)info->edges;
    const uint64_t mask = (1ull << b) - 1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < A;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = keys[i], u = k >> b;
        const bool first = i == 0 || keys[i - 1] >> b != u;
        const bool second = !first && (i == 1 || keys[i - 2] >> b != u);
        if (which == 0 ? !first : which == 1 ? !second : first || second) continue;
        int32_t x = parent[u], y = parent[k & mask];
        if (x == y) continue;
        x = find_root(parent, x);
        y = find_root(parent, y);
        while (x != y) {  // hook the larger root under the smaller
            if (x < y) { const int32_t t = x; x = y; y = t; }
            const int32_t old = atomicCAS(&parent[x], x, y);
            if (old == x) break;
            x = find_root(parent, old);
            y = find_root(parent, y);
        }
    }
}

// Every node under its root (reads only roots' chains; a root stays itself).
__global__ void k_compress(int32_t *parent, int64_t n)
{
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        int32_t r = parent[v];
        while (parent[r] != r) r = parent[r];
        parent[v] = r;
    }
}

// size[root] += its nodes, one atomic per root and warp.
__global__ void k_label_count(const int32_t *parent, int64_t n, uint32_t *size)
{
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int32_t r = parent[v];
        const unsigned on = __activemask();
        const unsigned same = __match_any_sync(on, r);
        if ((threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(&size[r], (uint32_t)__popc(same));
    }
}

// best = max over roots of (size << 32 | ~root): largest, ties to smallest id
__global__ void k_pick(const uint32_t *size, int64_t n, unsigned long long *best)
{
    unsigned long long m = 0;
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x)
        if (size[v]) {
            const unsigned long long k = ((unsigned long long)size[v] << 32) |
                                         (0xFFFFFFFFull - (unsigned long long)v);
            m = k > m ? k : m;
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xFFFFFFFFu, m, o);
        m = y > m ? y : m;
    }
    if ((threadIdx.x & 31) == 0 && m) atomicMax(best, m);
}

__global__ void k_keep_flags(const int32_t *parent, int64_t n, const BuildInfo *info,
                             uint64_t *flags)
{
    const int32_t root = (int32_t)(0xFFFFFFFFull - (info->best & 0xFFFFFFFFull));
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x)
        flags[v] = !parent || parent[v] == root ? 1 : 0;
}

__global__ void k_new_ids(const uint64_t *flags, const uint64_t *pos, int64_t n, int32_t *newid,
                          int32_t *oldid)
{
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        newid[v] = flags[v] ? (int32_t)pos[v] : -1;
        if (flags[v]) oldid[pos[v]] = (int32_t)v;
    }
}

// starts[u] = first of the merged keys with an upper end >= u, u = 0 .. n.
__global__ void k_row_starts(const uint64_t *keys, const BuildInfo *info, int64_t n, int b,
                             uint32_t *starts)
{
    const int64_t A = (int64_t)info->edges;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= A;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t cur = i < A ? (int64_t)(keys[i] >> b) : n;
        const int64_t prev = i > 0 ? (int64_t)(keys[i - 1] >> b) : -1;
        for (int64_t u = prev + 1; u <= cur; ++u) starts[u] = (uint32_t)i;
    }
}

// Keys (larger << b | smaller); beyond the merged edges the largest key.
__global__ void k_swap_ends(const uint64_t *keys, const uint32_t *vals, const BuildInfo *info,
                            int64_t m, int b, uint64_t *okeys, uint32_t *ovals)
{
    const int64_t A = (int64_t)info->edges;
    const uint64_t mask = (1ull << b) - 1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        okeys[i] = i < A ? ((keys[i] & mask) << b) | (keys[i] >> b) : (1ull << (2 * b)) - 1;
        if (vals) ovals[i] = i < A ? vals[i] : 0u;
    }
}

// deg[new id] of the kept nodes (the rest of deg is zero).
__global__ void k_kept_deg(const uint32_t *fs, const uint32_t *rs, const int32_t *newid,
                           int64_t n, uint64_t *deg)
{
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x)
        if (newid[v] >= 0) deg[newid[v]] = (fs[v + 1] - fs[v]) + (rs[v + 1] - rs[v]);
}

__global__ void k_row_ptr_kept(const uint64_t *pos, int64_t nk, int64_t arcs, int64_t *rp)
{
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x <= nk;
         x += (int64_t)gridDim.x * blockDim.x)
        rp[x] = x < nk ? (int64_t)pos[x] : arcs;
}

// Both arcs of every merged edge: fk by (smaller, larger), rk by (larger,
// smaller).  A row is its smaller neighbours, then its larger ones.
__global__ void k_fill_rows(const uint64_t *fk, const uint64_t *rk, const uint32_t *fw,
                            const uint32_t *rw, int64_t A, int b, const uint32_t *fs,
                            const uint32_t *rs, const int32_t *newid, const int64_t *rp,
                            int32_t *col, uint32_t *w)
{
    const uint64_t mask = (1ull << b) - 1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < A;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint64_t u = fk[i] >> b, v = fk[i] & mask;
        int32_t x = newid[u];
        if (x >= 0) {
            const int64_t p = rp[x] + (rs[u + 1] - rs[u]) + (i - fs[u]);
            col[p] = newid[v];
            if (w) w[p] = fw[i];
        }
        v = rk[i] >> b;
        u = rk[i] & mask;
        x = newid[v];
        if (x >= 0) {
            const int64_t p = rp[x] + (i - rs[v]);
            col[p] = newid[u];
            if (w) w[p] = rw[i];
        }
    }
}

// Temporaries of a build, carved from one allocation: taken twice, once for
// the sizes and once for the addresses.
struct Arena {
    void *base = nullptr;
    size_t off = 0;
    uint32_t *src, *dst, *w, *v0, *v1, *radix, *size, *fs, *rs;
    uint64_t *k0, *k1, *tiles, *flag, *pos, *scan;
    int32_t *parent, *newid, *oldid;
    BuildInfo *info;
    Arena() = default;
    Arena(const Arena &) = delete;
    Arena &operator=(const Arena &) = delete;
    ~Arena() { if (base) cudaFree(base); }
    template <class T> T *take(size_t count)
    {
        T *p = base ? reinterpret_cast<T *>(static_cast<char *>(base) + off) : nullptr;
        off += (count * sizeof(T) + 255) & ~size_t(255);
        return p;
    }
    int allocate()
    {
        if (cudaMalloc(&base, off ? off : 256) != cudaSuccess) {
            cudaGetLastError();
            base = nullptr;
            return CC_ERR_OOM;
        }
        off = 0;
        return CC_OK;
    }
};

// ---- degree classes ------------------------------------------------------

// Keys min(degree, kMediumMaxDeg + 1); counts[0..3]: tiny, light, medium and
// heavy nodes, counts[4]: chunk tasks of the heavy ones.
__global__ void k_degree_keys(const int64_t *rp, int64_t n, uint64_t *keys, uint32_t *vals,
                              unsigned long long *counts)
{
    __shared__ unsigned s_c[5];
    if (threadIdx.x < 5) s_c[threadIdx.x] = 0;
    __syncthreads();
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int64_t d = rp[v + 1] - rp[v];
        keys[v] = (uint64_t)(d <= kMediumMaxDeg ? d : kMediumMaxDeg + 1);
        vals[v] = (uint32_t)v;
        atomicAdd(&s_c[d <= kTinyMaxDeg ? 0 : d <= kLightMaxDeg ? 1 : d <= kMediumMaxDeg ? 2 : 3],
                  1u);
        if (d > kMediumMaxDeg) atomicAdd(&s_c[4], (unsigned)((d + kChunk - 1) / kChunk));
    }
    __syncthreads();
    if (threadIdx.x < 5 && s_c[threadIdx.x])
        atomicAdd(&counts[threadIdx.x], (unsigned long long)s_c[threadIdx.x]);
}

// Chunk tasks of the heavy nodes in order, by one CTA.
__global__ void __launch_bounds__(kThreads) k_heavy_chunks(const int32_t *H, int64_t nH,
                                                           const int64_t *rp, int32_t *Hn,
                                                           int64_t *Hb)
{
    __shared__ uint32_t s_w[kThreads / 32];
    int64_t run = 0;
    for (int64_t h0 = 0; h0 < nH; h0 += kThreads) {
        const int64_t h = h0 + threadIdx.x;
        int32_t v = 0;
        int64_t b = 0, d = 0;
        if (h < nH) {
            v = H[h];
            b = rp[v];
            d = rp[v + 1] - b;
        }
        const uint32_t c = (uint32_t)((d + kChunk - 1) / kChunk);
        uint32_t all;
        const int64_t at = run + block_scan256(c, s_w, &all);
        for (uint32_t q = 0; q < c; ++q) {
            Hn[at + q] = v;
            Hb[at + q] = b + (int64_t)q * kChunk;
        }
        run += all;
    }
}

// ---------------------------------------------------------------- directed

// Reverse arc keys (head << b | tail) with the lengths.
__global__ void k_swap_keys(const uint64_t *keys, const uint32_t *vals, int64_t a, int b,
                            uint64_t *okeys, uint32_t *ovals)
{
    const uint64_t mask = (1ull << b) - 1;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < a;
         e += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t u = keys[e] >> b, v = keys[e] & mask;
        okeys[e] = (v << b) | u;
        ovals[e] = vals[e];
    }
}

// ------------------------------------------------- strongly connected parts
//
// Largest strongly connected component (round trips need strong
// connectivity, section 6.1), found on the device.  Every live node
// carries the label of the part of the graph it lies in; a part holds every
// strongly connected component it meets.  The parts start as the weakly
// connected components.  Each round:
//   trim    a node without an arc from, or without one to, a live node of
//           its own part is a component by itself;
//   stats   per part: size, smallest id and a pivot (largest out x in
//           degree, ties to the smallest id);
//   prune   a part that cannot hold a component beating the best one found
//           so far (fewer nodes, or as many with a larger smallest id) dies;
//   search  forward and backward searches from every pivot, confined to its
//           part; the nodes reached both ways are the pivot's component, the
//           rest of the part splits into three new parts (reached forward
//           only, backward only, neither), each holding whole components.
// Labels: 2n + root for the weak components, p and n + p for the forward-
// and backward-only remainders of pivot p (p never pivots again), the
// remainder reached by neither keeps its label.
constexpr uint64_t kDeadLab = ~0ull;
constexpr unsigned kFull = 0xFFFFFFFFu;

__device__ __forceinline__ unsigned long long best_key(unsigned size, uint32_t min_id)
{
    return ((unsigned long long)size << 32) | (0xFFFFFFFFull - min_id);
}

__global__ void k_scc_init(const int32_t *parent, int64_t n, uint64_t *lab, int32_t *comp)
{
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        int32_t r = (int32_t)v;
        while (parent[r] != r) r = parent[r];
        lab[v] = (uint64_t)(2 * n + r);
        comp[v] = -1;
    }
}

// True when some arc of row v (a warp scans it 32 arcs at a time) leads to
// a node labelled L.
__device__ __forceinline__ bool row_meets(const int64_t *rp, const int32_t *col,
                                          const uint64_t *lab, int64_t v, uint64_t L, int lane)
{
    const int64_t end = rp[v + 1];
    for (int64_t e0 = rp[v]; e0 < end; e0 += 32) {
        const int64_t e = e0 + lane;
        const bool hit = e < end && lab[col[e]] == L;
        if (__any_sync(kFull, hit)) return true;
    }
    return false;
}

// Trim, a warp per node.  Labels change in place while other warps read
// them: a node seen live or dead either way keeps the decision valid, since
// a trimmed node is a component of its own.
__global__ void k_scc_trim(const int64_t *rp, const int32_t *col, const int64_t *rrp,
                           const int32_t *rcol, int64_t n, uint64_t *lab, int32_t *comp,
                           unsigned long long *removed, unsigned long long *best)
{
    const int lane = threadIdx.x & 31;
    unsigned long long cnt = 0, bk = 0;
    for (int64_t v = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; v < n;
         v += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const uint64_t L = lab[v];
        if (L == kDeadLab) continue;
        if (row_meets(rp, col, lab, v, L, lane) && row_meets(rrp, rcol, lab, v, L, lane))
            continue;
        if (lane == 0) {
            lab[v] = kDeadLab;
            comp[v] = (int32_t)v;
            ++cnt;
            bk = max(bk, best_key(1u, (uint32_t)v));
        }
    }
    if (lane == 0 && cnt) {
        atomicAdd(removed, cnt);
        atomicMax(best, bk);
    }
}

// Per part: size, smallest id, pivot key (out x in degree << 32 | ~id).
// Warps whose live lanes share one part reduce first (the common case: one
// large part).
__global__ void k_scc_stats(const int64_t *rp, const int64_t *rrp, int64_t n,
                            const uint64_t *lab, unsigned long long *pk, unsigned *sz,
                            unsigned *mn)
{
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n;
         base += stride) {
        const int64_t v = base + lane;
        const uint64_t L = v < n ? lab[v] : kDeadLab;
        const bool live = L != kDeadLab;
        const unsigned bal = __ballot_sync(kFull, live);
        if (!bal) continue;
        unsigned long long key = 0;
        if (live) {
            const unsigned long long s = (unsigned long long)(rp[v + 1] - rp[v]) *
                                         (unsigned long long)(rrp[v + 1] - rrp[v]);
            key = (min(s, 0xFFFFFFFFull) << 32) | (0xFFFFFFFFull - (uint64_t)v);
        }
        const uint64_t L0 = __shfl_sync(kFull, L, __ffs(bal) - 1);
        if (__all_sync(kFull, !live || L == L0)) {
            unsigned long long k = key;
            unsigned m = live ? (unsigned)v : kFull;
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) {
                k = max(k, __shfl_xor_sync(kFull, k, o));
                m = min(m, __shfl_xor_sync(kFull, m, o));
            }
            if (lane == 0) {
                atomicMax(&pk[L0], k);
                atomicAdd(&sz[L0], (unsigned)__popc(bal));
                atomicMin(&mn[L0], m);
            }
        } else if (live) {
            atomicMax(&pk[L], key);
            atomicAdd(&sz[L], 1u);
            atomicMin(&mn[L], (unsigned)v);
        }
    }
}

// Prune parts that cannot beat the best component so far; queue the pivots
// of the others (both searches start from them).
__global__ void k_scc_seed(int64_t n, uint64_t *lab, const unsigned long long *pk,
                           const unsigned *sz, const unsigned *mn,
                           const unsigned long long *best, unsigned *fw, unsigned *bw,
                           int32_t *q, unsigned long long *qn)
{
    const unsigned long long b = *best;
    const unsigned bs = (unsigned)(b >> 32);
    const unsigned bm = (unsigned)(0xFFFFFFFFull - (b & 0xFFFFFFFFull));
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t L = lab[v];
        if (L == kDeadLab) continue;
        if (sz[L] < bs || (sz[L] == bs && mn[L] > bm)) {
            lab[v] = kDeadLab;
            continue;
        }
        if ((uint32_t)pk[L] == (uint32_t)(0xFFFFFFFFull - (uint64_t)v)) {
            fw[v] = 1u;
            bw[v] = 1u;
            q[atomicAdd(qn, 1ull)] = (int32_t)v;
        }
    }
}

// One level of the confined searches: a warp per queued node, a lane per
// arc; the first to reach a node of the same part queues it (one queue
// reservation per warp step).
__global__ void k_scc_bfs(const int64_t *rp, const int32_t *col, const uint64_t *lab,
                          const int32_t *qin, int64_t nin, int32_t *qout,
                          unsigned long long *nout, unsigned *vis)
{
    const int lane = threadIdx.x & 31;
    for (int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; t < nin;
         t += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int32_t u = qin[t];
        const uint64_t L = lab[u];
        const int64_t end = rp[u + 1];
        for (int64_t e0 = rp[u]; e0 < end; e0 += 32) {
            const int64_t e = e0 + lane;
            int32_t x = -1;
            bool push = false;
            if (e < end) {
                x = col[e];
                push = lab[x] == L && vis[x] == 0u && atomicExch(&vis[x], 1u) == 0u;
            }
            const unsigned bal = __ballot_sync(kFull, push);
            if (!bal) continue;
            unsigned long long at = 0;
            if (lane == __ffs(bal) - 1) at = atomicAdd(nout, (unsigned long long)__popc(bal));
            at = __shfl_sync(kFull, at, __ffs(bal) - 1);
            if (push) qout[at + __popc(bal & ((1u << lane) - 1u))] = x;
        }
    }
}

// Split every searched part: both ways -> the pivot's component (dead),
// forward only -> label p, backward only -> n + p, neither -> unchanged.
__global__ void k_scc_split(int64_t n, uint64_t *lab, const unsigned long long *pk,
                            unsigned *fw, unsigned *bw, int32_t *comp, unsigned *csz,
                            unsigned *cmn)
{
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n;
         base += stride) {
        const int64_t v = base + lane;
        const uint64_t L = v < n ? lab[v] : kDeadLab;
        bool in_s = false;
        uint32_t p = 0;
        if (L != kDeadLab) {
            p = (uint32_t)(0xFFFFFFFFull - (pk[L] & 0xFFFFFFFFull));
            const bool f = fw[v] != 0u, b = bw[v] != 0u;
            if (f && b) {
                in_s = true;
                comp[v] = (int32_t)p;
                lab[v] = kDeadLab;
            } else if (f) {
                lab[v] = p;
            } else if (b) {
                lab[v] = (uint64_t)n + p;
            }
            if (f) fw[v] = 0u;
            if (b) bw[v] = 0u;
        }
        const unsigned bal = __ballot_sync(kFull, in_s);
        if (!bal) continue;
        const uint32_t p0 = __shfl_sync(kFull, p, __ffs(bal) - 1);
        if (__all_sync(kFull, !in_s || p == p0)) {
            if (lane == __ffs(bal) - 1) {
                atomicAdd(&csz[p0], (unsigned)__popc(bal));
                atomicMin(&cmn[p0], (unsigned)v);  // lowest member lane: smallest id
            }
        } else if (in_s) {
            atomicAdd(&csz[p], 1u);
            atomicMin(&cmn[p], (unsigned)v);
        }
    }
}

__global__ void k_scc_best(int64_t n, const unsigned *csz, const unsigned *cmn,
                           unsigned long long *best)
{
    unsigned long long k = 0;
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x)
        if (csz[v]) k = max(k, best_key(csz[v], cmn[v]));
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) k = max(k, __shfl_xor_sync(kFull, k, o));
    if ((threadIdx.x & 31) == 0 && k) atomicMax(best, k);
}

__global__ void k_comp_flags(const int32_t *comp, int64_t n, int32_t c, uint64_t *flags)
{
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x)
        flags[v] = comp[v] == c ? 1 : 0;
}

// Kept nodes: new ids, and per kept row the arcs whose head is kept too (a
// warp per row).
__global__ void k_kept_arcs(const int64_t *rp, const int32_t *col, const uint64_t *flags,
                            const uint64_t *pos, int64_t n, uint64_t *deg, int32_t *newid,
                            int32_t *old_id)
{
    const int lane = threadIdx.x & 31;
    for (int64_t v = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; v < n;
         v += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        if (!flags[v]) {
            if (lane == 0) newid[v] = -1;
            continue;
        }
        unsigned c = 0;
        for (int64_t e = rp[v] + lane; e < rp[v + 1]; e += 32) c += flags[col[e]] ? 1u : 0u;
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
        if (lane == 0) {
            deg[pos[v]] = c;
            newid[v] = (int32_t)pos[v];
            old_id[pos[v]] = (int32_t)v;
        }
    }
}

// Kept rows with their kept arcs, in order (ballot compaction per 32 arcs).
__global__ void k_rewrite_kept(const int64_t *rp, const int32_t *col, const uint32_t *w,
                               const uint64_t *flags, const int32_t *old_id,
                               const int32_t *newid, const uint64_t *nrp, int64_t nk,
                               int32_t *ncol, uint32_t *nw)
{
    const int lane = threadIdx.x & 31;
    for (int64_t x = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; x < nk;
         x += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int32_t v = old_id[x];
        int64_t o = (int64_t)nrp[x];
        for (int64_t e0 = rp[v]; e0 < rp[v + 1]; e0 += 32) {
            const int64_t e = e0 + lane;
            const bool in = e < rp[v + 1];
            const int32_t u = in ? col[e] : 0;
            const bool keep = in && flags[u];
            const unsigned bal = __ballot_sync(0xFFFFFFFFu, keep);
            if (keep) {
                const int64_t q = o + __popc(bal & ((1u << lane) - 1u));
                ncol[q] = newid[u];
                if (w) nw[q] = w[e];
            }
            o += __popc(bal);
        }
    }
}

__global__ void k_u64_to_i64(const uint64_t *in, int64_t n, int64_t *out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (int64_t)in[i];
}

int gsz(int64_t n) { return (int)std::min<int64_t>(std::max<int64_t>(1, (n + 255) / 256), 152 * 32); }

struct Buf {
    void *p = nullptr;
    ~Buf() { if (p) cudaFree(p); }
    template <class T> T *as() { return static_cast<T *>(p); }
    int alloc(size_t bytes)
    {
        if (cudaMalloc(&p, bytes ? bytes : 16) != cudaSuccess) {
            cudaGetLastError();
            p = nullptr;
            return CC_ERR_OOM;
        }
        return CC_OK;
    }
};

#define G_RC(x)                      \
    do {                             \
        int r_ = (x);                \
        if (r_ != CC_OK) return r_;  \
    } while (0)
#define G_CK(x)                                          \
    do {                                                 \
        const cudaError_t e_ = (x);                      \
        if (e_ != cudaSuccess) {                         \
            note_cuda_error(e_, __FILE__, __LINE__);     \
            cudaGetLastError();                          \
            return CC_ERR_CUDA;                          \
        }                                                \
    } while (0)

// Exclusive scan of n uint64 values (in -> out, may alias), *total (device):
// the sum.  sums: one entry per 1,024 values and one more.  Stream work only.
int64_t scan_tiles(int64_t n) { return (n + kThreads * 4 - 1) / (kThreads * 4); }

void scan_rounds(const uint64_t *in, uint64_t *out, int64_t n, uint64_t *sums, uint64_t *total,
                 cudaStream_t st)
{
    const int64_t nb = scan_tiles(n);
    if (n > 0) k_tile_sums<<<(int)nb, kThreads, 0, st>>>(in, n, sums);
    k_scan_sums<<<1, 1024, 0, st>>>(sums, nb, total);
    if (n > 0) k_tile_scan<<<(int)nb, kThreads, 0, st>>>(in, n, sums, out);
}

// The same with its own scratch, returning the total; synchronises.
int scan_u64(const uint64_t *in, uint64_t *out, int64_t n, uint64_t *total, cudaStream_t st)
{
    const int64_t nb = scan_tiles(n);
    Buf sums;
    G_RC(sums.alloc((size_t)(nb + 1) * 8));
    scan_rounds(in, out, n, sums.as<uint64_t>(), sums.as<uint64_t>() + nb, st);
    G_CK(cudaMemcpyAsync(total, sums.as<uint64_t>() + nb, 8, cudaMemcpyDeviceToHost, st));
    G_CK(cudaStreamSynchronize(st));
    return CC_OK;
}

// Scratch of radix_rounds for n keys, in bytes.
size_t radix_scratch(int64_t n)
{
    const int64_t ntiles = (n + kTile - 1) / kTile;
    return (size_t)kRadix * (std::max<int64_t>(ntiles, 1) + 1) * 4;
}

// Stable LSD radix sort of (keys, vals) by the bits [lo, hi) of the keys
// (vals null: keys alone); *in_tmp: the result is in tk / tv.  Stream work
// only.
int radix_rounds(uint64_t *keys, uint32_t *vals, int64_t n, int lo, int hi, uint64_t *tk,
                 uint32_t *tv, uint32_t *scratch, cudaStream_t st, bool *in_tmp)
{
    *in_tmp = false;
    if (n <= 0) return CC_OK;
    const int ntiles = (int)((n + kTile - 1) / kTile);
    uint32_t *counts = scratch, *tot = scratch + (size_t)kRadix * ntiles;
    for (int shift = lo; shift < hi; shift += 8) {
        const int nb = std::min(8, hi - shift);
        k_digit_hist<<<ntiles, kThreads, 0, st>>>(keys, n, shift, nb, counts, ntiles);
        k_digit_rows<<<kRadix, kThreads, 0, st>>>(counts, ntiles, tot);
        if (vals)
            k_digit_scatter<true><<<ntiles, kThreads, 0, st>>>(keys, vals, n, shift, nb, counts,
                                                               tot, ntiles, tk, tv);
        else
            k_digit_scatter<false><<<ntiles, kThreads, 0, st>>>(keys, nullptr, n, shift, nb,
                                                                counts, tot, ntiles, tk, nullptr);
        std::swap(keys, tk);
        std::swap(vals, tv);
        *in_tmp = !*in_tmp;
    }
    G_CK(cudaGetLastError());
    return CC_OK;
}

// The same over the low `bits` bits with its own scratch; synchronises.
int radix_sort(uint64_t *keys, uint32_t *vals, int64_t n, int bits, uint64_t *tk,
               uint32_t *tv, cudaStream_t st, bool *in_tmp)
{
    Buf scratch;
    G_RC(scratch.alloc(radix_scratch(n)));
    G_RC(radix_rounds(keys, vals, n, 0, bits, tk, tv, scratch.as<uint32_t>(), st, in_tmp));
    G_CK(cudaStreamSynchronize(st));
    return CC_OK;
}


}  // namespace

int degree_order(int64_t n, const int64_t *rp, int32_t *order, int64_t (&counts)[5])
{
    Buf k0, k1, v0, v1, c;
    G_RC(k0.alloc(n * 8));
    G_RC(k1.alloc(n * 8));
    G_RC(v0.alloc(n * 4));
    G_RC(v1.alloc(n * 4));
    G_RC(c.alloc(40 + radix_scratch(n)));
    cudaStream_t st = 0;
    G_CK(cudaMemsetAsync(c.p, 0, 40, st));
    k_degree_keys<<<std::min(gsz(n), 152 * 4), 256, 0, st>>>(
        rp, n, k0.as<uint64_t>(), v0.as<uint32_t>(), c.as<unsigned long long>());
    bool tmp = false;
    int bits = 1;
    while ((1 << bits) < kMediumMaxDeg + 2) ++bits;
    G_RC(radix_rounds(k0.as<uint64_t>(), v0.as<uint32_t>(), n, 0, bits, k1.as<uint64_t>(),
                      v1.as<uint32_t>(), c.as<uint32_t>() + 10, st, &tmp));
    G_CK(cudaMemcpyAsync(order, tmp ? v1.p : v0.p, n * 4, cudaMemcpyDeviceToDevice, st));
    unsigned long long h[5];
    G_CK(cudaMemcpyAsync(h, c.p, 40, cudaMemcpyDeviceToHost, st));
    G_CK(cudaStreamSynchronize(st));
    for (int i = 0; i < 5; ++i) counts[i] = (int64_t)h[i];
    return CC_OK;
}

int heavy_chunks(const int32_t *H, int64_t nH, const int64_t *rp, int32_t *Hn, int64_t *Hb)
{
    if (nH > 0) k_heavy_chunks<<<1, kThreads>>>(H, nH, rp, Hn, Hb);
    G_CK(cudaGetLastError());
    return CC_OK;
}

int device_scan_u64(const uint64_t *in, uint64_t *out, int64_t n, uint64_t *total,
                    cudaStream_t st)
{
    return scan_u64(in, out, n, total, st);
}

int device_radix_sort(uint64_t *keys, uint32_t *vals, int64_t n, int bits, uint64_t *tk,
                      uint32_t *tv, cudaStream_t st, bool *in_tmp)
{
    return radix_sort(keys, vals, n, bits, tk, tv, st, in_tmp);
}

// Undirected graph to CSR on the device (see the top of this file).  On
// success the device buffers rp / col / w (w only when lengths are given)
// are owned by the caller (cudaFree); old_id holds a host copy.  Every
// temporary comes from one allocation.
int build_csr_device(int64_t n, int64_t m, const uint32_t *h_src, const uint32_t *h_dst,
                     const uint32_t *h_w, bool keep_component, DeviceCSR &out)
{
    if (n < 2 || m < 0 || (m > 0 && (!h_src || !h_dst))) return CC_ERR_ARG;
    if (n > 0x7FFFFFFFLL || 2 * m > 0x7FFFFFFFLL) return CC_ERR_TOO_LARGE;
    cudaStream_t st = 0;
    int b = 1;
    while ((1ll << b) < n) ++b;
    const int64_t ntile = (m + kEdgeTile - 1) / kEdgeTile;
    const int64_t nscan = scan_tiles(std::max<int64_t>(n + 1, 1)) + 1;
    Arena A;
    for (int pass = 0; pass < 2; ++pass) {  // sizes, then addresses
        if (pass) G_RC(A.allocate());
        A.src = A.take<uint32_t>(m);
        A.dst = A.take<uint32_t>(m);
        A.w = A.take<uint32_t>(h_w ? m : 0);
        A.k0 = A.take<uint64_t>(m);
        A.k1 = A.take<uint64_t>(m);
        A.v0 = A.take<uint32_t>(h_w ? m : 0);
        A.v1 = A.take<uint32_t>(h_w ? m : 0);
        A.radix = A.take<uint32_t>(radix_scratch(m) / 4);
        A.tiles = A.take<uint64_t>(ntile + 2);
        A.parent = A.take<int32_t>(n);
        A.size = A.take<uint32_t>(n);
        A.newid = A.take<int32_t>(n);
        A.oldid = A.take<int32_t>(n);
        A.flag = A.take<uint64_t>(n + 1);
        A.pos = A.take<uint64_t>(n + 1);
        A.scan = A.take<uint64_t>(nscan);
        A.fs = A.take<uint32_t>(n + 2);
        A.rs = A.take<uint32_t>(n + 2);
        A.info = A.take<BuildInfo>(1);
    }
    if (m > 0) {
        G_CK(cudaMemcpyAsync(A.src, h_src, m * 4, cudaMemcpyHostToDevice, st));
        G_CK(cudaMemcpyAsync(A.dst, h_dst, m * 4, cudaMemcpyHostToDevice, st));
        if (h_w) G_CK(cudaMemcpyAsync(A.w, h_w, m * 4, cudaMemcpyHostToDevice, st));
    }
    G_CK(cudaMemsetAsync(A.info, 0, sizeof(BuildInfo), st));
    // 1. edges as (smaller, larger) keys, loops as the largest key of all
    if (m > 0)
        k_pack_edges<<<gsz(m), 256, 0, st>>>(A.src, A.dst, h_w ? A.w : nullptr, m, n, b, A.k0,
                                             h_w ? A.v0 : nullptr, A.info);
    // 2. sorted
    bool tmp = false;
    G_RC(radix_rounds(A.k0, h_w ? A.v0 : nullptr, m, 0, 2 * b, A.k1, h_w ? A.v1 : nullptr,
                      A.radix, st, &tmp));
    uint64_t *ks = tmp ? A.k1 : A.k0, *ko = tmp ? A.k0 : A.k1;
    uint32_t *vs = tmp ? A.v1 : A.v0, *vo = tmp ? A.v0 : A.v1;
    // 3. parallel edges merged (smallest length)
    if (m > 0) {
        k_runs_count<<<(int)ntile, kThreads, 0, st>>>(ks, A.info, A.tiles);
        k_scan_sums<<<1, 1024, 0, st>>>(A.tiles, ntile, &A.info->edges);
        k_runs_write<<<(int)ntile, kThreads, 0, st>>>(ks, h_w ? vs : nullptr, A.info, A.tiles, ko,
                                                      vo);
    }
    std::swap(ks, ko);
    std::swap(vs, vo);  // ks, vs: the merged edges by (smaller, larger)
    // 4. components: the first two edges of each node, then the others, most
    //    of whose ends share a root by then; the largest one's nodes
    if (keep_component) {
        k_iota32<<<gsz(n), 256, 0, st>>>(A.parent, n);
        for (int which = 0; which < 3 && m > 0; ++which) {
            k_link<<<gsz(m), 256, 0, st>>>(ks, A.info, b, which, A.parent);
            k_compress<<<gsz(n), 256, 0, st>>>(A.parent, n);
        }
        G_CK(cudaMemsetAsync(A.size, 0, n * 4, st));
        k_label_count<<<gsz(n), 256, 0, st>>>(A.parent, n, A.size);
        k_pick<<<std::min(gsz(n), 152 * 2), 256, 0, st>>>(A.size, n, &A.info->best);
    }
    k_keep_flags<<<gsz(n), 256, 0, st>>>(keep_component ? A.parent : nullptr, n, A.info, A.flag);
    scan_rounds(A.flag, A.pos, n, A.scan, &A.info->nodes, st);
    k_new_ids<<<gsz(n), 256, 0, st>>>(A.flag, A.pos, n, A.newid, A.oldid);
    // 5. the other way round: sorted by the larger end (the smaller ones stay
    //    in order)
    if (m > 0) {
        k_row_starts<<<gsz(m + 1), 256, 0, st>>>(ks, A.info, n, b, A.fs);
        k_swap_ends<<<gsz(m), 256, 0, st>>>(ks, h_w ? vs : nullptr, A.info, m, b, ko, vo);
    } else {
        G_CK(cudaMemsetAsync(A.fs, 0, (n + 1) * 4, st));
    }
    // keys past the merged ones are the largest of all and sort to the end
    uint64_t *rk = ko, *rt = nullptr;
    uint32_t *rv = vo, *rtv = nullptr;
    // the scratch of this sort: the arrays of the input, no longer needed
    // (8 bytes an edge), and of the lengths
    rt = reinterpret_cast<uint64_t *>(A.src);
    rtv = A.w;
    G_RC(radix_rounds(rk, h_w ? rv : nullptr, m, b, 2 * b, rt, h_w ? rtv : nullptr, A.radix, st,
                      &tmp));
    if (tmp) {
        std::swap(rk, rt);
        std::swap(rv, rtv);
    }
    if (m > 0)
        k_row_starts<<<gsz(m + 1), 256, 0, st>>>(rk, A.info, n, b, A.rs);
    else
        G_CK(cudaMemsetAsync(A.rs, 0, (n + 1) * 4, st));
    // 6. row offsets of the kept nodes
    G_CK(cudaMemsetAsync(A.flag, 0, n * 8, st));
    k_kept_deg<<<gsz(n), 256, 0, st>>>(A.fs, A.rs, A.newid, n, A.flag);
    scan_rounds(A.flag, A.pos, n, A.scan, &A.info->arcs, st);
    BuildInfo h;
    G_CK(cudaMemcpyAsync(&h, A.info, sizeof(h), cudaMemcpyDeviceToHost, st));
    G_CK(cudaStreamSynchronize(st));
    G_CK(cudaGetLastError());
    if (h.err) return h.err;
    const int64_t nk = (int64_t)h.nodes, arcs = (int64_t)h.arcs;
    if (keep_component && nk < 2) return CC_ERR_GRAPH;
    Buf rp, col, nw;
    G_RC(rp.alloc((nk + 1) * 8));
    G_RC(col.alloc(std::max<int64_t>(arcs, 1) * 4));
    if (h_w) G_RC(nw.alloc(std::max<int64_t>(arcs, 1) * 4));
    k_row_ptr_kept<<<gsz(nk + 1), 256, 0, st>>>(A.pos, nk, arcs, rp.as<int64_t>());
    // 7. both halves of every row: the smaller neighbours (by the larger
    //    end), then the larger ones, each ascending
    if (m > 0)
        k_fill_rows<<<gsz((int64_t)h.edges), 256, 0, st>>>(
            ks, rk, h_w ? vs : nullptr, h_w ? rv : nullptr, (int64_t)h.edges, b, A.fs, A.rs,
            A.newid, rp.as<int64_t>(), col.as<int32_t>(), h_w ? nw.as<uint32_t>() : nullptr);
    out.old_id.resize(nk);
    G_CK(cudaMemcpyAsync(out.old_id.data(), A.oldid, nk * 4, cudaMemcpyDeviceToHost, st));
    G_CK(cudaStreamSynchronize(st));
    G_CK(cudaGetLastError());
    out.n = nk;
    out.arcs = arcs;
    std::swap(out.rp, rp.p);
    std::swap(out.col, col.p);
    if (h_w) std::swap(out.w, nw.p);
    return CC_OK;
}

// Sorted, merged arcs (keys tail << b | head, lengths) -> CSR over n nodes.
static int csr_from_sorted(const uint64_t *keys, const uint32_t *vals, int64_t a, int64_t n, int b,
                           bool weighted, Buf &rp, Buf &col, Buf &w, cudaStream_t st)
{
    G_RC(rp.alloc((n + 1) * 8));
    G_RC(col.alloc(std::max<int64_t>(a, 1) * 4));
    k_row_ptr<<<gsz(a + 1), 256, 0, st>>>(keys, a, n, b, rp.as<int64_t>());
    if (a > 0) k_heads<<<gsz(a), 256, 0, st>>>(keys, a, b, col.as<int32_t>());
    if (weighted) {
        G_RC(w.alloc(std::max<int64_t>(a, 1) * 4));
        if (a > 0) G_CK(cudaMemcpyAsync(w.p, vals, a * 4, cudaMemcpyDeviceToDevice, st));
    }
    return CC_OK;
}

// Rows of the kept nodes with their kept arcs, renumbered.
static int filter_csr(const int64_t *rp, const int32_t *col, const uint32_t *w, int64_t n,
                      const uint64_t *flags, const uint64_t *pos, int64_t nk, Buf &newid,
                      Buf &oldid, DeviceCSR &out, cudaStream_t st)
{
    Buf degs, nrp, ncol, nw;
    G_RC(degs.alloc((nk + 1) * 8));
    k_kept_arcs<<<gsz(n * 32), 256, 0, st>>>(rp, col, flags, pos, n, degs.as<uint64_t>(),
                                             newid.as<int32_t>(), oldid.as<int32_t>());
    uint64_t arcs = 0;
    G_RC(scan_u64(degs.as<uint64_t>(), degs.as<uint64_t>(), nk, &arcs, st));
    G_CK(cudaMemcpy(degs.as<uint64_t>() + nk, &arcs, 8, cudaMemcpyHostToDevice));
    G_RC(nrp.alloc((nk + 1) * 8));
    G_RC(ncol.alloc(std::max<uint64_t>(arcs, 1) * 4));
    if (w) G_RC(nw.alloc(std::max<uint64_t>(arcs, 1) * 4));
    k_u64_to_i64<<<gsz(nk + 1), 256, 0, st>>>(degs.as<uint64_t>(), nk + 1, nrp.as<int64_t>());
    k_rewrite_kept<<<gsz(nk * 32), 256, 0, st>>>(rp, col, w, flags, oldid.as<int32_t>(),
                                                 newid.as<int32_t>(), degs.as<uint64_t>(), nk,
                                                 ncol.as<int32_t>(), w ? nw.as<uint32_t>() : nullptr);
    out.n = nk;
    out.arcs = (int64_t)arcs;
    std::swap(out.rp, nrp.p);
    std::swap(out.col, ncol.p);
    if (w) std::swap(out.w, nw.p);
    return CC_OK;
}

// Largest strongly connected component (see the kernels above): flags[v] =
// 1 for its nodes, *kept = its size.  Ties go to the component holding the
// smallest id.
static int largest_scc(const int64_t *rp, const int32_t *col, const int64_t *rrp,
                       const int32_t *rcol, int64_t n, uint64_t *flags, int64_t *kept,
                       cudaStream_t st)
{
    Buf parent, lab, comp, fw, bw, qp, q0, q1, pk, sz, mn, csz, cmn, ctr;
    const int64_t nl = 3 * n;  // label space
    G_RC(parent.alloc(n * 4));
    G_RC(lab.alloc(n * 8));
    G_RC(comp.alloc(n * 4));
    G_RC(fw.alloc(n * 4));
    G_RC(bw.alloc(n * 4));
    G_RC(qp.alloc(n * 4));
    G_RC(q0.alloc(n * 4));
    G_RC(q1.alloc(n * 4));
    G_RC(pk.alloc(nl * 8));
    G_RC(sz.alloc(nl * 4));
    G_RC(mn.alloc(nl * 4));
    G_RC(csz.alloc(n * 4));
    G_RC(cmn.alloc(n * 4));
    G_RC(ctr.alloc(3 * 8));  // best, removed, queue count
    unsigned long long *best = ctr.as<unsigned long long>(), *removed = best + 1,
                       *qn = best + 2;
    // weak components by union-find over the arcs of G and of G^T
    k_iota32<<<gsz(n), 256, 0, st>>>(parent.as<int32_t>(), n);
    k_hook<<<gsz(n * 32), 256, 0, st>>>(rp, col, n, parent.as<int32_t>());
    k_hook<<<gsz(n * 32), 256, 0, st>>>(rrp, rcol, n, parent.as<int32_t>());
    k_scc_init<<<gsz(n), 256, 0, st>>>(parent.as<int32_t>(), n, lab.as<uint64_t>(),
                                       comp.as<int32_t>());
    G_CK(cudaMemsetAsync(fw.p, 0, n * 4, st));
    G_CK(cudaMemsetAsync(bw.p, 0, n * 4, st));
    G_CK(cudaMemsetAsync(csz.p, 0, n * 4, st));
    G_CK(cudaMemsetAsync(cmn.p, 0xFF, n * 4, st));
    G_CK(cudaMemsetAsync(best, 0, 8, st));
    uint64_t *L = lab.as<uint64_t>();
    for (;;) {
        // trim while it removes nodes (at most 16 sweeps a round; the
        // searches settle whatever is left)
        for (int it = 0; it < 16; ++it) {
            G_CK(cudaMemsetAsync(removed, 0, 8, st));
            k_scc_trim<<<gsz(n * 32), 256, 0, st>>>(rp, col, rrp, rcol, n, L,
                                                    comp.as<int32_t>(), removed, best);
            unsigned long long h = 0;
            G_CK(cudaMemcpyAsync(&h, removed, 8, cudaMemcpyDeviceToHost, st));
            G_CK(cudaStreamSynchronize(st));
            if (h == 0) break;
        }
        G_CK(cudaMemsetAsync(pk.p, 0, nl * 8, st));
        G_CK(cudaMemsetAsync(sz.p, 0, nl * 4, st));
        G_CK(cudaMemsetAsync(mn.p, 0xFF, nl * 4, st));
        G_CK(cudaMemsetAsync(qn, 0, 8, st));
        k_scc_stats<<<gsz(n), 256, 0, st>>>(rp, rrp, n, L, pk.as<unsigned long long>(),
                                            sz.as<unsigned>(), mn.as<unsigned>());
        k_scc_seed<<<gsz(n), 256, 0, st>>>(n, L, pk.as<unsigned long long>(), sz.as<unsigned>(),
                                           mn.as<unsigned>(), best, fw.as<unsigned>(),
                                           bw.as<unsigned>(), qp.as<int32_t>(), qn);
        unsigned long long npiv = 0;
        G_CK(cudaMemcpyAsync(&npiv, qn, 8, cudaMemcpyDeviceToHost, st));
        G_CK(cudaStreamSynchronize(st));
        if (npiv == 0) break;  // every part settled or pruned
        for (int dir = 0; dir < 2; ++dir) {
            const int64_t *r = dir ? rrp : rp;
            const int32_t *c = dir ? rcol : col;
            unsigned *vis = dir ? bw.as<unsigned>() : fw.as<unsigned>();
            int32_t *qin = q0.as<int32_t>(), *qout = q1.as<int32_t>();
            G_CK(cudaMemcpyAsync(qin, qp.p, npiv * 4, cudaMemcpyDeviceToDevice, st));
            int64_t nin = (int64_t)npiv;
            while (nin > 0) {
                G_CK(cudaMemsetAsync(qn, 0, 8, st));
                k_scc_bfs<<<gsz(nin * 32), 256, 0, st>>>(r, c, L, qin, nin, qout, qn, vis);
                unsigned long long h = 0;
                G_CK(cudaMemcpyAsync(&h, qn, 8, cudaMemcpyDeviceToHost, st));
                G_CK(cudaStreamSynchronize(st));
                nin = (int64_t)h;
                std::swap(qin, qout);
            }
        }
        k_scc_split<<<gsz(n), 256, 0, st>>>(n, L, pk.as<unsigned long long>(), fw.as<unsigned>(),
                                            bw.as<unsigned>(), comp.as<int32_t>(),
                                            csz.as<unsigned>(), cmn.as<unsigned>());
        k_scc_best<<<gsz(n), 256, 0, st>>>(n, csz.as<unsigned>(), cmn.as<unsigned>(), best);
    }
    unsigned long long hb = 0;
    G_CK(cudaMemcpyAsync(&hb, best, 8, cudaMemcpyDeviceToHost, st));
    G_CK(cudaStreamSynchronize(st));
    const int64_t size = (int64_t)(hb >> 32);
    const int64_t min_id = (int64_t)(0xFFFFFFFFull - (hb & 0xFFFFFFFFull));
    if (size < 2 || min_id >= n) {
        *kept = size;
        return CC_OK;
    }
    int32_t c = -1;
    G_CK(cudaMemcpyAsync(&c, comp.as<int32_t>() + min_id, 4, cudaMemcpyDeviceToHost, st));
    G_CK(cudaStreamSynchronize(st));
    k_comp_flags<<<gsz(n), 256, 0, st>>>(comp.as<int32_t>(), n, c, flags);
    *kept = size;
    return CC_OK;
}

int build_csr_device_directed(int64_t n, int64_t m, const uint32_t *h_src, const uint32_t *h_dst,
                              const uint32_t *h_w, bool keep_component, DeviceCSR &F,
                              DeviceCSR &R)
{
    if (n < 2 || m < 0 || (m > 0 && (!h_src || !h_dst))) return CC_ERR_ARG;
    if (n > 0x7FFFFFFFLL || m > 0x7FFFFFFFLL) return CC_ERR_TOO_LARGE;
    cudaStream_t st = 0;
    int b = 1;
    while ((1ll << b) < n) ++b;
    Buf dsrc, ddst, dw, k0, v0, k1, v1, fl, pos, err;
    G_RC(dsrc.alloc(m * 4));
    G_RC(ddst.alloc(m * 4));
    if (h_w) G_RC(dw.alloc(m * 4));
    G_RC(k0.alloc(std::max<int64_t>(m, 1) * 8));
    G_RC(v0.alloc(std::max<int64_t>(m, 1) * 4));
    G_RC(k1.alloc(std::max<int64_t>(m, 1) * 8));
    G_RC(v1.alloc(std::max<int64_t>(m, 1) * 4));
    const int64_t FL = std::max<int64_t>(m, n) + 1;
    G_RC(fl.alloc(FL * 8));
    G_RC(pos.alloc(FL * 8));
    G_RC(err.alloc(4));
    if (m > 0) {
        G_CK(cudaMemcpy(dsrc.p, h_src, m * 4, cudaMemcpyHostToDevice));
        G_CK(cudaMemcpy(ddst.p, h_dst, m * 4, cudaMemcpyHostToDevice));
        if (h_w) G_CK(cudaMemcpy(dw.p, h_w, m * 4, cudaMemcpyHostToDevice));
    }
    G_CK(cudaMemset(err.p, 0, 4));
    // 1. arcs one way, self-loops dropped; sorted by (tail, head); parallel
    //    arcs merged (smallest length)
    if (m > 0)
        k_make_arcs<<<gsz(m), 256, 0, st>>>(dsrc.as<uint32_t>(), ddst.as<uint32_t>(),
                                            h_w ? dw.as<uint32_t>() : nullptr, m, n, b,
                                            k0.as<uint64_t>(), v0.as<uint32_t>(),
                                            fl.as<uint64_t>(), err.as<int>());
    int herr = 0;
    G_CK(cudaMemcpy(&herr, err.p, 4, cudaMemcpyDeviceToHost));
    if (herr) return herr;
    uint64_t A1 = 0;
    G_RC(scan_u64(fl.as<uint64_t>(), pos.as<uint64_t>(), m, &A1, st));
    if (m > 0)
        k_compact<<<gsz(m), 256, 0, st>>>(k0.as<uint64_t>(), v0.as<uint32_t>(), fl.as<uint64_t>(),
                                          pos.as<uint64_t>(), m, k1.as<uint64_t>(),
                                          v1.as<uint32_t>());
    bool in_tmp = false;
    if (A1 > 0)
        G_RC(radix_sort(k1.as<uint64_t>(), v1.as<uint32_t>(), (int64_t)A1, 2 * b,
                        k0.as<uint64_t>(), v0.as<uint32_t>(), st, &in_tmp));
    uint64_t *ks = in_tmp ? k0.as<uint64_t>() : k1.as<uint64_t>();
    uint32_t *vs = in_tmp ? v0.as<uint32_t>() : v1.as<uint32_t>();
    uint64_t *ko = in_tmp ? k1.as<uint64_t>() : k0.as<uint64_t>();
    uint32_t *vo = in_tmp ? v1.as<uint32_t>() : v0.as<uint32_t>();
    uint64_t A2 = 0;
    if (A1 > 0) {
        k_first_of_run<<<gsz(A1), 256, 0, st>>>(ks, (int64_t)A1, fl.as<uint64_t>());
        k_run_min<<<gsz(A1), 256, 0, st>>>(ks, vs, fl.as<uint64_t>(), (int64_t)A1);
        G_RC(scan_u64(fl.as<uint64_t>(), pos.as<uint64_t>(), (int64_t)A1, &A2, st));
        k_compact<<<gsz(A1), 256, 0, st>>>(ks, vs, fl.as<uint64_t>(), pos.as<uint64_t>(),
                                           (int64_t)A1, ko, vo);
    }
    // 2. forward CSR (G) and reverse CSR (G^T, from the swapped keys)
    Buf frp, fcol, fw, rrp, rcol, rw;
    G_RC(csr_from_sorted(ko, vo, (int64_t)A2, n, b, h_w != nullptr, frp, fcol, fw, st));
    if (A2 > 0) {
        k_swap_keys<<<gsz(A2), 256, 0, st>>>(ko, vo, (int64_t)A2, b, ks, vs);
        G_RC(radix_sort(ks, vs, (int64_t)A2, 2 * b, ko, vo, st, &in_tmp));
    }
    const uint64_t *rks = (A2 > 0 && in_tmp) ? ko : ks;
    const uint32_t *rvs = (A2 > 0 && in_tmp) ? vo : vs;
    G_RC(csr_from_sorted(rks, rvs, (int64_t)A2, n, b, h_w != nullptr, rrp, rcol, rw, st));
    // 3. the largest strongly connected component (largest_scc), unless
    //    every node is kept
    if (!keep_component) {
        std::vector<int32_t> ids(n);
        for (int64_t v = 0; v < n; ++v) ids[v] = (int32_t)v;
        for (DeviceCSR *o : {&F, &R}) {
            o->n = n;
            o->arcs = (int64_t)A2;
            o->old_id = ids;
        }
        std::swap(F.rp, frp.p); std::swap(F.col, fcol.p); if (h_w) std::swap(F.w, fw.p);
        std::swap(R.rp, rrp.p); std::swap(R.col, rcol.p); if (h_w) std::swap(R.w, rw.p);
        G_CK(cudaDeviceSynchronize());
        return CC_OK;
    }
    int64_t nk = 0;
    G_RC(largest_scc(frp.as<int64_t>(), fcol.as<int32_t>(), rrp.as<int64_t>(),
                     rcol.as<int32_t>(), n, fl.as<uint64_t>(), &nk, st));
    if (nk < 2) return CC_ERR_GRAPH;
    uint64_t kept = 0;
    G_RC(scan_u64(fl.as<uint64_t>(), pos.as<uint64_t>(), n, &kept, st));
    if ((int64_t)kept != nk) return CC_ERR_CUDA;  // flags disagree with the component size
    // 4. renumber the kept nodes (increasing original id) and keep the arcs
    //    between them, in G and in G^T
    Buf newid, oldid, newid2, oldid2;
    G_RC(newid.alloc(n * 4));
    G_RC(oldid.alloc(nk * 4));
    G_RC(newid2.alloc(n * 4));
    G_RC(oldid2.alloc(nk * 4));
    G_RC(filter_csr(frp.as<int64_t>(), fcol.as<int32_t>(), h_w ? fw.as<uint32_t>() : nullptr, n,
                    fl.as<uint64_t>(), pos.as<uint64_t>(), nk, newid, oldid, F, st));
    G_RC(filter_csr(rrp.as<int64_t>(), rcol.as<int32_t>(), h_w ? rw.as<uint32_t>() : nullptr, n,
                    fl.as<uint64_t>(), pos.as<uint64_t>(), nk, newid2, oldid2, R, st));
    F.old_id.resize(nk);
    G_CK(cudaMemcpy(F.old_id.data(), oldid.p, nk * 4, cudaMemcpyDeviceToHost));
    R.old_id = F.old_id;
    G_CK(cudaDeviceSynchronize());
    return CC_OK;
}

}  // namespace ccg
