// Distances of graphs of small diameter as bit planes.
//
// A bit-packed traversal finds the distance of every (node, source) pair; the
// estimates that need the distances themselves (round trips, node weights,
// the error estimate, the adaptive hybrid) used to write them out as rows of
// 32-bit integers or to traverse again per threshold.  While distances stay
// below 16 the traversal instead ORs the bits of a level into the planes of
// the level's binary digits: four words per 64 pairs, half a byte a pair in
// place of four.  Sums over sources are then population counts of planes
// under masks (sum of d = sum over planes of 2^b |P_b|, sum of d^2 over pairs
// of planes, products of two distances likewise), the nearest sampled node
// is found plane by plane, a round trip is a bit-sliced addition of two sets
// of planes, and L(v) n C is a mask looked up by pivot and threshold.  All
// sums are exact integers, the same as over the rows.
#include <algorithm>
#include <cstdint>

#include "estimate_dev.cuh"
#include "planes.h"

namespace ccg {

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int kT = 256;
constexpr int kB = kPlanes + 1;  // planes of a sum of two distances
template <bool RT>
constexpr int plane_rows_dev = plane_rows(RT);

int grid_of(int64_t threads)
{
    return (int)std::min<int64_t>(std::max<int64_t>(1, (threads + kT - 1) / kT), 152 * 16);
}

__device__ __forceinline__ uint64_t valid_mask(int k, int w)
{
    const int lo = w * 64;
    if (k <= lo) return 0ull;
    if (k >= lo + 64) return ~0ull;
    return (1ull << (k - lo)) - 1ull;
}

__device__ __forceinline__ void load4(const uint64_t *p, uint64_t (&x)[kPlanes])
{
    const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(p);
    const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(p + 2);
    x[0] = a.x; x[1] = a.y; x[2] = b.x; x[3] = b.y;
}

// Planes of the distances at word vw = v W + w (round trip: of both sums).
template <bool RT>
__device__ __forceinline__ void load_planes(const PlaneJob &J, int64_t vw, uint64_t (&S)[kB])
{
    uint64_t f[kPlanes];
    load4(J.F + vw * kPlanes, f);
    if (!RT) {
#pragma unroll
        for (int b = 0; b < kPlanes; ++b) S[b] = f[b];
        S[kPlanes] = 0ull;
        return;
    }
    uint64_t r[kPlanes], c = 0ull;
    load4(J.R + vw * kPlanes, r);
#pragma unroll
    for (int b = 0; b < kPlanes; ++b) {
        const uint64_t x = f[b] ^ r[b];
        S[b] = x ^ c;
        c = (f[b] & r[b]) | (x & c);
    }
    S[kPlanes] = c;
}

// Sum of d and of d^2 over the pairs of mask m.
template <bool RT>
__device__ __forceinline__ void sums(const uint64_t (&S)[kB], uint64_t m, unsigned &s,
                                     unsigned &sq)
{
    constexpr int N = RT ? kB : kPlanes;
    s = sq = 0;
#pragma unroll
    for (int a = 0; a < N; ++a) {
        const uint64_t x = S[a] & m;
        const unsigned p = __popcll(x);
        s += p << a;
        sq += p << (2 * a);
#pragma unroll
        for (int b = a + 1; b < N; ++b) sq += (unsigned)__popcll(x & S[b]) << (a + b + 1);
    }
}

// Sum over a node's W lanes.
__device__ __forceinline__ unsigned group_sum(unsigned x, int W)
{
    for (int o = 1; o < W; o <<= 1) x += __shfl_xor_sync(FULL, x, o);
    return x;
}

// The nodes of a grid-strided sweep, W lanes each, whole warps together:
// body(v, w, ok).
template <class Body>
__device__ __forceinline__ void for_nodes(int64_t n, int W, Body body)
{
    const int lane = threadIdx.x & 31, w = lane & (W - 1), npw = 32 / W;
    const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v0 = gw * npw; v0 < n; v0 += nw * npw) {
        const int64_t v = v0 + lane / W;
        body(v, w, v < n);
    }
}

template <bool RT>
__global__ void k_pl_nodes(PlaneJob J)
{
    const int W = J.W, lane = threadIdx.x & 31, g0 = lane & ~(W - 1);
    const unsigned gm = W == 32 ? FULL : ((1u << W) - 1u) << g0;
    unsigned top = 0;
    for_nodes(J.n, W, [&](int64_t v, int w, bool ok) {
        uint64_t S[kB] = {0, 0, 0, 0, 0};
        if (ok) load_planes<RT>(J, v * W + w, S);
        uint64_t m = ok ? valid_mask(J.k, w) : 0ull;
        unsigned s, sq;
        sums<RT>(S, m, s, sq);
        // largest distance of the word, plane by plane from the top
        uint64_t x = m;
        unsigned mx = 0;
#pragma unroll
        for (int b = kB - 1; b >= 0; --b) {
            const uint64_t y = x & S[b];
            if (y) {
                x = y;
                mx |= 1u << b;
            }
        }
        top = max(top, mx);
        // the nearest source over the node's words: a plane with a clear bit
        // among the candidates keeps only those
        unsigned d = 0;
#pragma unroll
        for (int b = kB - 1; b >= 0; --b) {
            const uint64_t z = m & ~S[b];
            if (__ballot_sync(FULL, z != 0ull) & gm) m = z;
            else d |= 1u << b;
        }
        const unsigned has = __ballot_sync(FULL, m != 0ull) & gm;
        const int first = __ffs(has ? has : gm) - 1;
        const int p = __shfl_sync(FULL, w * 64 + __ffsll((long long)m) - 1, first);
        s = group_sum(s, W);
        sq = group_sum(sq, W);
        if (ok && w == 0) {
            J.sum2[2 * v] = s;
            J.sum2[2 * v + 1] = sq;
            J.pivot[v] = p;
            J.delta[v] = d;
        }
    });
    top = __reduce_max_sync(FULL, top);
    __shared__ unsigned s_top;
    if (threadIdx.x == 0) s_top = 0;
    __syncthreads();
    if (lane == 0) atomicMax(&s_top, top);
    __syncthreads();
    if (threadIdx.x == 0) atomicMax(J.dmax, (unsigned long long)s_top);
}

template <bool RT>
__device__ __forceinline__ unsigned pair_distance(const PlaneJob &J, int64_t v, int i)
{
    uint64_t S[kB];
    load_planes<RT>(J, v * J.W + (i >> 6), S);
    unsigned d = 0;
#pragma unroll
    for (int b = 0; b < kB; ++b) d |= (unsigned)((S[b] >> (i & 63)) & 1ull) << b;
    return d;
}

template <bool RT>
__global__ void k_pl_dcc(PlaneJob J)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < (int64_t)J.k * J.k;
         q += (int64_t)gridDim.x * blockDim.x)
        J.dcc[q] = pair_distance<RT>(J, J.sources[q % J.k], (int)(q / J.k));
}

// 32 x 32 bit transpose across a warp (lane c ends with bit c of every lane).
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane)
{
#pragma unroll
    for (int j = 16; j >= 1; j >>= 1) {
        const uint32_t m = j == 16 ? 0x0000FFFFu : j == 8 ? 0x00FF00FFu : j == 4 ? 0x0F0F0F0Fu
                         : j == 2 ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(FULL, x, j);
        x = (lane & j) ? ((x & ~m) | ((y & ~m) >> j)) : ((x & m) | ((y & m) << j));
    }
    return x;
}

// A lane per node, blockIdx.y the word: per distance the mask of the sources
// at it, transposed so that a lane counts the nodes of its two sources.
template <bool RT>
__global__ void k_pl_hist(PlaneJob J)
{
    __shared__ unsigned s_h[32][64];
    const int w = blockIdx.y, lane = threadIdx.x & 31, D = (int)J.D;
    for (int i = threadIdx.x; i < 32 * 64; i += blockDim.x) (&s_h[0][0])[i] = 0u;
    __syncthreads();
    const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const uint64_t vm = valid_mask(J.k, w);
    for (int64_t v0 = gw * 32; v0 < J.n; v0 += nw * 32) {
        const int64_t v = v0 + lane;
        const bool ok = v < J.n && J.sidx[v] < 0;
        uint64_t S[kB] = {0, 0, 0, 0, 0};
        if (ok) load_planes<RT>(J, v * J.W + w, S);
        const uint64_t m = ok ? vm : 0ull;
        for (int d = 1; d <= D; ++d) {
            uint64_t x = m;
#pragma unroll
            for (int b = 0; b < kB; ++b) x &= (d >> b) & 1 ? S[b] : ~S[b];
            if (!__any_sync(FULL, x != 0ull)) continue;
            const unsigned lo = __popc(transpose32((uint32_t)x, lane));
            const unsigned hi = __popc(transpose32((uint32_t)(x >> 32), lane));
            if (lo) atomicAdd(&s_h[d][lane], lo);
            if (hi) atomicAdd(&s_h[d][32 + lane], hi);
        }
    }
    __syncthreads();
    for (int c = threadIdx.x; c < 64 * (D + 1); c += blockDim.x) {
        const int d = c >> 6, i = 64 * w + (c & 63);
        if (i < J.k && s_h[d][c & 63]) atomicAdd(&J.hist[(int64_t)d * J.k + i], s_h[d][c & 63]);
    }
}

__device__ __forceinline__ bool skip_lc(const PlaneJob &J)
{
    return J.ovf && (*J.ovf != 0 || (J.npartial[0] == 0u && J.npartial[1] == 0u));
}

// masks[(p rows + t) W + w] = sources of word w within t of c_p; cplanes: the
// planes of row p of delta_cc.  A thread per (p, w).
template <bool RT>
__global__ void k_pl_masks(PlaneJob J)
{
    constexpr int kRows = plane_rows_dev<RT>;
    if (J.gate && blockIdx.x == 0 && threadIdx.x == 0) {
        J.gate[0] = *J.ovf ? J.npartial[0] + J.npartial[1] : 0u;
        J.gate[1] = 0u;
    }
    if (skip_lc(J)) return;
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < J.k * J.W;
         q += gridDim.x * blockDim.x) {
        const int p = q / J.W, w = q % J.W;
        uint64_t C[kB] = {0, 0, 0, 0, 0};
        const int hi = min(J.k, 64 * w + 64);
        for (int i = 64 * w; i < hi; ++i) {
            const unsigned d = J.dcc[(int64_t)p * J.k + i];
#pragma unroll
            for (int b = 0; b < kB; ++b) C[b] |= (uint64_t)((d >> b) & 1u) << (i & 63);
        }
        uint64_t m = 0ull;
        const uint64_t vm = valid_mask(J.k, w);
        for (int t = 0; t < kRows; ++t) {
            uint64_t x = vm;
#pragma unroll
            for (int b = 0; b < kB; ++b) x &= (t >> b) & 1 ? C[b] : ~C[b];
            m |= x;
            J.masks[((int64_t)p * kRows + t) * J.W + w] = m;
        }
#pragma unroll
        for (int b = 0; b < kB; ++b) J.cplanes[(int64_t)q * kB + b] = C[b];
    }
}

template <bool RT>
__global__ void k_pl_lc(PlaneJob J)
{
    constexpr int kRows = plane_rows_dev<RT>;
    if (skip_lc(J)) return;
    const int W = J.W;
    for_nodes(J.n, W, [&](int64_t v, int w, bool ok) {
        HybPrep h{0, 0, 0, 0};
        uint8_t f = 0;
        if (ok && J.sidx[v] < 0) {
            h = J.hp[v];
            f = J.sqflag ? J.sqflag[v] : 0;
        }
        const bool part = (h.LCnum & kPartialBit) != 0;
        if (!__any_sync(FULL, part || f != 0)) return;
        unsigned s = 0, sq = 0, e2 = 0;
        if (part || f) {
            uint64_t S[kB];
            load_planes<RT>(J, v * W + w, S);
            const int p = J.pivot[v];
            const int t = h.thr < (uint64_t)(kRows - 1) ? (int)h.thr : kRows - 1;
            const uint64_t L = J.masks[((int64_t)p * kRows + t) * W + w];
            if (part) sums<RT>(S, L, s, sq);
            if (f & 1) {
                // sum of (d - c)^2 over the sources beyond the threshold
                const uint64_t H = valid_mask(J.k, w) & ~L;
                uint64_t C[kB];
#pragma unroll
                for (int b = 0; b < kB; ++b) C[b] = J.cplanes[((int64_t)p * W + w) * kB + b];
                unsigned a0, dd, cc, x = 0;
                sums<RT>(S, H, a0, dd);
                sums<RT>(C, H, a0, cc);
#pragma unroll
                for (int a = 0; a < kB; ++a)
#pragma unroll
                    for (int b = 0; b < kB; ++b)
                        x += (unsigned)__popcll(S[a] & C[b] & H) << (a + b);
                e2 = dd + cc - 2u * x;
            }
            if (f & 2) {
                const int is = J.istar[p];
                if ((is >> 6) == w) {
                    unsigned d = 0;
#pragma unroll
                    for (int b = 0; b < kB; ++b) d |= (unsigned)((S[b] >> (is & 63)) & 1ull) << b;
                    J.fdist[v] = d;
                }
            }
        }
        s = group_sum(s, W);
        sq = group_sum(sq, W);
        e2 = group_sum(e2, W);
        if (w == 0 && part) {
            J.lc2[2 * v] = s;
            J.lc2[2 * v + 1] = sq;
        }
        if (w == 0 && (f & 1)) {
            J.hcse[2 * v] = e2;
            J.hcse[2 * v + 1] = 0;
        }
    });
}

// The adaptive hybrid, W lanes a node.  Thresholds at or beyond the largest
// distance give the same classes (most small eps do), and a later eps wins
// only by a smaller squared error, so an eps whose threshold equals the one
// before it is passed over; the others' sums are collected lane by lane until
// W are together, since the FP64 of one estimate takes a warp as long as that
// of 32.  One pass over the planes for all eps in place of five kernels and
// 150 bytes of state per node and eps (R-MAT 18, k = 256, seven eps: 594 of
// 920 us of kernels before, 150 now).
template <bool RT>
__global__ void k_pl_adaptive(PlaneJob J, AdaptiveJob A)
{
    constexpr int kRows = plane_rows_dev<RT>;
    const int W = J.W, lane = threadIdx.x & 31, g0 = lane & ~(W - 1);
    const int64_t D = count_of(A.D);
    const uint64_t nm1 = (uint64_t)(J.n - 1);
    for_nodes(J.n, W, [&](int64_t v, int w, bool ok) {
        const int j = ok ? J.sidx[v] : 0;
        const bool live = ok && j < 0;
        uint64_t S[kB] = {0, 0, 0, 0, 0};
        int p = 0;
        uint32_t delta = 0, maxd = 0;
        uint64_t sum = 0, sumsq = 0;
        if (live) {
            load_planes<RT>(J, v * W + w, S);
            p = J.pivot[v];
            delta = J.delta[v];
            maxd = A.maxd[p];
            sum = J.sum2[2 * v];
            sumsq = J.sum2[2 * v + 1];
        }
        double best = live || !ok ? 0.0 : (double)A.S_samp[j], bsq = 0.0;
        int choice = -1;
        int64_t before = -1;  // threshold of the eps last taken
        int held = 0;         // estimates collected, lane w the w-th
        // the one of this lane: LCnum, sums over L n C, the pivoting term's
        // sum (or the one distance), threshold, eps
        uint64_t c_lc = 0, c_s = 0, c_sq = 0, c_e2 = 0;
        int64_t c_tt = 0;
        int c_e = 0;
        for (int e = 0; e <= A.n_eps; ++e) {
            const bool end = e == A.n_eps;
            if (!end) {
                const uint64_t thr = (uint64_t)delta * A.den[e] / A.num[e];
                const int64_t tt = thr < (uint64_t)D ? (int64_t)thr : D;
                const bool take = live && tt != before;
                if (!__any_sync(FULL, take)) continue;
                const bool part = take && thr < maxd;
                unsigned lc = 0, s = 0, sq = 0, e2 = 0;
                if (part) {
                    const uint64_t L = J.masks[((int64_t)p * kRows + tt) * W + w];
                    lc = __popcll(L);
                    sums<RT>(S, L, s, sq);
                    const uint64_t H = valid_mask(J.k, w) & ~L;
                    uint64_t C[kB];
#pragma unroll
                    for (int b = 0; b < kB; ++b) C[b] = J.cplanes[((int64_t)p * W + w) * kB + b];
                    unsigned a0, dd, cc, x = 0;
                    sums<RT>(S, H, a0, dd);
                    sums<RT>(C, H, a0, cc);
#pragma unroll
                    for (int a = 0; a < kB; ++a)
#pragma unroll
                        for (int b = 0; b < kB; ++b)
                            x += (unsigned)__popcll(S[a] & C[b] & H) << (a + b);
                    e2 = dd + cc - 2u * x;
                } else if (take) {
                    const int is = J.istar[p];
                    if ((is >> 6) == w) {
#pragma unroll
                        for (int b = 0; b < kB; ++b)
                            e2 |= (unsigned)((S[b] >> (is & 63)) & 1ull) << b;
                    }
                }
                lc = group_sum(lc, W);
                s = group_sum(s, W);
                sq = group_sum(sq, W);
                e2 = group_sum(e2, W);
                if (take) {
                    if (w == held) {
                        c_lc = part ? lc : (uint64_t)J.k;
                        c_s = part ? s : sum;
                        c_sq = part ? sq : sumsq;
                        c_e2 = e2;
                        c_tt = tt;
                        c_e = e;
                    }
                    ++held;
                    before = tt;
                }
            }
            if (!(end ? __any_sync(FULL, held > 0) : __any_sync(FULL, held == W))) continue;
            double est = 0.0, err = 0.0;
            if (w < held) {
                const uint64_t Hnum = A.TN[(int64_t)p * A.tstride + c_tt];
                const uint64_t Hsum = A.TS[(int64_t)p * A.tstride + c_tt];
                const uint64_t HCsum = sum - c_s, HCnum = (uint64_t)J.k - c_lc;
                const uint64_t Lnum = nm1 - Hnum - HCnum;
                const u128 N = (u128)(Hsum + HCsum) * c_lc + (u128)c_s * Lnum;
                est = u128_to_double(N) / (double)c_lc;
                if (c_lc == (uint64_t)J.k && Hnum == 0)
                    est = u128_to_double((u128)nm1 * sum) / (double)J.k;
                u128 t2num = 0;
                if (HCnum > 0) {
                    t2num = (u128)c_e2 * Hnum;
                } else if (Hnum > 0) {
                    const int64_t x = (int64_t)c_e2 -
                                      (int64_t)J.dcc[(int64_t)p * J.k + J.istar[p]];
                    const uint64_t ax = (uint64_t)(x < 0 ? -x : x);
                    t2num = (u128)ax * ax * Hnum;
                }
                err = sq_err_of(c_lc, c_s, c_sq, Lnum, HCnum, t2num);
            }
            for (int i = 0; i < W; ++i) {
                const double xe = __shfl_sync(FULL, est, g0 + i);
                const double xq = __shfl_sync(FULL, err, g0 + i);
                const int xi = __shfl_sync(FULL, c_e, g0 + i);
                if (i < held && (choice < 0 || xq < bsq)) {
                    best = xe;
                    bsq = xq;
                    choice = xi;
                }
            }
            held = 0;
        }
        if (ok && w == 0) {
            A.est[v] = best;
            A.sq[v] = bsq;
            A.clo[v] = (double)nm1 / best;
            A.choice[v] = choice;
        }
    });
}

// ---- node weights ---------------------------------------------------------

// S[i] += sum over v of beta(v) d(c_i, v): a warp per node, lane l the
// sources 64 w + l and 64 w + 32 + l of up to four words (blockIdx.y).
template <bool RT>
__global__ void k_pl_nw_sources(PlaneJob J)
{
    const int lane = threadIdx.x & 31, w0 = 4 * blockIdx.y, nwd = min(4, J.W - w0);
    const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long acc[4][2] = {};
    for (int64_t v = gw; v < J.n; v += nw) {
        const unsigned long long beta = J.beta[v];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (q >= nwd) break;
            uint64_t S[kB];
            load_planes<RT>(J, v * J.W + w0 + q, S);
            unsigned lo = 0, hi = 0;
#pragma unroll
            for (int b = 0; b < kB; ++b) {
                lo |= (((unsigned)S[b] >> lane) & 1u) << b;
                hi |= (((unsigned)(S[b] >> 32) >> lane) & 1u) << b;
            }
            acc[q][0] += beta * lo;
            acc[q][1] += beta * hi;
        }
    }
    __shared__ unsigned long long s_S[256];
    s_S[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (q >= nwd) break;
        atomicAdd(&s_S[64 * q + lane], acc[q][0]);
        atomicAdd(&s_S[64 * q + 32 + lane], acc[q][1]);
    }
    __syncthreads();
    const int i = 64 * w0 + threadIdx.x;
    if (threadIdx.x < 64 * nwd && i < J.k && s_S[threadIdx.x]) atomicAdd(&J.S[i], s_S[threadIdx.x]);
}

// Bit i of a word: distance of its source.
__device__ __forceinline__ unsigned bit_distance(const uint64_t (&S)[kB], int i)
{
    unsigned d = 0;
#pragma unroll
    for (int b = 0; b < kB; ++b) d |= (unsigned)((S[b] >> i) & 1ull) << b;
    return d;
}

// sum of mu_i d(c_i, v) over the sources of mask m: mu = tn (tau, times its
// denominator) for all but the few certain ones.
template <bool RT>
__device__ __forceinline__ unsigned long long mu_sum(const PlaneJob &J, const uint64_t (&S)[kB],
                                                     uint64_t m, uint64_t certain, int w,
                                                     unsigned long long tn)
{
    unsigned s, sq;
    sums<RT>(S, m & ~certain, s, sq);
    unsigned long long x = tn * s;
    for (uint64_t c = m & certain; c; c &= c - 1) {
        const int i = __ffsll((long long)c) - 1;
        x += J.mu[64 * w + i] * bit_distance(S, i);
    }
    return x;
}

// Sources of word w whose mu is not tn.
__device__ __forceinline__ uint64_t certain_mask(const PlaneJob &J, int w)
{
    const uint64_t tn = J.tau[0];
    uint64_t m = 0ull;
    const int hi = min(J.k, 64 * w + 64);
    for (int i = 64 * w; i < hi; ++i)
        if (J.mu[i] != tn) m |= 1ull << (i & 63);
    return m;
}

__device__ __forceinline__ unsigned long long group_sum64(unsigned long long x, int W)
{
    for (int o = 1; o < W; o <<= 1) x += __shfl_xor_sync(FULL, x, o);
    return x;
}

template <bool RT>
__global__ void k_pl_nw_nodes(PlaneJob J)
{
    const int W = J.W;
    const unsigned long long tn = J.tau[0];
    __shared__ uint64_t s_c[32];
    if (threadIdx.x < W) s_c[threadIdx.x] = certain_mask(J, threadIdx.x);
    __syncthreads();
    for_nodes(J.n, W, [&](int64_t v, int w, bool ok) {
        unsigned long long x = 0;
        if (ok) {
            uint64_t S[kB];
            load_planes<RT>(J, v * W + w, S);
            x = mu_sum<RT>(J, S, valid_mask(J.k, w), s_c[w], w, tn);
        }
        x = group_sum64(x, W);
        if (ok && w == 0) J.wsum[v] = x;
    });
}

template <bool RT>
__global__ void k_pl_nw_lc(PlaneJob J)
{
    constexpr int kRows = plane_rows_dev<RT>;
    const int W = J.W;
    const unsigned long long tn = J.tau[0];
    __shared__ uint64_t s_c[32];
    if (threadIdx.x < W) s_c[threadIdx.x] = certain_mask(J, threadIdx.x);
    __syncthreads();
    for_nodes(J.n, W, [&](int64_t v, int w, bool ok) {
        unsigned long long lp = 0, hc = 0;
        const bool on = ok && J.sidx[v] < 0;
        if (on) {
            uint64_t S[kB];
            load_planes<RT>(J, v * W + w, S);
            const uint64_t thr = (uint64_t)J.delta[v] * J.eps_b / J.eps_a;
            const int t = thr < (uint64_t)(kRows - 1) ? (int)thr : kRows - 1;
            const uint64_t L = J.masks[((int64_t)J.pivot[v] * kRows + t) * W + w];
            lp = mu_sum<RT>(J, S, L, s_c[w], w, tn);
            for (uint64_t c = valid_mask(J.k, w) & ~L; c; c &= c - 1) {
                const int i = __ffsll((long long)c) - 1;
                hc += (unsigned long long)J.bsrc[64 * w + i] * bit_distance(S, i);
            }
        }
        lp = group_sum64(lp, W);
        hc = group_sum64(hc, W);
        if (on && w == 0) {
            J.lc[2 * v] = lp;
            J.lc[2 * v + 1] = hc;
        }
    });
}

// Beta mass of V \ C per (distance, source): a warp per node, blockIdx.y the
// word, lanes its sources.
template <bool RT>
__global__ void k_pl_nw_hist(PlaneJob J)
{
    __shared__ unsigned long long s_h[32][64];
    const int w = blockIdx.y, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < 32 * 64; i += blockDim.x) (&s_h[0][0])[i] = 0;
    __syncthreads();
    const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const bool v0 = 64 * w + lane < J.k, v1 = 64 * w + 32 + lane < J.k;
    for (int64_t v = gw; v < J.n; v += nw) {
        const unsigned long long beta = J.beta[v];
        if (J.sidx[v] >= 0 || beta == 0) continue;
        uint64_t S[kB];
        load_planes<RT>(J, v * J.W + w, S);
        if (v0) atomicAdd(&s_h[bit_distance(S, lane)][lane], beta);
        if (v1) atomicAdd(&s_h[bit_distance(S, 32 + lane)][32 + lane], beta);
    }
    __syncthreads();
    for (int c = threadIdx.x; c < 64 * ((int)J.D + 1); c += blockDim.x) {
        const int d = c >> 6, i = 64 * w + (c & 63);
        if (i < J.k && s_h[d][c & 63])
            atomicAdd(&J.bhist[(int64_t)d * J.k + i], s_h[d][c & 63]);
    }
}

}  // namespace

#define PLANES(kernel, grid, j, st)                                   \
    do {                                                              \
        if ((j).R) kernel<true><<<grid, kT, 0, st>>>(j);              \
        else kernel<false><<<grid, kT, 0, st>>>(j);                   \
    } while (0)

void run_planes_nodes(const PlaneJob &j, cudaStream_t st)
{
    PLANES(k_pl_nodes, grid_of(j.n * j.W), j, st);
    PLANES(k_pl_dcc, grid_of((int64_t)j.k * j.k), j, st);
}

void run_planes_hist(const PlaneJob &j, cudaStream_t st)
{
    const dim3 grid((unsigned)std::min<int64_t>((j.n + kT - 1) / kT, 152 * 4), (unsigned)j.W);
    PLANES(k_pl_hist, grid, j, st);
}

void run_planes_lc(const PlaneJob &j, cudaStream_t st)
{
    PLANES(k_pl_masks, grid_of((int64_t)j.k * j.W), j, st);
    PLANES(k_pl_lc, grid_of(j.n * j.W), j, st);
}

void run_planes_adaptive(const PlaneJob &j, const AdaptiveJob &a, cudaStream_t st)
{
    PLANES(k_pl_masks, grid_of((int64_t)j.k * j.W), j, st);
    const int grid = grid_of(j.n * j.W);
    if (j.R) k_pl_adaptive<true><<<grid, kT, 0, st>>>(j, a);
    else k_pl_adaptive<false><<<grid, kT, 0, st>>>(j, a);
}

void run_planes_nw1(const PlaneJob &j, cudaStream_t st)
{
    PLANES(k_pl_nw_nodes, grid_of(j.n * j.W), j, st);
    const dim3 grid((unsigned)std::min<int64_t>((j.n * 32 + kT - 1) / kT, 152 * 4),
                    (unsigned)((j.W + 3) / 4));
    PLANES(k_pl_nw_sources, grid, j, st);
}

void run_planes_nw2(const PlaneJob &j, cudaStream_t st)
{
    PLANES(k_pl_masks, grid_of((int64_t)j.k * j.W), j, st);
    PLANES(k_pl_nw_lc, grid_of(j.n * j.W), j, st);
    if (!j.bhist) return;
    const dim3 grid((unsigned)std::min<int64_t>((j.n * 32 + kT - 1) / kT, 152 * 4),
                    (unsigned)j.W);
    PLANES(k_pl_nw_hist, grid, j, st);
}

}  // namespace ccg
