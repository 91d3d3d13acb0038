// Distances kept as bit planes (planes.cu).
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

#include "cc_internal.h"
#include "estimate.h"

namespace ccg {

// Largest distance of a plane job: the one-way limit, or two of them added.
constexpr int plane_rows(bool roundtrip) { return roundtrip ? 32 : 16; }

struct PlaneJob {
    int64_t n;
    int k, W;
    const uint64_t *F, *R;          // n x W x kPlanes words (R null unless round trip)
    const int32_t *sources, *sidx;  // k; n
    uint64_t *sum2;                 // n x 2
    int32_t *pivot;                 // n
    uint32_t *delta;                // n
    uint32_t *dcc;                  // k x k
    unsigned long long *dmax;       // 1
    uint32_t *hist;                 // rows x k (level-major), zeroed
    // hybrid: L(v) n C by pivot and threshold, and the rows of dcc as planes
    uint64_t *masks;                // k x plane_rows x W
    uint64_t *cplanes;              // k x W x 5
    const HybPrep *hp;
    uint64_t *lc2;                  // n x 2
    const uint8_t *sqflag;          // error estimate (null: not wanted; see ReduceJob)
    const int32_t *istar;
    uint64_t *hcse;
    uint32_t *fdist;
    // When set: nothing is done unless *ovf = 0 and npartial has a node, and
    // gate[0..1] of the second traversal pass is written (open only when the
    // planes overflowed).
    const int *ovf;
    const unsigned *npartial;
    unsigned *gate;
    // node weights (see NwJob)
    const uint32_t *beta, *bsrc;
    const uint64_t *mu, *tau;
    uint64_t *wsum, *lc;
    unsigned long long *S, *bhist;  // bhist: (D + 1) x k
    uint32_t eps_a, eps_b;
    int64_t D;
};

// The adaptive hybrid over n_eps values of eps = num / den.
struct AdaptiveJob {
    DevCount D;
    int64_t tstride;           // of the tail tables
    const uint32_t *maxd;      // k: largest distance between samples
    const uint64_t *TN, *TS, *S_samp;
    int n_eps;
    uint32_t num[64], den[64];
    double *est, *sq, *clo;    // n: of the eps of smallest squared error
    int32_t *choice;           // n: its index (-1: sampled node)
};

// Sums, pivots, Delta, the largest distance and delta_cc from the planes.
void run_planes_nodes(const PlaneJob &j, cudaStream_t st);
// Per-source distance histogram over V \ C, rows 0 .. D.
void run_planes_hist(const PlaneJob &j, cudaStream_t st);
// Sums over L(v) n C and the error estimate's inputs of the nodes that need
// them (after the thresholds).
void run_planes_lc(const PlaneJob &j, cudaStream_t st);
// The adaptive hybrid from the planes, the tail tables and istar: for every
// node the estimate, squared error and closeness of its best eps.
void run_planes_adaptive(const PlaneJob &j, const AdaptiveJob &a, cudaStream_t st);
// Node weights: per node sum_i mu_i d(c_i, v), per source sum_v beta(v) d.
void run_planes_nw1(const PlaneJob &j, cudaStream_t st);
// The hybrid's sums per node, and (bhist set) the beta mass per (distance,
// source).
void run_planes_nw2(const PlaneJob &j, cudaStream_t st);

}  // namespace ccg
