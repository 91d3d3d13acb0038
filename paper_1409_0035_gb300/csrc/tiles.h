// Shortest paths on graphs of narrow frontiers, tile by tile (tiles.cu).
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

#include "cc_internal.h"
#include "estimate.h"

namespace ccg {

// Nodes of a tile at most (a cluster centre stands for half as many).  Larger
// tiles take fewer rounds, smaller ones leave room for more CTAs with their
// arcs' lengths and correct fewer labels twice: 1024^2 grid, k = 256, 512 /
// 384 / 256: 17.5 / 19.4 / 24.5 ms an estimate; road-like lattice, 491 K
// nodes, k = 64: 18.8 / 13.1 / 15.4 ms.
constexpr int tile_cap(bool lengths) { return lengths ? 384 : 512; }
constexpr int kUnitWords = 8;      // words of 32 sources a CTA takes at once

// A graph cut into tiles of neighbouring nodes.  Slots are the nodes' numbers
// tile by tile, each tile padded to whole 32-slot words (perm = -1 there).
struct TileGraph {
    int64_t n = 0, slots = 0;
    int32_t tiles = 0;
    double levels = 0.0;                         // estimated hops across the graph
    int32_t *perm = nullptr, *iperm = nullptr;   // slot -> node, node -> slot
    int32_t *tb = nullptr;                       // tiles + 1: first slot of each
    int32_t *word_tile = nullptr;                // slots / 32: the word's tile
    uint32_t *irp = nullptr, *erp = nullptr;     // slots + 1: arcs inside, leaving the tile
    uint16_t *icol = nullptr;                    // head's slot within the tile
    int32_t *ecol = nullptr;                     // head's slot
    uint16_t *etail = nullptr;                   // tail's slot within the tile
    ushort4 *icol4 = nullptr;                    // inside rows of up to four arcs inline
    uint4 *iw4 = nullptr;                        // and their lengths
    uint32_t *iw = nullptr, *ew = nullptr;       // their lengths (null: unit lengths)
};

// How its tiles lie: for the host.  (The kernels take a TileGraph by value; with
// these three in it the road network's estimate took 0.5 % longer.)
struct TileShape {
    double depth = 0.0;       // tiles across the graph, from one of them
    double neighbours = 0.0;  // neighbouring tiles of a tile, mean
    double border = 0.0;      // arcs to each over the nodes of a tile's side
};

// Cuts an undirected CSR (rows of at most kLightMaxDeg entries; w null: unit
// lengths) into tiles.  *ok = false, and nothing kept, when the tiles would
// not be local: see tiles.cu.
int tiles_build(int64_t n, int64_t arcs, const int64_t *rp, const int32_t *col,
                const uint32_t *w, TileGraph &out, TileShape &shape, bool *ok, cudaStream_t st);
void tiles_free(TileGraph &g);

struct TileJob {
    TileGraph g;
    int k;                      // sources
    int kw;                     // words of 32 sources
    int uw, ku;                 // words per unit of work (at most kUnitWords), units per tile
    uint32_t delta;             // arc lengths: labels a round carries on beyond the last one's
    const int32_t *sources;     // k node ids
    uint32_t *dist;             // k x slots, source-major
    uint32_t *dirty[2];         // k x slots/32: slots lowered from outside, by round parity
    uint32_t *act[2];           // tiles x kw: sources with dirty slots in the tile
    uint32_t *stamp;            // tiles x ku: last round a unit was queued for
    int32_t *Q[2];              // tiles x ku: units (tile, words) to process
    Ctl *ctl;                   // band_ovf: some candidate label reached 2^32 - 1
    uint64_t timeout_ns;
};

// Whether a search of k sources by tiles is the faster one; passes: traversals
// of all sources that a level-synchronous estimate would make in its place.
bool tiles_pay(const TileGraph &g, const TileShape &s, int64_t k, int passes);

// Words per unit for k sources: as many as leave a fully active round 1,216
// units, two for every CTA on unit lengths (4 a SM) and about one with arc
// lengths (6 or 7 a SM).
int tile_unit_words(const TileGraph &g, int k);
int launch_tiles(const TileJob &job, cudaStream_t st);

// Reductions of the distances (source-major, dist[i * slots + slot]).
struct TileReduce {
    TileGraph g;
    int k, W;
    const uint32_t *dist;
    const int32_t *sources, *sidx;
    uint64_t *sum2;                 // n x 2
    int32_t *pivot;
    uint32_t *delta;
    uint32_t *dcc;                  // k x k
    unsigned long long *S_samp;     // k
    unsigned long long *dmax;       // 1
    int *err;                       // 1
    // hybrid: distance histogram (source-major, hs = row stride >= D + 1 and a
    // multiple of 64), suffix sums over its blocks of 64 distances
    int64_t D, hs;
    uint32_t *hist;
    uint64_t *TN, *TS;              // k x (hs / 64 + 1)
    HybPrep *hp;
    const uint64_t *Lmask;          // n x W
    uint64_t *lc2;                  // n x 2
    // error estimate (null sqflag: not wanted; see ReduceJob)
    const uint8_t *sqflag;
    const int32_t *istar;
    uint64_t *hcse;
    uint32_t *fdist;
};

// Sums, pivots, Delta, delta_cc, exact S of the sampled nodes, the largest
// distance and the reachability check.
void run_tiles_reduce1(const TileReduce &r, cudaStream_t st);
// After the thresholds and L(v) masks: histogram, tails, H statistics of
// every node and the sums over L(v) n C.
void run_tiles_reduce2(const TileReduce &r, cudaStream_t st);

}  // namespace ccg
