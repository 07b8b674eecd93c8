// Spatial index of the nearest-neighbour search (knn_index.cu), shared with
// the entry points in knn.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace mr {

// Written by the first kernel of a call.
struct NnControl {
    int unfit;   // the clouds' ranges are not ascending and disjoint
};

// One batch of clouds in sorted form.  Cloud i keeps its own row range of the
// packed arrays, its leaves start at (first >> 5) + i and its nodes at
// (first >> 10) + i: first is non-decreasing and the ranges are disjoint, so
// these never collide and no prefix over the clouds is needed.  Clouds in other
// ranges -- in any order, or one candidate cloud shared by many query clouds --
// are not sorted; the search then scans every candidate where it lies.
struct NnSide {
    const float *x;
    const int64_t *first, *len;
    int64_t P;
    NnControl *control;         // one for both batches
    long long *plan;            // N + 1: the scan's tiles of this batch as queries (NULL: never queries)
    int per;                    // queries of such a tile
    int N, bits, cells, tiles;  // cells = 2^(bits D) per cloud, tiles of kNnTile cells
    unsigned *box;              // N x 8: running bounds, order-preserving bits
    float *span;                // N x 8: what k_nn_bounds sampled
    float4 *grid;               // N x 2: low corner; cells per unit
    int *start;                 // N x cells: counts, then the first sorted position of each cell
    int *tile_sum;              // N x tiles
    int2 *cell_rank;            // P: cell of the point, its rank there
    float4 *pts;                // P: sorted coordinates (D <= 3: the local row's bits in w)
    int *row;                   // P (D = 4): local row
    float4 *leaf, *node;        // low and high corner of every 32 (1,024) sorted points
};

struct NnQuery {
    NnSide q, c;                // query side, candidate side
    int64_t *idx;
    float *dists;
    int K;
};

// Whether searching through the index beats scanning every candidate.
bool nn_index_wins(int64_t N, int64_t P1, int64_t P2, int D, int K);
// Whether its search gives every query a warp instead of a lane.
bool nn_search_per_warp(int64_t P1, int64_t P2, int K);
size_t nn_index_bytes(int64_t N, int64_t P1, int64_t P2, int D);
// Sides laid out in `ws` (nn_index_bytes), built on `st`: sides[0] the first batch, sides[1] the second.  The
// first is searched for K neighbours; with `both_ways` the second is, too.  `plans`: 2 (N + 1) words.
cudaError_t nn_index_build(NnSide (&sides)[2], const float *p1, int64_t P1, const int64_t *first1,
                           const int64_t *len1, const float *p2, int64_t P2, const int64_t *first2,
                           const int64_t *len2, int64_t N, int D, int K, bool both_ways, long long *plans, char *ws,
                           cudaStream_t st);
cudaError_t nn_index_search(const NnSide &q, const NnSide &c, int D, int K, int64_t *idx, float *dists,
                            cudaStream_t st);

}  // namespace mr
