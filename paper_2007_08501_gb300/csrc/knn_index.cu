// Spatial index for exact K nearest neighbours on packed batches of point
// clouds (Section 3.1 of the paper, "K Nearest Neighbors"), sm_103a.
//
// Scanning every candidate costs |P| |Q| distances.  Here both batches are
// sorted along a Hilbert curve (one counting sort over a grid per cloud), every
// 32 consecutive points form a leaf and every 32 leaves a node, each with its
// box, and a search skips the leaves and nodes whose box is farther than the
// K-th neighbour found so far.
//
// Skipping is exact in fp32, not merely up to rounding: the distance to a box
// is evaluated with the very steps of the ranking distance (subtract, square,
// fma in the same order), every step is monotone under round-to-nearest, and
// a box coordinate lies at or before the point's, so box distance <= point
// distance bit for bit.  A box is skipped only when it is strictly farther
// than the K-th entry, since an equal distance may still win by its row.  The
// lists rank by (distance, row), so the visiting order does not matter and
// the results are those of the scan.
//
// The clouds' ranges decide where everything lies, and only the device knows
// them: the first kernel checks that they are ascending and disjoint.  If they
// are not, the building kernels leave everything alone and the search kernels
// scan all candidates in place (a launch of knn.cu's scan behind every search,
// to do nothing, cost 32 pairs of 1,000 and 50,000 points 14 of 384 us).  8
// clouds of 30,000 points against one of 30,000: K = 1 2,299 us, K = 8 2,799; the
// scan of knn.cu 1,810 and 3,729.
//
//   k_nn_bounds   bounds of every cloud; one more block per batch checks its
//                 ranges and plans the tiles of such a scan, one per cloud
//                 bounds its grid by a sample
//   k_nn_count    cell of every point and its rank there (warp-aggregated)
//   k_nn_tiles    sums of kNnTile cells (clouds of more cells than that)
//   k_nn_starts   exclusive scan of a cloud's cells
//   k_nn_scatter  points to their sorted places
//   k_nn_boxes    one block per node: boxes of its 32 leaves and its own
//   k_nn_lanes    search, a query per lane: 32 neighbouring queries share the
//                 walk, each skips the leaves it does not need
//   k_nn_warps    search, a query per warp (few queries: a query's 32 lanes
//                 take a leaf's 32 candidates)
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>

#include "knn_index.h"
#include "knn_plan.cuh"
#include "rast_common.cuh"

namespace mr {
namespace {

constexpr int kNnTile = 4096;   // cells scanned by one block
constexpr int kLeaf = 32, kNode = 1024;
constexpr unsigned kAll = 0xffffffffu;

// float order as unsigned order
__device__ __forceinline__ unsigned enc(float x) {
    const unsigned u = __float_as_uint(x);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float dec(unsigned e) {
    return __uint_as_float((e & 0x80000000u) ? (e & 0x7fffffffu) : ~e);
}

// Cloud and tile of block b when cloud i's tiles of 2^shift rows start at
// (first[i] >> shift) + i.  False when the block has no rows, or the ranges are
// unfit (the word is asked for first and looked at last: waiting for it on
// entry cost each kernel 0.7 us).
__device__ __forceinline__ bool tile_of(const NnSide &s, long long b, int shift, int &cloud, long long &row0, int &n) {
    const int unfit = s.control->unfit;
    int lo = 0, hi = s.N;   // last i with start <= b
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if ((s.first[mid] >> shift) + mid <= b) lo = mid; else hi = mid;
    }
    const long long t = b - ((s.first[lo] >> shift) + lo);
    cloud = lo;
    row0 = t << shift;
    n = (int)s.len[lo];
    return t >= 0 && row0 < n && !unfit;
}

// The same for a search kernel: with unfit ranges the tile of the scan's plan.
__device__ __forceinline__ bool query_tile(const NnSide &s, long long b, int shift, int &cloud, long long &row0, int &n,
                                           bool &scan) {
    scan = false;
    if (tile_of(s, b, shift, cloud, row0, n)) return true;
    if (!s.control->unfit || b >= s.plan[s.N]) return false;
    scan = true;
    cloud = planned_cloud(s.plan, s.N, b);
    row0 = (b - s.plan[cloud]) << shift;
    n = (int)s.len[cloud];
    return true;
}

template <int D>
__device__ __forceinline__ void load_point(const float *x, long long row, float (&v)[D]) {
#pragma unroll
    for (int c = 0; c < D; ++c) v[c] = __ldg(x + row * D + c);
}

// ---------------------------------------------------------------------------
// building
// ---------------------------------------------------------------------------
// Ends of a cloud's grid, from 32 of its points: per axis, all but the outermost
// two, and as much again on either side.  That takes in the whole of most clouds;
// what lies farther out goes to the border cells.  A grid over everything lets one
// far point put all others into one cell, in no order, and their boxes part
// nothing: 8 clouds of 30,000 + 30,000 points with one outlier each, K = 1: 3,680 ->
// 215 us (K = 8: 3,202 -> 422; the scan takes 1,857 and 3,738).  One warp's work.
template <int D>
__device__ __forceinline__ void sample_span(const NnSide &s, int cloud) {
    const int t = threadIdx.x;
    const long long n = s.len[cloud];
    if (t >= 32 || n <= 0) return;   // (an empty cloud has no cells to fill)
    float v[D];
    load_point<D>(s.x, s.first[cloud] + t * n / 32, v);
    float *o = s.span + 8 * (size_t)cloud;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        int rank = 0;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            const float u = __shfl_sync(kAll, v[c], j);
            rank += u < v[c] || (u == v[c] && j < t);
        }
        if (rank == 1) o[c] = v[c];
        if (rank == 30) o[4 + c] = v[c];
    }
}

// box[cloud]: enc(high) in 0..3, enc(-low) in 4..7, both by atomicMax from 0.
// A block takes 4,096 rows, so that few atomics meet at a cloud's words.  (It
// runs beside the check of the ranges; unfit ones have it read rows of their own
// clouds and write their clouds' words, nothing else.)
template <int D>
__global__ void __launch_bounds__(256) k_nn_bounds(NnSide a, NnSide b) {
    const NnSide &s = blockIdx.y ? b : a;
    if ((int)blockIdx.x < s.N) {
        sample_span<D>(s, (int)blockIdx.x);
        return;
    }
    if ((int)blockIdx.x == s.N) {
        for (int i = threadIdx.x; i < s.N; i += 256) {
            const long long f = s.first[i], n = s.len[i], next = i + 1 < s.N ? s.first[i + 1] : s.P;
            if (f < 0 || n < 0 || n > s.P || f > next - n) s.control->unfit = 1;
        }
        if (s.plan) plan_tiles<256>(s.len, s.N, s.per, s.plan);
        return;
    }
    __shared__ unsigned s_m[2 * D];
    int cloud, n;
    long long row0;
    if (!tile_of(s, (long long)blockIdx.x - s.N - 1, 12, cloud, row0, n)) return;   // uniform for the block
    if (threadIdx.x < 2 * D) s_m[threadIdx.x] = 0u;
    __syncthreads();
    float hi[D], lo[D];
#pragma unroll
    for (int c = 0; c < D; ++c) { hi[c] = -INFINITY; lo[c] = INFINITY; }
#pragma unroll 4
    for (int k = 0; k < 16; ++k) {
        const long long r = row0 + k * 256 + threadIdx.x;
        if (r >= n) continue;
        float v[D];
        load_point<D>(s.x, s.first[cloud] + r, v);
#pragma unroll
        for (int c = 0; c < D; ++c)
            if (isfinite(v[c])) { hi[c] = fmaxf(hi[c], v[c]); lo[c] = fminf(lo[c], v[c]); }
    }
#pragma unroll
    for (int c = 0; c < D; ++c) {
        const unsigned h = __reduce_max_sync(kAll, enc(hi[c])), l = __reduce_max_sync(kAll, enc(-lo[c]));
        if ((threadIdx.x & 31) == 0) {
            atomicMax(s_m + c, h);
            atomicMax(s_m + D + c, l);
        }
    }
    __syncthreads();
    if (threadIdx.x < 2 * D) {
        const int c = threadIdx.x % D;
        atomicMax(s.box + 8 * (size_t)cloud + (threadIdx.x < D ? c : 4 + c), s_m[threadIdx.x]);
    }
}

// Position of grid cell g (2^bits cells per axis) along the D-dimensional
// Hilbert curve, after Skilling ("Programming the Hilbert curve", 2004): from
// the top bit down, an axis whose bit is set flips the lower bits of axis 0,
// one whose bit is clear trades them with axis 0; the bits are then a Gray
// code read across the axes.  Consecutive cells are neighbours, so 32 points
// in a row are compact; along a Morton curve some groups span a jump across
// the cloud, and one such warp of queries walks most of it.
template <int D>
__device__ __forceinline__ unsigned curve_of(unsigned (&g)[D], int bits) {
    for (int i = bits - 1; i > 0; --i) {
        const unsigned low = (1u << i) - 1u;
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const bool set = (g[c] >> i) & 1u;
            const unsigned t = set ? low : (g[0] ^ g[c]) & low;
            g[0] ^= t;
            if (!set && c > 0) g[c] ^= t;
        }
    }
    unsigned code = 0, parity = 0;   // Gray decoding: running parity of the bits in curve order
    for (int i = bits - 1; i >= 0; --i) {
#pragma unroll
        for (int c = 0; c < D; ++c) {
            parity ^= (g[c] >> i) & 1u;
            code = (code << 1) | parity;
        }
    }
    return code;
}

// A cloud's grid: cubic cells, 2^bits along the longest side of its bounds within
// the span.
template <int D>
struct Grid {
    float lo[D], scale;
};

template <int D>
__device__ __forceinline__ Grid<D> grid_of(const NnSide &s, int cloud) {
    const unsigned *bx = s.box + 8 * (size_t)cloud;
    const float *span = s.span + 8 * (size_t)cloud;
    Grid<D> g;
    float ext = 0.f;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        const float a = __ldg(span + c), b = __ldg(span + 4 + c), w = b > a ? b - a : INFINITY;
        g.lo[c] = fmaxf(-dec(__ldg(bx + 4 + c)), a - w);
        ext = fmaxf(ext, fminf(dec(__ldg(bx + c)), b + w) - g.lo[c]);
    }
    g.scale = (ext > 0.f && ext < 1e37f) ? (float)(1 << s.bits) / ext : 0.f;
    return g;
}

// the same once k_nn_count has left it behind
template <int D>
__device__ __forceinline__ Grid<D> kept_grid(const NnSide &s, int cloud) {
    const float4 a = __ldg(s.grid + 2 * (size_t)cloud);
    const float v[4] = {a.x, a.y, a.z, a.w};
    Grid<D> g;
#pragma unroll
    for (int c = 0; c < D; ++c) g.lo[c] = v[c];
    g.scale = __ldg(&s.grid[2 * (size_t)cloud + 1].x);
    return g;
}

// Cell of v, numbered along the curve.  Any point maps to some cell (outside
// ones to the border).
template <int D>
__device__ __forceinline__ int cell_of(const NnSide &s, const Grid<D> &grid, const float (&v)[D]) {
    const float top = (float)((1 << s.bits) - 1);
    unsigned g[D];
#pragma unroll
    for (int c = 0; c < D; ++c) g[c] = (unsigned)fminf(fmaxf((v[c] - grid.lo[c]) * grid.scale, 0.f), top);
    return (int)curve_of<D>(g, s.bits);
}

template <int D>
__global__ void __launch_bounds__(256) k_nn_count(NnSide a, NnSide b) {
    const NnSide &s = blockIdx.y ? b : a;
    int cloud, n;
    long long row0;
    if (!tile_of(s, blockIdx.x, 8, cloud, row0, n)) return;
    const long long r = row0 + threadIdx.x;
    const Grid<D> grid = grid_of<D>(s, cloud);
    int cell = -1;
    if (r < n) {
        float v[D];
        load_point<D>(s.x, s.first[cloud] + r, v);
        cell = cell_of<D>(s, grid, v);
    }
    if (r == 0) {   // (a cloud without points has no search)
        float lo[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < D; ++c) lo[c] = grid.lo[c];
        s.grid[2 * (size_t)cloud] = make_float4(lo[0], lo[1], lo[2], lo[3]);
        s.grid[2 * (size_t)cloud + 1].x = grid.scale;
    }
    // lanes of one cell (clustered points, duplicates) share an atomic
    const unsigned peers = __match_any_sync(kAll, cell);
    const int lane = threadIdx.x & 31, lead = __ffs(peers) - 1;
    int base = 0;
    if (cell >= 0 && lane == lead) base = atomicAdd(s.start + (size_t)cloud * s.cells + cell, __popc(peers));
    base = __shfl_sync(kAll, base, lead);
    if (cell >= 0) s.cell_rank[s.first[cloud] + r] = make_int2(cell, base + __popc(peers & ((1u << lane) - 1u)));
}

__device__ __forceinline__ int block_sum_1024(int v, int *s_w) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kAll, v, o);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = v;
    __syncthreads();
    int t = s_w[threadIdx.x & 31];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(kAll, t, o);
    __syncthreads();
    return t;
}

// cells 4 t .. 4 t + 3 of a tile, 0 past the grid's end
__device__ __forceinline__ int4 tile_cells(const NnSide &s, const int *start, int tile) {
    const int i = tile * kNnTile + 4 * threadIdx.x;
    if (i + 3 < s.cells) return *reinterpret_cast<const int4 *>(start + i);
    int4 v = make_int4(0, 0, 0, 0);
    if (i < s.cells) v.x = start[i];
    if (i + 1 < s.cells) v.y = start[i + 1];
    if (i + 2 < s.cells) v.z = start[i + 2];
    return v;
}

__global__ void __launch_bounds__(1024) k_nn_tiles(NnSide a, NnSide b) {
    const NnSide &s = blockIdx.y ? b : a;
    __shared__ int s_w[32];
    const int cloud = blockIdx.x / s.tiles, tile = blockIdx.x - cloud * s.tiles;
    if (cloud >= s.N) return;   // uniform
    const int4 v = tile_cells(s, s.start + (size_t)cloud * s.cells, tile);
    const int t = block_sum_1024(v.x + v.y + v.z + v.w, s_w);
    if (threadIdx.x == 0) s.tile_sum[(size_t)cloud * s.tiles + tile] = t;
}

__global__ void __launch_bounds__(1024) k_nn_starts(NnSide a, NnSide b) {
    const NnSide &s = blockIdx.y ? b : a;
    __shared__ int s_w[32];
    const int cloud = blockIdx.x / s.tiles, tile = blockIdx.x - cloud * s.tiles;
    if (cloud >= s.N) return;   // uniform
    int before = 0;
    for (int i = threadIdx.x; i < tile; i += 1024) before += s.tile_sum[(size_t)cloud * s.tiles + i];
    before = block_sum_1024(before, s_w);
    int *start = s.start + (size_t)cloud * s.cells;
    int4 v = tile_cells(s, start, tile);
    const int mine = v.x + v.y + v.z + v.w, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kAll, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_w[w] = x;
    __syncthreads();
    int t = s_w[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kAll, t, o);
        if (lane >= o) t += y;
    }
    const int warps_before = w ? __shfl_sync(kAll, t, w - 1) : 0;
    const int e = before + warps_before + x - mine;
    v = make_int4(e, e + v.x, e + v.x + v.y, e + v.x + v.y + v.z);
    const int i = tile * kNnTile + 4 * threadIdx.x;
    if (i + 3 < s.cells) {
        *reinterpret_cast<int4 *>(start + i) = v;
    } else {
        if (i < s.cells) start[i] = v.x;
        if (i + 1 < s.cells) start[i + 1] = v.y;
        if (i + 2 < s.cells) start[i + 2] = v.z;
    }
}

template <int D>
__global__ void __launch_bounds__(256) k_nn_scatter(NnSide a, NnSide b) {
    const NnSide &s = blockIdx.y ? b : a;
    int cloud, n;
    long long row0;
    if (!tile_of(s, blockIdx.x, 8, cloud, row0, n)) return;
    const long long r = row0 + threadIdx.x;
    if (r >= n) return;
    const long long first = s.first[cloud];
    float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < D; ++c) v[c] = __ldg(s.x + (first + r) * D + c);
    const int2 cr = s.cell_rank[first + r];
    const long long at = first + s.start[(size_t)cloud * s.cells + cr.x] + cr.y;
    if (D < 4) v[3] = __int_as_float((int)r);
    else s.row[at] = (int)r;
    s.pts[at] = make_float4(v[0], v[1], v[2], v[3]);
}

template <int D>
__global__ void __launch_bounds__(kNode) k_nn_boxes(NnSide a, NnSide b) {
    const NnSide &s = blockIdx.y ? b : a;
    __shared__ unsigned s_box[2][4][32];
    int cloud, n;
    long long row0;
    if (!tile_of(s, blockIdx.x, 10, cloud, row0, n)) return;   // uniform for the block
    const long long r = row0 + threadIdx.x, first = s.first[cloud];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
    const bool has = r < n;
    if (has) p = s.pts[first + r];
    const float v[4] = {p.x, p.y, p.z, p.w};
    float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < D; ++c) {
        // NaN coordinates (never a neighbour) leave the box alone
        const bool use = has && v[c] == v[c];
        const unsigned h = __reduce_max_sync(kAll, use ? enc(v[c]) : enc(-INFINITY));
        const unsigned l = __reduce_min_sync(kAll, use ? enc(v[c]) : enc(INFINITY));
        hi[c] = dec(h);
        lo[c] = dec(l);
        if (lane == 0) { s_box[0][c][w] = h; s_box[1][c][w] = l; }
    }
    const int leaves = (n + kLeaf - 1) / kLeaf, leaf = (int)(row0 >> 5) + w;
    if (lane == 0 && leaf < leaves) {
        float4 *o = s.leaf + 2 * ((first >> 5) + cloud + leaf);
        o[0] = make_float4(lo[0], lo[1], lo[2], lo[3]);
        o[1] = make_float4(hi[0], hi[1], hi[2], hi[3]);
    }
    __syncthreads();
    if (w != 0) return;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        hi[c] = dec(__reduce_max_sync(kAll, s_box[0][c][lane]));
        lo[c] = dec(__reduce_min_sync(kAll, s_box[1][c][lane]));
    }
    if (lane == 0) {
        float4 *o = s.node + 2 * ((first >> 10) + cloud + (row0 >> 10));
        o[0] = make_float4(lo[0], lo[1], lo[2], lo[3]);
        o[1] = make_float4(hi[0], hi[1], hi[2], hi[3]);
    }
}

// ---------------------------------------------------------------------------
// searching
// ---------------------------------------------------------------------------
template <int D>
struct Box {
    float lo[D], hi[D];
};

template <int D>
__device__ __forceinline__ Box<D> load_box(const float4 *b) {
    const float4 l = __ldg(b), h = __ldg(b + 1);
    const float lv[4] = {l.x, l.y, l.z, l.w}, hv[4] = {h.x, h.y, h.z, h.w};
    Box<D> r;
#pragma unroll
    for (int c = 0; c < D; ++c) { r.lo[c] = lv[c]; r.hi[c] = hv[c]; }
    return r;
}

// squared distance between a box and the box [lo, hi] (a point: lo = hi), in
// the steps of the ranking distance
template <int D>
__device__ __forceinline__ float box_dist(const Box<D> &b, const float (&lo)[D], const float (&hi)[D]) {
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        const float t = fmaxf(fmaxf(__fsub_rn(b.lo[c], hi[c]), __fsub_rn(lo[c], b.hi[c])), 0.f);
        s = c == 0 ? __fmul_rn(t, t) : __fmaf_rn(t, t, s);
    }
    return s;
}

template <int D>
__device__ __forceinline__ float point_dist(const float (&q)[D], const float (&p)[D]) {
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        const float t = __fsub_rn(q[c], p[c]);
        s = c == 0 ? __fmul_rn(t, t) : __fmaf_rn(t, t, s);
    }
    return s;
}

__device__ __forceinline__ bool before(float d, int j, float e, int k) { return d < e || (d == e && j < k); }

// lane of the smallest non-negative value (NaN counts as larger than all)
__device__ __forceinline__ int nearest_lane(float v, unsigned &bits) {
    const unsigned u = __float_as_uint(v);
    bits = __reduce_min_sync(kAll, u);
    return __ffs(__ballot_sync(kAll, u == bits)) - 1;
}

constexpr unsigned kDone = 0x7fffffffu;   // above every distance, +inf included

// Ascending list of the K nearest, right-aligned in KM slots: the slots below
// KM - K hold -inf and never move, an empty slot is (+inf, -1), which no
// candidate at distance +inf precedes.
template <int KM>
struct Nearest {
    float z[KM];
    int f[KM];
    __device__ __forceinline__ void init(int K) {
#pragma unroll
        for (int k = 0; k < KM; ++k) {
            z[k] = k < KM - K ? -INFINITY : INFINITY;
            f[k] = -1;
        }
    }
    // every comparison against the old list, so the moves form no chain
    __device__ __forceinline__ void insert(float d, int j) {
        bool c = before(d, j, z[KM - 1], f[KM - 1]);
#pragma unroll
        for (int k = KM - 1; k >= 0; --k) {
            const bool cp = k > 0 && before(d, j, z[k > 0 ? k - 1 : 0], f[k > 0 ? k - 1 : 0]);
            z[k] = c ? (cp ? z[k > 0 ? k - 1 : 0] : d) : z[k];
            f[k] = c ? (cp ? f[k > 0 ? k - 1 : 0] : j) : f[k];
            c = cp;
        }
    }
};

constexpr int kLaneThreads = 128;
constexpr int kLaneShift = 7, kWarpShift = 2;   // queries per block, as powers of two

// Sorted candidate at global place `at` and its row.
template <int D>
__device__ __forceinline__ int load_leaf(const NnSide &s, long long at, float (&v)[D]) {
    const float4 p = __ldg(s.pts + at);
    const float x[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
    for (int c = 0; c < D; ++c) v[c] = x[c];
    return D < 4 ? __float_as_int(p.w) : s.row[at];
}

// Candidate of row `at`, for the scan; past the end one that is never inserted
// (distance +inf or NaN).
template <int D>
__device__ __forceinline__ void load_row(const NnSide &s, long long first, int cn, int at, float (&v)[D]) {
    if (at < cn) {
        load_point<D>(s.x, first + at, v);
    } else {
#pragma unroll
        for (int c = 0; c < D; ++c) v[c] = INFINITY;
    }
}

// A query per lane.  The warp's 32 queries are neighbours on the curve; it
// walks nodes and leaves in order of their distance to the queries' common
// box, nearest first, until none lies within the largest K-th distance.  In a
// leaf every lane marks the candidates within its own K-th distance (a mask
// of 32 bits), then inserts its marked ones, each lane its own at a time: the
// warp takes as many insertion steps as its busiest lane, not as many as
// there are candidates any lane wants.
template <int D, int KM>
__global__ void __launch_bounds__(kLaneThreads, KM <= 8 ? 8 : 4) k_nn_lanes(NnQuery a) {
    __shared__ __align__(16) float s_c[kLaneThreads / 32][D + 1][32];
    int cloud, n;
    long long row0;
    bool scan;
    if (!query_tile(a.q, blockIdx.x, kLaneShift, cloud, row0, n, scan)) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long pos = row0 + threadIdx.x;
    if (row0 + (w << 5) >= n) return;   // uniform for the warp; no block barrier below
    const bool valid = pos < n;
    const long long qfirst = a.q.first[cloud], cfirst = a.c.first[cloud];
    const int cn = (int)a.c.len[cloud];
    float q[D];
    int qrow = 0;
    {
        const long long r = valid ? pos : n - 1, at = qfirst + r;
        if (scan) {
            load_point<D>(a.q.x, at, q);
            qrow = (int)r;
        } else {
            const float4 p = __ldg(a.q.pts + at);
            const float v[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
            for (int c = 0; c < D; ++c) q[c] = v[c];
            qrow = D < 4 ? __float_as_int(p.w) : a.q.row[at];
        }
    }
    float glo[D], ghi[D];
#pragma unroll
    for (int c = 0; c < D; ++c) {
        glo[c] = dec(__reduce_min_sync(kAll, enc(q[c])));
        ghi[c] = dec(__reduce_max_sync(kAll, enc(q[c])));
    }
    Nearest<KM> L;
    L.init(a.K);
    const int nleaf = (cn + kLeaf - 1) / kLeaf, nnode = (cn + kNode - 1) / kNode;
    const float4 *leafbox = a.c.leaf + 2 * ((cfirst >> 5) + cloud);
    const float4 *nodebox = a.c.node + 2 * ((cfirst >> 10) + cloud);
    auto thr = [&]() { return valid ? L.z[KM - 1] : -1.f; };
    // the lane's own candidate of 32, offered to every lane's query
    auto offer = [&](const float (&v)[D], int row) {
        __syncwarp();   // the previous candidates are done with
#pragma unroll
        for (int c = 0; c < D; ++c) s_c[w][c][lane] = v[c];
        s_c[w][D][lane] = __int_as_float(row);
        __syncwarp();
        if constexpr (KM == 1) {   // a running minimum, no mask
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                float p[D];
#pragma unroll
                for (int c = 0; c < D; ++c) p[c] = s_c[w][c][j];
                const float d = point_dist<D>(q, p);
                const int f = __float_as_int(s_c[w][D][j]);
                const bool take = before(d, f, L.z[0], L.f[0]);
                L.z[0] = take ? d : L.z[0];
                L.f[0] = take ? f : L.f[0];
            }
            return;
        }
        unsigned mask = 0;
        const float t = thr();
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            float p[D];
#pragma unroll
            for (int c = 0; c < D; ++c) p[c] = s_c[w][c][j];
            if (point_dist<D>(q, p) <= t) mask |= 1u << j;
        }
        while (__any_sync(kAll, mask != 0u)) {
            if (mask) {
                const int j = __ffs(mask) - 1;
                mask &= mask - 1;
                float p[D];
#pragma unroll
                for (int c = 0; c < D; ++c) p[c] = s_c[w][c][j];   // lanes' j differ in bank, or read one word
                const float d = point_dist<D>(q, p);
                const int f = __float_as_int(s_c[w][D][j]);
                if (before(d, f, L.z[KM - 1], L.f[KM - 1])) L.insert(d, f);
            }
        }
    };
    auto visit = [&](int leaf) {
        const int at = leaf * kLeaf + lane;
        float v[D];
        int row = 0;
        if (at < cn) {
            row = load_leaf<D>(a.c, cfirst + at, v);
        } else {
#pragma unroll
            for (int c = 0; c < D; ++c) v[c] = INFINITY;   // distance +inf or NaN: never inserted
        }
        offer(v, row);
    };
    int seed = -1;
    if (cn > 0 && !scan) {
        // the leaf where the middle query would lie: a first bound
        float m[D];
#pragma unroll
        for (int c = 0; c < D; ++c) m[c] = __shfl_sync(kAll, q[c], 16);
        const int s = __ldg(a.c.start + (size_t)cloud * a.c.cells + cell_of<D>(a.c, kept_grid<D>(a.c, cloud), m));
        seed = min(s / kLeaf, nleaf - 1);
        visit(seed);
    }
    unsigned bits;
    for (int nb = 0; nb < nnode && !scan; nb += 32) {
        float nd = __uint_as_float(kDone);
        if (nb + lane < nnode) nd = box_dist<D>(load_box<D>(nodebox + 2 * (nb + lane)), glo, ghi);
        while (true) {
            const int nl = nearest_lane(nd, bits);
            const float wthr = __int_as_float(__reduce_max_sync(kAll, __float_as_int(thr())));
            if (bits == kDone || !(__uint_as_float(bits) <= wthr)) break;
            if (lane == nl) nd = __uint_as_float(kDone);
            const int base = (nb + nl) * 32;
            float ld = __uint_as_float(kDone);
            if (base + lane < nleaf && base + lane != seed)
                ld = box_dist<D>(load_box<D>(leafbox + 2 * (base + lane)), glo, ghi);
            while (true) {
                const int ll = nearest_lane(ld, bits);
                const float lthr = __int_as_float(__reduce_max_sync(kAll, __float_as_int(thr())));
                if (bits == kDone || !(__uint_as_float(bits) <= lthr)) break;
                if (lane == ll) ld = __uint_as_float(kDone);
                const float own = box_dist<D>(load_box<D>(leafbox + 2 * (base + ll)), q, q);
                if (__any_sync(kAll, own <= thr())) visit(base + ll);
            }
        }
    }
    if (scan) {
        float v[D];
        load_row<D>(a.c, cfirst, cn, lane, v);
        for (int at = lane; at - lane < cn; at += 32) {
            float next[D];   // asked for before the present ones are offered
            load_row<D>(a.c, cfirst, cn, at + 32, next);
            if constexpr (KM == 1 && D >= 3) {   // one load of shared memory per candidate, rows in order
                float4 *s4 = reinterpret_cast<float4 *>(s_c[w]);
                __syncwarp();
                s4[lane] = make_float4(v[0], v[1], v[2], v[D - 1]);
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const float4 c4 = s4[j];
                    const float x[4] = {c4.x, c4.y, c4.z, c4.w};
                    float p[D];
#pragma unroll
                    for (int c = 0; c < D; ++c) p[c] = x[c];
                    const float d = point_dist<D>(q, p);
                    const bool take = d < L.z[0];
                    L.z[0] = take ? d : L.z[0];
                    L.f[0] = take ? at - lane + j : L.f[0];
                }
            } else {
                offer(v, at);
            }
#pragma unroll
            for (int c = 0; c < D; ++c) v[c] = next[c];
        }
    }
    if (!valid) return;
    const long long out = (qfirst + qrow) * a.K;
#pragma unroll
    for (int k = 0; k < KM; ++k) {
        const int r = k - (KM - a.K);
        if (r < 0) continue;
        a.idx[out + r] = L.f[k] >= 0 ? cfirst + L.f[k] : -1;
        a.dists[out + r] = L.z[k];
    }
}

// A query per warp: lane k keeps the k-th entry of the list, the 32 lanes
// take a leaf's candidates, and an admitted one is inserted by the whole warp
// (a ballot ranks it, the later entries move one lane up).
template <int D>
__global__ void __launch_bounds__(kLaneThreads, 16) k_nn_warps(NnQuery a) {
    int cloud, n;
    long long row0;
    bool scan;
    if (!query_tile(a.q, blockIdx.x, kWarpShift, cloud, row0, n, scan)) return;
    const int lane = threadIdx.x & 31, K = a.K;
    const long long pos = row0 + (threadIdx.x >> 5);
    if (pos >= n) return;   // uniform for the warp; no block barrier below
    const long long qfirst = a.q.first[cloud], cfirst = a.c.first[cloud];
    const int cn = (int)a.c.len[cloud];
    float q[D];
    int qrow;
    if (scan) {
        load_point<D>(a.q.x, qfirst + pos, q);
        qrow = (int)pos;
    } else {
        const float4 p = __ldg(a.q.pts + qfirst + pos);
        const float v[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
        for (int c = 0; c < D; ++c) q[c] = v[c];
        qrow = D < 4 ? __float_as_int(p.w) : a.q.row[qfirst + pos];
    }
    float ez = INFINITY, tz = INFINITY;   // this lane's entry, the K-th entry
    int ef = -1, tf = -1;
    const int nleaf = (cn + kLeaf - 1) / kLeaf, nnode = (cn + kNode - 1) / kNode;
    const float4 *leafbox = a.c.leaf + 2 * ((cfirst >> 5) + cloud);
    const float4 *nodebox = a.c.node + 2 * ((cfirst >> 10) + cloud);
    // the lanes' 32 candidates, offered to the query
    auto offer = [&](float d, int f) {
        if (K == 1) {
            if (!before(d, f, tz, tf)) { d = INFINITY; f = INT_MAX; }   // NaN as well
            const unsigned u = __float_as_uint(d), m = __reduce_min_sync(kAll, u);
            if (m != 0x7f800000u) {
                tf = __reduce_min_sync(kAll, u == m ? f : INT_MAX);
                tz = __uint_as_float(m);
                ez = tz;
                ef = tf;
            }
            return;
        }
        unsigned pend = __ballot_sync(kAll, before(d, f, tz, tf));
        while (pend) {
            const int src = __ffs(pend) - 1;
            pend &= pend - 1;
            const float nd = __shfl_sync(kAll, d, src);
            const int nf = __shfl_sync(kAll, f, src);
            if (!before(nd, nf, tz, tf)) continue;   // uniform
            const int at_k = __popc(__ballot_sync(kAll, lane < K && before(ez, ef, nd, nf)));
            const float pz = __shfl_up_sync(kAll, ez, 1);
            const int pf = __shfl_up_sync(kAll, ef, 1);
            ez = lane < at_k ? ez : (lane == at_k ? nd : pz);
            ef = lane < at_k ? ef : (lane == at_k ? nf : pf);
            tz = __shfl_sync(kAll, ez, K - 1);
            tf = __shfl_sync(kAll, ef, K - 1);
        }
    };
    auto visit = [&](int leaf) {
        const int at = leaf * kLeaf + lane;
        float d = INFINITY;
        int f = INT_MAX;
        if (at < cn) {
            float v[D];
            f = load_leaf<D>(a.c, cfirst + at, v);
            d = point_dist<D>(q, v);
        }
        offer(d, f);
    };
    if (!scan) {
        int seed = -1;
        if (cn > 0) {
            seed = min(__ldg(a.c.start + (size_t)cloud * a.c.cells + cell_of<D>(a.c, kept_grid<D>(a.c, cloud), q)) / kLeaf, nleaf - 1);
            visit(seed);
        }
        unsigned bits;
        for (int nb = 0; nb < nnode; nb += 32) {
            float nd = __uint_as_float(kDone);
            if (nb + lane < nnode) nd = box_dist<D>(load_box<D>(nodebox + 2 * (nb + lane)), q, q);
            while (true) {
                const int nl = nearest_lane(nd, bits);
                if (bits == kDone || !(__uint_as_float(bits) <= tz)) break;
                if (lane == nl) nd = __uint_as_float(kDone);
                const int base = (nb + nl) * 32;
                float ld = __uint_as_float(kDone);
                if (base + lane < nleaf && base + lane != seed)
                    ld = box_dist<D>(load_box<D>(leafbox + 2 * (base + lane)), q, q);
                while (true) {
                    const int ll = nearest_lane(ld, bits);
                    if (bits == kDone || !(__uint_as_float(bits) <= tz)) break;
                    if (lane == ll) ld = __uint_as_float(kDone);
                    visit(base + ll);
                }
            }
        }
    } else if (K == 1) {   // each lane its own candidates, in order of their rows
        float z = INFINITY;
        int f = INT_MAX;
#pragma unroll 4
        for (int at = lane; at < cn; at += 32) {
            float v[D];
            load_point<D>(a.c.x, cfirst + at, v);
            const float d = point_dist<D>(q, v);
            f = d < z ? at : f;
            z = d < z ? d : z;
        }
        const unsigned u = __float_as_uint(z), m = __reduce_min_sync(kAll, u);
        if (m != 0x7f800000u) {
            ef = __reduce_min_sync(kAll, u == m ? f : INT_MAX);
            ez = __uint_as_float(m);
        }
    } else {
        float v[2][D];   // two rounds ahead
        load_row<D>(a.c, cfirst, cn, lane, v[0]);
        load_row<D>(a.c, cfirst, cn, lane + 32, v[1]);
        for (int at = lane; at - lane < cn; at += 32) {
            float next[D];
            load_row<D>(a.c, cfirst, cn, at + 64, next);
            offer(point_dist<D>(q, v[0]), at);
#pragma unroll
            for (int c = 0; c < D; ++c) {
                v[0][c] = v[1][c];
                v[1][c] = next[c];
            }
        }
    }
    if (lane < K) {
        const long long out = (qfirst + qrow) * K + lane;
        a.idx[out] = ef >= 0 ? cfirst + ef : -1;
        a.dists[out] = ez;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

// bits per axis: about four cells per point of an average cloud
int bits_for(int64_t N, int64_t P, int D) {
    const double avg = N > 0 ? (double)P / (double)N : 0.0;
    int b = (int)std::lround(std::log2(std::max(2.0, 4.0 * avg)) / D);
    b = std::max(1, std::min(b, 24 / D));
    while (b > 1 && (double)N * (double)(1LL << (b * D)) > 1.5e9) --b;
    return b;
}

void layout_side(NnSide &s, int64_t N, int64_t P, int D, char *ws, size_t &zero, size_t &off) {
    s.N = (int)N;
    s.P = P;
    s.bits = bits_for(N, P, D);
    s.cells = 1 << (s.bits * D);
    s.tiles = (s.cells + kNnTile - 1) / kNnTile;
    s.box = reinterpret_cast<unsigned *>(ws + zero);
    zero = up256(zero + (size_t)N * 8 * sizeof(unsigned));
    s.start = reinterpret_cast<int *>(ws + zero);
    zero = up256(zero + (size_t)N * s.cells * sizeof(int));
    s.span = reinterpret_cast<float *>(ws + off);
    off = up256(off + (size_t)N * 8 * sizeof(float));
    s.grid = reinterpret_cast<float4 *>(ws + off);
    off = up256(off + (size_t)N * 2 * sizeof(float4));
    s.tile_sum = reinterpret_cast<int *>(ws + off);
    off = up256(off + (size_t)N * s.tiles * sizeof(int));
    s.cell_rank = reinterpret_cast<int2 *>(ws + off);
    off = up256(off + (size_t)P * sizeof(int2));
    s.pts = reinterpret_cast<float4 *>(ws + off);
    off = up256(off + (size_t)P * sizeof(float4));
    s.row = reinterpret_cast<int *>(ws + off);
    off = up256(off + (D == 4 ? (size_t)P * sizeof(int) : 0));
    s.leaf = reinterpret_cast<float4 *>(ws + off);
    off = up256(off + (size_t)((P >> 5) + N + 1) * 2 * sizeof(float4));
    s.node = reinterpret_cast<float4 *>(ws + off);
    off = up256(off + (size_t)((P >> 10) + N + 1) * 2 * sizeof(float4));
}

// both sides; the part to be zeroed first comes first, the control word at its head.  Returns the total,
// `zero` its leading bytes.
size_t layout(NnSide (&sides)[2], int64_t N, int64_t P1, int64_t P2, int D, char *ws, size_t &zero) {
    size_t z = 0, off = 0;
    for (int pass = 0; pass < 2; ++pass) {   // the first pass finds the length of the zeroed part
        off = z;
        z = up256(sizeof(NnControl));
        sides[0].control = sides[1].control = reinterpret_cast<NnControl *>(ws);
        layout_side(sides[0], N, P1, D, ws, z, off);
        layout_side(sides[1], N, P2, D, ws, z, off);
    }
    zero = z;
    return off;
}

template <int D>
cudaError_t build_t(NnSide (&s)[2], int64_t N, bool boxes1, size_t zero, char *ws, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(ws, 0, zero, st);
    if (e != cudaSuccess) return e;
    const int64_t P = std::max(s[0].P, s[1].P);
    const unsigned g12 = (unsigned)((P >> 12) + N), g10 = (unsigned)((P >> 10) + N), g8 = (unsigned)((P >> 8) + N);
    const unsigned gt = (unsigned)(N * std::max(s[0].tiles, s[1].tiles));
    k_nn_bounds<D><<<dim3(g12 + 1 + (unsigned)N, 2), 256, 0, st>>>(s[0], s[1]);
    k_nn_count<D><<<dim3(g8, 2), 256, 0, st>>>(s[0], s[1]);
    if (s[0].tiles > 1 || s[1].tiles > 1) k_nn_tiles<<<dim3(gt, 2), 1024, 0, st>>>(s[0], s[1]);
    k_nn_starts<<<dim3(gt, 2), 1024, 0, st>>>(s[0], s[1]);
    k_nn_scatter<D><<<dim3(g8, 2), 256, 0, st>>>(s[0], s[1]);
    if (boxes1) k_nn_boxes<D><<<dim3(g10, 2), kNode, 0, st>>>(s[0], s[1]);
    else k_nn_boxes<D><<<dim3((unsigned)((s[1].P >> 10) + N), 1), kNode, 0, st>>>(s[1], s[1]);
    return cudaGetLastError();
}

template <int D>
cudaError_t search_t(const NnQuery &a, bool warps, cudaStream_t st) {
    if (warps) {
        k_nn_warps<D><<<(unsigned)((a.q.P >> kWarpShift) + a.q.N), kLaneThreads, 0, st>>>(a);
        return cudaGetLastError();
    }
    const unsigned g = (unsigned)((a.q.P >> kLaneShift) + a.q.N);
    if (a.K <= 1) k_nn_lanes<D, 1><<<g, kLaneThreads, 0, st>>>(a);
    else if (a.K <= 2) k_nn_lanes<D, 2><<<g, kLaneThreads, 0, st>>>(a);
    else if (a.K <= 4) k_nn_lanes<D, 4><<<g, kLaneThreads, 0, st>>>(a);
    else if (a.K <= 8) k_nn_lanes<D, 8><<<g, kLaneThreads, 0, st>>>(a);
    else if (a.K <= 16) k_nn_lanes<D, 16><<<g, kLaneThreads, 0, st>>>(a);
    else k_nn_lanes<D, 32><<<g, kLaneThreads, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace

// Building takes about 40 us plus the points' share, so short scans stay.
// Measured (D = 3 unless said; index, scan in us of one call):
//   K >= 5: the scan serves admissions one by one; 1 cloud of 100 + 100 points,
//     normally distributed, K = 5: 25, 87, and at D = 1, 2, 3, 4 and K = 5, 8, 16, 32 alike
//     (20 to 33, 37 to 240); 32 clouds of 1,000 + 20, K = 16: 60, 72; 1 of 1,000 + 1,000, K =
//     8: 27, 497; 32 of 50,000 + 50,000: 947, 23,640
//   K <= 4: by the pairs and the length of a candidate cloud; K = 1, 32 of
//     2,500 + 2,500: 87, 90, but D = 1 74, 67 and D = 2 82, 75, whose distances cost the
//     scan less; 32 of 4,000 + 4,000: 101, 168; 1 of 5,000 + 8,192: 31, 43; 1 of 1,000 +
//     32,000: 33, 101
// The order of two or three distinct points repeated thousands of times parts
// nothing, and the scan, which meets equal distances in the order of their rows,
// stays up to 6 times as fast there (D = 1, coordinates of -1 and 1 only).
bool nn_index_wins(int64_t N, int64_t P1, int64_t P2, int D, int K) {
    if (N <= 0 || P1 <= 0 || P2 <= 0 || N > (1 << 20) || P1 > (1LL << 30) || P2 > (1LL << 30)) return false;
    const double pairs = (double)P1 * (double)P2 / (double)N;
    if (K >= 5) return pairs >= 1e4;
    return pairs >= (D <= 2 ? 3e8 : 2e8) || (pairs >= 3e7 && P2 / N >= 8192);
}

// Whether a search gives every query a warp instead of a lane.  A warp per
// query needs no neighbours to share its walk and fills the GPU with few
// queries; a lane per query shares loads and box tests among 32.  Measured
// (D = 3; warps, lanes in us): K = 1: 32 clouds of 2,000 + 2,000 points 79,
// 81; 32 of 4,000 136, 114; 1 of 30,000 65, 144; 32 of 50,000 1,429, 755; K = 8:
// 32 of 2,000 151, 114; 1 of 30,000 104, 230; 32 of 50,000 3,299, 1,441.  Above
// K = 8 a lane's insertions are long (K = 20: 32 of 50,000 4,737, 6,596),
// unless 32 queries share the very same few candidates (32 of 50,000 + 1,000:
// 3,617, 1,831).
bool nn_search_per_warp(int64_t P1, int64_t P2, int K) {
    if (P1 <= P2 / 8) return true;
    if (K > 8) return P1 < 8 * P2 || P1 < 200000;
    return P1 < (K <= 4 ? 100000 : 60000);
}

size_t nn_index_bytes(int64_t N, int64_t P1, int64_t P2, int D) {
    NnSide s[2];
    size_t zero;
    return layout(s, N, P1, P2, D, nullptr, zero);
}

cudaError_t nn_index_build(NnSide (&s)[2], const float *p1, int64_t P1, const int64_t *first1, const int64_t *len1,
                           const float *p2, int64_t P2, const int64_t *first2, const int64_t *len2, int64_t N, int D,
                           int K, bool both_ways, long long *plans, char *ws, cudaStream_t st) {
    size_t zero;
    layout(s, N, P1, P2, D, ws, zero);
    s[0].plan = plans;
    s[0].per = 1 << (nn_search_per_warp(P1, P2, K) ? kWarpShift : kLaneShift);
    s[1].plan = both_ways ? plans + N + 1 : nullptr;
    s[1].per = 1 << (nn_search_per_warp(P2, P1, K) ? kWarpShift : kLaneShift);
    s[0].x = p1;
    s[0].first = first1;
    s[0].len = len1;
    s[1].x = p2;
    s[1].first = first2;
    s[1].len = len2;
    switch (D) {
        case 1: return build_t<1>(s, N, both_ways, zero, ws, st);
        case 2: return build_t<2>(s, N, both_ways, zero, ws, st);
        case 3: return build_t<3>(s, N, both_ways, zero, ws, st);
        default: return build_t<4>(s, N, both_ways, zero, ws, st);
    }
}

cudaError_t nn_index_search(const NnSide &q, const NnSide &c, int D, int K, int64_t *idx, float *dists,
                            cudaStream_t st) {
    const NnQuery a{q, c, idx, dists, K};
    const bool warps = nn_search_per_warp(q.P, c.P, K);
    switch (D) {
        case 1: return search_t<1>(a, warps, st);
        case 2: return search_t<2>(a, warps, st);
        case 3: return search_t<3>(a, warps, st);
        default: return search_t<4>(a, warps, st);
    }
}

}  // namespace mr
