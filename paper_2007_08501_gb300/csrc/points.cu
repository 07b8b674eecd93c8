// Point-cloud rasterizer and compositing for sm_103a (Section 3.2 of the
// paper, "Differentiable point cloud renderer"), with the C ABI of
// include/points.h.
//
//   k_pstage   double-float projection, 32-byte record per point (NDC position
//              hi/lo, depth), bin counts; eight points per thread and a block's
//              counts in shared memory where there are many
//   k_scan     (shared with the mesh rasterizer) clamp counts, prefix scan
//   k_pfill    append depth-keyed entries to the points' bins, as many to a thread
//   k_sort_long (sort_long.cu) where bins may hold more than kLongList
//              entries: long lists, where few are long
//   k_pfine    persistent blocks over (image, bin) items: the bin's entries
//              front to back in windows, each pixel's points appended in
//              (depth, id) order; stops a bin once every pixel holds K
//   k_pnaive   the plain form: one launch per image, every pixel against
//              every point of its cloud
//   k_pcomp_fwd / k_pcomp_bwd   Alpha / Norm compositing and its adjoint
//   k_prast_bwd  dL/d(zbuf, dists) -> dL/dpoints through the projection
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>

#include "bin_common.cuh"
#include "meshrast.h"
#include "points.h"
#include "rast_common.cuh"
#include "rast_internal.h"

namespace mr {

// Point record (32 bytes): a = (x_hi, y_hi, x_lo, y_lo) in NDC, b = (depth,
// 0, 0, 0); culled points have depth +inf and are never binned.
struct __align__(16) PtRec {
    float4 a, b;
};
static_assert(sizeof(PtRec) == 32, "point record is 32 bytes");

constexpr float kPtSlack = 1e-5f;  // relative widening of a splat's box for binning

struct PtArgs {
    const float *points;
    int64_t P;
    const int64_t *first, *num;
    int N;
    const float *cams;
    float radius, r2;
    int S, K, bin, nb;
    int64_t items;
    PtRec *rec;
    int *cloud;
    int *counts, *cursor;
    const int *eff, *offsets;
    unsigned long long *lists;
    unsigned *queue, *status;
    const long long *total;  // entries of all bins, where long lists are sorted (else NULL)
    const int *maxcount;     // and of the fullest
    int64_t *idx;
    float *zbuf, *dists;
    // rendering on packed slots (distance bits << 32 | id, ended by kPtEnd)
    unsigned long long *slots;
    const float *features;
    float *image;
    int D, mode;
    float inv_r2;
};

constexpr unsigned long long kPtEnd = ~0ull;  // its high word is a NaN: not a distance

// box of a splat, widened so that every pixel passing d < r^2 in fp32 lies in it
__device__ __forceinline__ float4 splat_box(const PtRec &R, float radius) {
    const float w = radius * (1.f + kPtSlack);
    return make_float4(__fsub_rd(R.a.x, w), __fadd_ru(R.a.x, w), __fsub_rd(R.a.y, w), __fadd_ru(R.a.y, w));
}

// squared NDC distance from the pixel centre to the point (corner-relative
// double-float difference, then fp32 squares)
__device__ __forceinline__ float splat_d(const float4 &a, const PixC &p) {
    const float qx = __fadd_rn(__fsub_rn(p.xh, a.x), __fsub_rn(p.xl, a.z));
    const float qy = __fadd_rn(__fsub_rn(p.yh, a.y), __fsub_rn(p.yl, a.w));
    return __fmaf_rn(qx, qx, __fmul_rn(qy, qy));
}

// ---------------------------------------------------------------------------
// staging and binning
// ---------------------------------------------------------------------------
// Points come in any order, so a warp's land in as many bins, and those of the
// one or two clouds the GPU is at share a few dozen cache lines: every addition
// to a count waits its turn at its line.  A block of many points therefore
// counts in shared memory (one cloud's bins, at most kPtHist) and adds each bin
// once; with few points, where blocks must be small, each pair goes to memory.
// 8 x 200,000 points, bins of 8 at 256 px: k_pstage 137 -> 58 us, k_pfill
// 145 -> 53 us.
constexpr int kPtHist = 4096;
constexpr int kPtPerThread = 8;

// record of point i of cloud n (-1: none); returns the cloud, or -1 when culled
__device__ __forceinline__ int stage_point(const PtArgs &a, int64_t i, int n, const float *cam, PtRec &R) {
    R.a = make_float4(0.f, 0.f, 0.f, 0.f);
    R.b = make_float4(__int_as_float(0x7f800000), 0.f, 0.f, 0.f);
    if (n < 0) return -1;
    const float px = a.points[3 * i], py = a.points[3 * i + 1], pz = a.points[3 * i + 2];
    if (!(isfinite(px) && isfinite(py) && isfinite(pz))) {
        set_status(a.status, MESHRAST_ST_NONFINITE);
        return -1;
    }
    df X, Y, Z;
    project_corner(cam, px, py, pz, X, Y, Z);
    const float z = __fadd_rn(Z.hi, Z.lo);
    if (!(z >= cam[13]) || !isfinite(z) || !isfinite(X.hi) || !isfinite(Y.hi)) return -1;
    R.a = make_float4(X.hi, Y.hi, X.lo, Y.lo);
    R.b.x = z;
    return n;
}

__device__ __forceinline__ void point_bins(const PtArgs &a, int n, const PtRec &R, int &bx0, int &bx1, int &by0,
                                           int &by1) {
    bx0 = by0 = 1;
    bx1 = by1 = 0;
    if (n >= 0) bin_rect_box(splat_box(R, a.radius), a.S, a.bin, bx0, bx1, by0, by1);
}

// PER points per thread; HIST: counted in shared memory first (nb * nb <= kPtHist)
template <int PER, bool HIST>
__global__ void __launch_bounds__(256) k_pstage(PtArgs a, int do_count) {
    __shared__ float s_cam[16];
    __shared__ int s_hist[HIST ? kPtHist : 1];
    const int64_t i0 = (int64_t)blockIdx.x * 256 * PER + threadIdx.x;
    const int nb2 = a.nb * a.nb;
    int block;
    int64_t lo, hi;
    block_image(a.first, a.num, a.N, a.P, (int64_t)blockIdx.x * 256 * PER, block, lo, hi);
    if (threadIdx.x < 16 && block >= 0) s_cam[threadIdx.x] = a.cams[16 * block + threadIdx.x];
    if (HIST)
        for (int b = threadIdx.x; b < nb2; b += 256) s_hist[b] = 0;
    __syncthreads();
    for (int u = 0; u < PER; ++u) {
        const int64_t i = i0 + 256 * u;
        PtRec R;
        int n = i < a.P ? image_of(a.first, a.num, a.N, i, block, lo, hi) : -1;
        n = stage_point(a, i, n, n == block ? s_cam : a.cams + 16 * n, R);
        if (i < a.P) {
            reinterpret_cast<float4 *>(a.rec + i)[0] = R.a;
            reinterpret_cast<float4 *>(a.rec + i)[1] = R.b;
            a.cloud[i] = n;
        }
        if (!do_count) continue;
        int bx0, bx1, by0, by1;
        point_bins(a, n, R, bx0, bx1, by0, by1);
        if (!HIST) {
            count_bins(a.counts, n, a.nb, bx0, bx1, by0, by1);
        } else {
            for (int by = by0; by <= by1; ++by)
                for (int bx = bx0; bx <= bx1; ++bx) {
                    if (n == block) atomicAdd(&s_hist[by * a.nb + bx], 1);
                    else atomicAdd(a.counts + (n * a.nb + by) * a.nb + bx, 1);
                }
        }
    }
    if (!HIST || !do_count) return;
    __syncthreads();
    for (int b = threadIdx.x; b < nb2; b += 256)
        if (s_hist[b] > 0) atomicAdd(a.counts + block * nb2 + b, s_hist[b]);
}

template <int PER, bool HIST>
__global__ void __launch_bounds__(256) k_pfill(PtArgs a) {
    __shared__ int s_hist[HIST ? kPtHist : 1];
    const int64_t i0 = (int64_t)blockIdx.x * 256 * PER + threadIdx.x;
    const int nb2 = a.nb * a.nb;
    int block = -1;
    if (HIST) {
        int64_t lo, hi;
        block_image(a.first, a.num, a.N, a.P, (int64_t)blockIdx.x * 256 * PER, block, lo, hi);
        for (int b = threadIdx.x; b < nb2; b += 256) s_hist[b] = 0;
        __syncthreads();
    }
    auto load = [&](int64_t i, PtRec &R) {
        const int n = i < a.P ? a.cloud[i] : -1;
        if (n >= 0) {
            R.a = reinterpret_cast<const float4 *>(a.rec + i)[0];
            R.b = reinterpret_cast<const float4 *>(a.rec + i)[1];
        }
        return n;
    };
    // depth in the high word, so that integer order is front to back, ties by id
    auto entry = [](const PtRec &R, int64_t i) {
        return ((unsigned long long)signed_key_bits(R.b.x) << 32) | (unsigned)i;
    };
    if constexpr (!HIST) {
        for (int u = 0; u < PER; ++u) {
            const int64_t i = i0 + 256 * u;
            PtRec R;
            int bx0, bx1, by0, by1;
            const int n = load(i, R);
            point_bins(a, n, R, bx0, bx1, by0, by1);
            fill_bins(a.lists, a.cursor, a.eff, a.offsets, n >= 0 ? entry(R, i) : 0ull, n, a.nb, bx0, bx1, by0, by1);
        }
    } else {
        for (int u = 0; u < PER; ++u) {
            PtRec R;
            int bx0, bx1, by0, by1;
            const int n = load(i0 + 256 * u, R);
            if (n < 0 || n != block) continue;
            point_bins(a, n, R, bx0, bx1, by0, by1);
            for (int by = by0; by <= by1; ++by)
                for (int bx = bx0; bx <= bx1; ++bx) atomicAdd(&s_hist[by * a.nb + bx], 1);
        }
        __syncthreads();
        // the block's place in each of its bins
        for (int b = threadIdx.x; b < nb2; b += 256)
            if (s_hist[b] > 0) s_hist[b] = atomicAdd(a.cursor + block * nb2 + b, s_hist[b]);
        __syncthreads();
        for (int u = 0; u < PER; ++u) {
            const int64_t i = i0 + 256 * u;
            PtRec R;
            int bx0, bx1, by0, by1;
            const int n = load(i, R);
            if (n < 0) continue;
            point_bins(a, n, R, bx0, bx1, by0, by1);
            for (int by = by0; by <= by1; ++by)
                for (int bx = bx0; bx <= bx1; ++bx) {
                    const int key = (n * a.nb + by) * a.nb + bx;
                    const int slot = n == block ? atomicAdd(&s_hist[by * a.nb + bx], 1) : atomicAdd(a.cursor + key, 1);
                    if (slot < a.eff[key]) a.lists[a.offsets[key] + slot] = entry(R, i);
                }
        }
    }
}

// ---------------------------------------------------------------------------
// writing one pixel's K fragments
// ---------------------------------------------------------------------------
__device__ __forceinline__ void pt_slot(const PtArgs &a, int64_t s, int id, const PixC &p) {
    if (id == 0x7fffffff) {
        a.idx[s] = -1;
        a.zbuf[s] = -1.f;
        a.dists[s] = -1.f;
    } else {
        a.idx[s] = id;
        a.zbuf[s] = __ldg(reinterpret_cast<const float *>(a.rec + id) + 4);
        a.dists[s] = splat_d(__ldg(reinterpret_cast<const float4 *>(a.rec + id)), p);
    }
}

template <int KM>
__device__ __forceinline__ void pt_write(const PtArgs &a, int64_t pix, const TopK<KM> &tk, const PixC &p) {
    const int64_t s0 = pix * (int64_t)a.K;
    if (a.K == KM && (KM % 4) == 0) {
        longlong2 *ip = reinterpret_cast<longlong2 *>(a.idx + s0);
        float4 *zp = reinterpret_cast<float4 *>(a.zbuf + s0);
        float4 *dp = reinterpret_cast<float4 *>(a.dists + s0);
#pragma unroll
        for (int j = 0; j < KM / 2; ++j) {
            longlong2 v;
            v.x = tk.f[2 * j] == 0x7fffffff ? -1ll : (long long)tk.f[2 * j];
            v.y = tk.f[2 * j + 1] == 0x7fffffff ? -1ll : (long long)tk.f[2 * j + 1];
            ip[j] = v;
        }
#pragma unroll
        for (int j = 0; j < KM / 4; ++j) {
            float zz[4], dd[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int k = 4 * j + i;
                const bool e = tk.f[k] == 0x7fffffff;
                zz[i] = e ? -1.f : tk.z[k];
                dd[i] = e ? -1.f : splat_d(__ldg(reinterpret_cast<const float4 *>(a.rec + tk.f[k])), p);
            }
            zp[j] = make_float4(zz[0], zz[1], zz[2], zz[3]);
            dp[j] = make_float4(dd[0], dd[1], dd[2], dd[3]);
        }
        return;
    }
#pragma unroll
    for (int k = 0; k < KM; ++k) {
        if (k < KM - a.K) continue;
        pt_slot(a, s0 + k - (KM - a.K), tk.f[k], p);
    }
}

// ---------------------------------------------------------------------------
// fine pass: persistent blocks, one bin per item
// ---------------------------------------------------------------------------
// A splat's depth is the same at every pixel, so once a bin's entries are in
// (depth, id) order every pixel gets its fragments by appending.  Per window of
// the bin's list (depth buckets, bin_common.cuh):
//   1. the entries of a bucket (a handful; a list sorted before is in order) are put in order by counting, for
//      each, the bucket's smaller ones;
//   2. small splats: one thread per point sets the point's bit in the row of
//      each pixel it covers; large splats: a warp walks the points for its 32
//      pixels (below);
//   3. one thread per pixel appends the points of its row's bits until it
//      holds K.
// The tile is then written slot by slot, coalesced.  Walking the points pixel
// by pixel is what bounded small splats: at the benchmark's 1.28 pixel radius a
// point covers 5 of a warp's 32 pixels.  8 clouds of 200,000 points, 256 px, K =
// 50, bins of 8: 874 -> 275 us; 3 clouds of 9,000 at 100 px, K = 10, bins of 16:
// 165 -> 36 us.
// 256 threads also for the 64 pixels of a bin of 8: the ordering and the tile's
// slots take them all, and 512 entries a window keep 5 blocks on an SM (8 x
// 200,000 points, forward and backward: 128 threads and 1,024 entries 645 us, 256
// and 1,024 584, 256 and 512 574, 64 and 512 736)
constexpr int kPfineThreads = 256, kPfineWindow = 512;
constexpr int kPtCount = 64;  // a bucket beyond this has its window sorted instead

// Composites a pixel's points, ids and 1 - alpha in shared memory (the
// arithmetic of k_pcomp_fwd).
template <int DM>
__device__ __forceinline__ void pt_composite(const PtArgs &a, const int *ids, const float *q, int held, int64_t pix) {
    float acc[DM], T = 1.f, asum = 0.f;
#pragma unroll
    for (int ch = 0; ch < DM; ++ch) acc[ch] = 0.f;
    for (int k = 0; k < held; ++k) {
        const float *f = a.features + (int64_t)ids[k] * a.D;
        const float al = 1.f - q[k];
        const float wgt = a.mode == PTS_COMPOSITE_ALPHA ? al * T : al;
#pragma unroll
        for (int ch = 0; ch < DM; ++ch)
            if (ch < a.D) acc[ch] += wgt * __ldg(f + ch);
        T *= q[k];
        asum += al;
    }
    const float sc = a.mode == PTS_COMPOSITE_NORM ? (asum > 0.f ? 1.f / asum : 0.f) : 1.f;
#pragma unroll
    for (int ch = 0; ch < DM; ++ch)
        if (ch < a.D) a.image[pix * a.D + ch] = acc[ch] * sc;
}

// RENDER: the tile's pixels are composited and their points left as packed
// slots, 8 bytes for each there is, in place of 16 for every slot.
template <int BS, bool RENDER>
__global__ void __launch_bounds__(kPfineThreads) k_pfine(PtArgs a) {
    constexpr int BD = kPfineThreads, WIN = kPfineWindow, PX = BS * BS;
    __shared__ WindowShared<WIN, true> s_win;
    __shared__ int s_ids[WIN];             // the window's points, in order
    __shared__ unsigned s_bits[WIN / 32][PX];
    __shared__ float2 s_cx[BS], s_cy[BS];  // pixel centres of the bin's columns and rows
    __shared__ int s_cnt[PX];              // fragments each pixel holds (K outside the image)
    __shared__ int s_item;
    extern __shared__ int s_list[];        // [pixel][K] ids, rows an odd number of words apart
    const int tid = threadIdx.x, lane = tid & 31;
    const int nb2 = a.nb * a.nb, K = a.K, stride = K | 1;
    const int sorted_from = a.total ? long_list(*a.total, *a.maxcount) : 0x7fffffff;
    const unsigned magic_K = (unsigned)((0x100000000ull + (unsigned)K - 1) / (unsigned)K);
    const float w = a.radius * (1.f + kPtSlack);
    // a splat's half width in pixels, with slack for the rounding of its centre's column
    const float rpx = w * 0.5f * (float)a.S + 0.02f;
    // large splats meet in the same pixels, and their bits would queue for the same words
    const bool small = rpx * 2.f < (float)BS;
    while (true) {
        if (tid == 0) s_item = (int)atomicAdd(a.queue, 1u);
        __syncthreads();
        const int item = s_item;
        if ((int64_t)item >= a.items) break;
        const int n = item / nb2, rem = item - n * nb2;
        const int by = rem / a.nb, bx = rem - by * a.nb;
        const int rows = min(BS, a.S - by * BS), cols = min(BS, a.S - bx * BS);
        if (tid < BS) {
            pix_coord(bx * BS + tid, a.S, s_cx[tid].x, s_cx[tid].y);
            pix_coord(by * BS + tid, a.S, s_cy[tid].x, s_cy[tid].y);
        }
        for (int i = tid; i < PX; i += BD) s_cnt[i] = (i / BS < rows && i % BS < cols) ? 0 : K;
        auto centre = [&](int r, int c) { return PixC{s_cx[c].x, s_cx[c].y, s_cy[r].x, s_cy[r].y}; };
        const int cnt = a.eff[item];
        const bool ascending = cnt > sorted_from;
        window_begin<BD>(s_win, a.lists + a.offsets[item], cnt, cnt > 32, ascending);
        while (const int m = window_next<BD>(s_win)) {
            // pieces of a bucket that fits no window come in any order, and so do
            // their entries: those are inserted
            const bool pieces = s_win.st.seg >= 0 && !s_win.st.plain;
            const int lvl = s_win.st.sorted, words = (m + 31) >> 5;
            bool big = false;
            for (int i = tid; i < m && !pieces; i += BD) {
                const unsigned long long e = s_win.ent[i];
                if (ascending) {
                    s_ids[i] = (int)(unsigned)(e & 0xffffffffull);
                    continue;
                }
                int lo = 0, hi = m;
                if (lvl >= 0) {
                    const int k = s_win.rank(s_win.key(e));
                    lo = s_win.pre[lvl][k] - s_win.st.base;
                    hi = s_win.pre[lvl][k + 1] - s_win.st.base;
                }
                big = big || hi - lo > kPtCount;
                if (big) break;
                int at = lo;
                for (int j = lo; j < hi; ++j) at += s_win.ent[j] < e ? 1 : 0;
                s_ids[at] = (int)(unsigned)(e & 0xffffffffull);
            }
            if (small && !pieces)
                for (int i = tid; i < words * PX; i += BD) (&s_bits[0][0])[i] = 0u;
            if (__syncthreads_or(big)) {
                int n2 = 32;
                while (n2 < m) n2 <<= 1;
                for (int i = m + tid; i < n2; i += BD) s_win.ent[i] = ~0ull;
                __syncthreads();
                bitonic_shared<BD>(s_win.ent, n2);
                for (int i = tid; i < m; i += BD) s_ids[i] = (int)(unsigned)(s_win.ent[i] & 0xffffffffull);
                __syncthreads();
            }
            if (small && !pieces) {
                for (int i = tid; i < m; i += BD) {
                    const float4 q = __ldg(reinterpret_cast<const float4 *>(a.rec + s_ids[i]));
                    // columns and rows of the bin within the splat's box (fractional pixel of its centre)
                    const float cf = ((1.f - q.x) * (float)a.S - 1.f) * 0.5f - (float)(bx * BS);
                    const float rf = ((1.f - q.y) * (float)a.S - 1.f) * 0.5f - (float)(by * BS);
                    const int c0 = max(0, (int)ceilf(cf - rpx)), c1 = min(cols - 1, (int)floorf(cf + rpx));
                    const int r0 = max(0, (int)ceilf(rf - rpx)), r1 = min(rows - 1, (int)floorf(rf + rpx));
                    unsigned *row = s_bits[i >> 5];
                    const unsigned bit = 1u << (i & 31);
                    for (int r = r0; r <= r1; ++r)
                        for (int c = c0; c <= c1; ++c)
                            if (splat_d(q, centre(r, c)) < a.r2) atomicOr(row + r * BS + c, bit);
                }
                __syncthreads();
                for (int px = tid; px < PX; px += BD) {
                    int held = s_cnt[px];
                    for (int wd = 0; wd < words && held < K; ++wd) {
                        unsigned bits = s_bits[wd][px];
                        while (bits && held < K) {
                            s_list[px * stride + held++] = s_ids[wd * 32 + __ffs(bits) - 1];
                            bits &= bits - 1;
                        }
                    }
                    s_cnt[px] = held;
                }
            } else {
                // a warp takes 8 x 4 pixels, one per lane, and walks the points whose box meets them
                for (int blk = tid >> 5; blk < PX / 32; blk += BD / 32) {
                    const int r0 = blk / (BS / 8) * 4, c0 = blk % (BS / 8) * 8;
                    if (r0 >= rows || c0 >= cols) continue;  // warp-uniform
                    const int r = r0 + (lane >> 3), c = c0 + (lane & 7), px = r * BS + c;
                    const bool valid = r < rows && c < cols;
                    const PixC p = centre(r, c);
                    const float wx1 = s_cx[c0].x, wx0 = s_cx[min(c0 + 7, cols - 1)].x;
                    const float wy1 = s_cy[r0].x, wy0 = s_cy[min(r0 + 3, rows - 1)].x;
                    int *const l = s_list + px * stride;
                    int held = s_cnt[px];
                    for (int jb = 0; jb < m; jb += 32) {
                        if (!pieces && __all_sync(0xffffffffu, held >= K)) break;
                        float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
                        int id = 0;
                        bool hit = false;
                        if (jb + lane < m) {
                            id = pieces ? (int)(unsigned)(s_win.ent[jb + lane] & 0xffffffffull) : s_ids[jb + lane];
                            q = __ldg(reinterpret_cast<const float4 *>(a.rec + id));
                            hit = q.x - w <= wx1 && q.x + w >= wx0 && q.y - w <= wy1 && q.y + w >= wy0;
                        }
                        unsigned mask = __ballot_sync(0xffffffffu, hit);
                        while (mask) {
                            const int src = __ffs(mask) - 1;
                            mask &= mask - 1;
                            const float4 o = make_float4(__shfl_sync(0xffffffffu, q.x, src), __shfl_sync(0xffffffffu, q.y, src),
                                                         __shfl_sync(0xffffffffu, q.z, src), __shfl_sync(0xffffffffu, q.w, src));
                            const int oid = __shfl_sync(0xffffffffu, id, src);
                            if (!valid || !(splat_d(o, p) < a.r2)) continue;
                            if (!pieces) {
                                if (held < K) l[held++] = oid;
                                continue;
                            }
                            const float z = s_win.key(s_win.ent[jb + src]);
                            auto before = [&](int other) {
                                return key_less(z, oid, __ldg(reinterpret_cast<const float *>(a.rec + other) + 4), other);
                            };
                            if (held == K && !before(l[K - 1])) continue;
                            int k = held < K ? held++ : K - 1;
                            for (; k > 0 && before(l[k - 1]); --k) l[k] = l[k - 1];
                            l[k] = oid;
                        }
                    }
                    if (valid) s_cnt[px] = held;
                }
            }
            // what is left lies behind everything handed out, unless pieces of a bucket remain
            bool full = !pieces;
            __syncthreads();
            for (int px = tid; px < PX; px += BD) full = full && s_cnt[px] >= K;
            if (__syncthreads_and(full)) break;
        }
        __syncthreads();
        if constexpr (RENDER) {
            float *const s_q = reinterpret_cast<float *>(s_list + PX * stride);
            int gw = 1;  // threads per pixel
            while (gw < K && gw < 32) gw <<= 1;
            for (int px = tid / gw; px < PX; px += BD / gw) {
                const int r = px / BS, c = px % BS;
                if (r >= rows || c >= cols) continue;
                const int64_t sl = (((int64_t)n * a.S + by * BS + r) * a.S + bx * BS + c) * K;
                const int held = s_cnt[px];
                const PixC p = centre(r, c);
                for (int k = tid % gw; k < held; k += gw) {
                    const int id = s_list[px * stride + k];
                    const float d = splat_d(__ldg(reinterpret_cast<const float4 *>(a.rec + id)), p);
                    s_q[px * stride + k] = d * a.inv_r2;  // 1 - alpha, without the cancellation
                    a.slots[sl + k] = ((unsigned long long)__float_as_uint(d) << 32) | (unsigned)id;
                }
                if (held < K && tid % gw == 0) a.slots[sl + held] = kPtEnd;
            }
            __syncthreads();
            for (int px = tid; px < PX; px += BD) {
                const int r = px / BS, c = px % BS;
                if (r >= rows || c >= cols) continue;
                const int64_t pix = ((int64_t)n * a.S + by * BS + r) * a.S + bx * BS + c;
                const int *ids = s_list + px * stride;
                const float *q = s_q + px * stride;
                if (a.D == 1) pt_composite<1>(a, ids, q, s_cnt[px], pix);
                else if (a.D <= 4) pt_composite<4>(a, ids, q, s_cnt[px], pix);
                else pt_composite<8>(a, ids, q, s_cnt[px], pix);
            }
            __syncthreads();
            continue;
        }
        // the block writes its tile slot by slot (coalesced along a tile row);
        // quotients by a 32-bit reciprocal, exact for these sizes (< 2^14 slots)
        const int per_row = cols * K;
        const unsigned magic_row = (unsigned)((0x100000000ull + (unsigned)per_row - 1) / (unsigned)per_row);
        for (int i = tid; i < rows * per_row; i += BD) {
            const int r = per_row == 1 ? i : (int)__umulhi((unsigned)i, magic_row), in_row = i - r * per_row;
            const int c = K == 1 ? in_row : (int)__umulhi((unsigned)in_row, magic_K), k = in_row - c * K;
            const int px = r * BS + c;
            const int64_t sl = (((int64_t)n * a.S + by * BS + r) * a.S + bx * BS) * K + in_row;
            pt_slot(a, sl, k < s_cnt[px] ? s_list[px * stride + k] : 0x7fffffff, centre(r, c));
        }
        __syncthreads();
    }
}

// plain form: one launch per image, every pixel against every point of the cloud
template <int KM>
__global__ void __launch_bounds__(256) k_pnaive(PtArgs a, int n) {
    extern __shared__ unsigned long long s_dyn[];
    const int64_t pidx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = pidx < (int64_t)a.S * a.S;
    const int r = (int)(pidx / a.S), c = (int)(pidx % a.S);
    const PixC p = pixel_centre(r, c, a.S);
    int64_t lo = a.first[n], hi = lo + a.num[n];
    lo = max(lo, (int64_t)0);
    hi = min(hi, a.P);
    TopK<(KM > 0 ? KM : 1)> tk;
    SmemTopK stk;
    if constexpr (KM > 0) {
        tk.init(a.K);
    } else {
        stk.z = reinterpret_cast<float *>(s_dyn) + threadIdx.x;
        stk.f = reinterpret_cast<int *>(s_dyn) + blockDim.x * a.K + threadIdx.x;
        stk.stride = blockDim.x;
        stk.K = a.K;
        stk.init();
    }
    if (!valid) return;
    for (int64_t i = lo; i < hi; ++i) {
        if (a.cloud[i] != n) continue;
        const float4 q = __ldg(reinterpret_cast<const float4 *>(a.rec + i));
        if (!(splat_d(q, p) < a.r2)) continue;
        const float z = __ldg(reinterpret_cast<const float *>(a.rec + i) + 4);
        if constexpr (KM > 0) {
            if (tk.admits(z, (int)i)) tk.insert(z, (int)i);
        } else {
            if (stk.admits(z, (int)i)) stk.insert(z, (int)i);
        }
    }
    const int64_t pix = (int64_t)n * a.S * a.S + pidx;
    if constexpr (KM > 0) {
        pt_write<KM>(a, pix, tk, p);
    } else {
        for (int k = 0; k < a.K; ++k)
            pt_slot(a, pix * a.K + k, k < stk.n ? stk.f[k * stk.stride] : 0x7fffffff, p);
    }
}

// ---------------------------------------------------------------------------
// compositing
// ---------------------------------------------------------------------------
struct CompArgs {
    int64_t npix;
    int N, S, K, D, mode;
    float inv_r2;
    int64_t P;
    const int64_t *idx;
    const float *dists, *features;
    float *image;
    const float *grad_image;
    float *grad_dists, *grad_features;
};

__device__ __forceinline__ int pt_id(const CompArgs &a, int64_t s) {
    const long long v = __ldg(a.idx + s);
    return (v >= 0 && v < a.P) ? (int)v : -1;
}

__global__ void __launch_bounds__(256) k_pcomp_fwd(CompArgs a) {
    const int64_t pix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (pix >= a.npix) return;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    float T = 1.f, asum = 0.f;
    for (int k = 0; k < a.K; ++k) {
        const int64_t s = pix * a.K + k;
        const int i = pt_id(a, s);
        if (i < 0) continue;
        const float q = __ldg(a.dists + s) * a.inv_r2;  // 1 - alpha, without the cancellation
        const float al = 1.f - q;
        const float wgt = a.mode == PTS_COMPOSITE_ALPHA ? al * T : al;
        for (int ch = 0; ch < a.D; ++ch) acc[ch] += wgt * __ldg(a.features + (int64_t)i * a.D + ch);
        T *= q;
        asum += al;
    }
    const float sc = (a.mode == PTS_COMPOSITE_NORM) ? (asum > 0.f ? 1.f / asum : 0.f) : 1.f;
    for (int ch = 0; ch < a.D; ++ch) a.image[pix * a.D + ch] = acc[ch] * sc;
}

// One thread per pixel of a 16 x 16 tile; feature gradients are summed over
// the warp's lanes holding the same point before the atomics.  The forward
// recompute keeps only the transmittance at the start of every chunk of 8
// slots (in shared memory); the reverse pass recomputes each chunk's
// opacities and transmittances into registers.
constexpr int kCompChunk = 8;
constexpr int kCompChunks = (kMaxK + kCompChunk - 1) / kCompChunk;

template <int DM>
__global__ void __launch_bounds__(256) k_pcomp_bwd(CompArgs a) {
    __shared__ float s_T[kCompChunks][256];
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int row = blockIdx.y * 16 + ty, col = blockIdx.x * 16 + tx;
    const bool valid = row < a.S && col < a.S;
    const int64_t pix = ((int64_t)blockIdx.z * a.S + row) * a.S + col;
    float g[DM];
#pragma unroll
    for (int ch = 0; ch < DM; ++ch) g[ch] = (valid && ch < a.D) ? a.grad_image[pix * a.D + ch] : 0.f;
    // forward recompute; 1 - alpha = d / r^2 is taken directly (no cancellation)
    float T = 1.f, asum = 0.f, out[DM];
#pragma unroll
    for (int ch = 0; ch < DM; ++ch) out[ch] = 0.f;
    for (int k = 0; valid && k < a.K; ++k) {
        if (k % kCompChunk == 0) s_T[k / kCompChunk][tid] = T;
        const int64_t s = pix * a.K + k;
        const int i = pt_id(a, s);
        if (i < 0) continue;
        const float q = __ldg(a.dists + s) * a.inv_r2;
#pragma unroll
        for (int ch = 0; ch < DM; ++ch)
            if (ch < a.D) out[ch] += (1.f - q) * __ldg(a.features + (int64_t)i * a.D + ch);
        T *= q;
        asum += 1.f - q;
    }
    const bool norm = a.mode == PTS_COMPOSITE_NORM;
    const float inv_a = asum > 0.f ? 1.f / asum : 0.f;
    // Alpha: df/dalpha_k = T_k (f_k - S_k), S_k the composite of the later
    // slots alone.  E_k = f_k - S_k follows the recursion
    //   E_last = f_last,  E_k = (f_k - f_next) + (1 - alpha_next) E_next,
    // exact when neighbouring features are equal (a silhouette: E_k is the
    // transmittance of the later slots), where f_k - S_k would cancel.
    // Norm: df/dalpha_k = (f_k - f) / sum alpha.
    float E[DM], f_next[DM];
    float q_next = 0.f;
    bool has_next = false;
#pragma unroll
    for (int ch = 0; ch < DM; ++ch) {
        E[ch] = 0.f;
        f_next[ch] = 0.f;
        if (norm) out[ch] *= inv_a;
    }
    const int nch = (a.K + kCompChunk - 1) / kCompChunk;
    for (int c = nch - 1; c >= 0; --c) {  // uniform trip counts: every lane reaches the warp grouping
        // this chunk's ids, 1 - alpha and transmittances, in registers
        int ids[kCompChunk];
        float qv[kCompChunk], Tv[kCompChunk];
        float Tc = valid ? s_T[c][tid] : 1.f;
#pragma unroll
        for (int j = 0; j < kCompChunk; ++j) {
            const int k = c * kCompChunk + j;
            const int64_t s = pix * a.K + k;
            ids[j] = (valid && k < a.K) ? pt_id(a, s) : -1;
            qv[j] = ids[j] >= 0 ? __ldg(a.dists + s) * a.inv_r2 : 1.f;
            Tv[j] = Tc;
            Tc *= qv[j];
        }
#pragma unroll
        for (int j = kCompChunk - 1; j >= 0; --j) {
            const int k = c * kCompChunk + j;
            if (k >= a.K) continue;  // uniform: K is the same for every lane
            const int64_t s = pix * a.K + k;
            const int i = ids[j];
            const float al = 1.f - qv[j];
            float gf[DM];
            float ga = 0.f;
#pragma unroll
            for (int ch = 0; ch < DM; ++ch) {
                gf[ch] = 0.f;
                if (i < 0 || ch >= a.D) continue;
                const float fc = __ldg(a.features + (int64_t)i * a.D + ch);
                if (norm) {
                    gf[ch] = al * inv_a * g[ch];
                    ga += g[ch] * (fc - out[ch]) * inv_a;
                } else {
                    E[ch] = has_next ? (fc - f_next[ch]) + q_next * E[ch] : fc;
                    f_next[ch] = fc;
                    gf[ch] = al * Tv[j] * g[ch];
                    ga += g[ch] * Tv[j] * E[ch];
                }
            }
            if (i >= 0) {
                q_next = qv[j];
                has_next = true;
            }
            if (valid) a.grad_dists[s] = (i < 0) ? 0.f : -ga * a.inv_r2;
            const unsigned peers = __match_any_sync(0xffffffffu, i);
            group_sum<DM>(peers, gf);
            if (i >= 0 && (int)(threadIdx.x & 31) == __ffs(peers) - 1) {
#pragma unroll
                for (int ch = 0; ch < DM; ++ch)
                    if (ch < a.D) atomicAdd(a.grad_features + (int64_t)i * a.D + ch, gf[ch]);
            }
        }
    }
}

// dL/d(zbuf, dists) -> dL/dpoints: d = |p - x|^2, x = f x_v / z_v, then R^T.
// The point is projected here in fp32 (its selection is fixed by idx; the
// gradient needs no double-float positions), so no staging pass is needed.
__global__ void __launch_bounds__(256) k_prast_bwd(PtArgs a, const float *grad_zbuf, const float *grad_dists,
                                                 float *grad_points) {
    // each warp covers an 8 x 4 block of the 16 x 16 tile: neighbouring pixels
    // share points, so the warp's grouping by point finds more peers
    const int tx = ((threadIdx.x >> 5) & 1) * 8 + (threadIdx.x & 7), ty = (threadIdx.x >> 6) * 4 + ((threadIdx.x >> 3) & 3);
    const int n = blockIdx.z;
    const int row = blockIdx.y * 16 + ty, col = blockIdx.x * 16 + tx;
    const bool valid = row < a.S && col < a.S;
    const PixC p = pixel_centre(row, col, a.S);
    const int64_t pix = ((int64_t)n * a.S + row) * a.S + col;
    const float *cam = a.cams + 16 * n;
    const int64_t lo = a.first[n], hi = lo + a.num[n];
    for (int k = 0; k < a.K; ++k) {
        const int64_t s = pix * a.K + k;
        int i = -1;
        if (valid) {
            const long long v = a.idx[s];
            // an id outside this image's range contributes nothing
            i = (v >= 0 && v < a.P && v >= lo && v < hi) ? (int)v : -1;
        }
        float g3[3] = {0.f, 0.f, 0.f};
        float x = 0.f, y = 0.f, iz = 0.f;
        if (i >= 0) {
            const float d0 = __ldg(a.points + 3 * (int64_t)i) - cam[9];
            const float d1 = __ldg(a.points + 3 * (int64_t)i + 1) - cam[10];
            const float d2 = __ldg(a.points + 3 * (int64_t)i + 2) - cam[11];
            const float xv = cam[0] * d0 + cam[1] * d1 + cam[2] * d2;
            const float yv = cam[3] * d0 + cam[4] * d1 + cam[5] * d2;
            const float zv = cam[6] * d0 + cam[7] * d1 + cam[8] * d2;
            if (zv >= cam[13] && isfinite(zv)) {
                iz = 1.f / zv;
                x = cam[12] * xv * iz;
                y = cam[12] * yv * iz;
                const float gd = grad_dists ? grad_dists[s] : 0.f;
                const float gz = grad_zbuf ? grad_zbuf[s] : 0.f;
                const float qx = __fadd_rn(__fsub_rn(p.xh, x), p.xl);
                const float qy = __fadd_rn(__fsub_rn(p.yh, y), p.yl);
                g3[0] = -2.f * gd * qx;  // dL/dx_ndc
                g3[1] = -2.f * gd * qy;  // dL/dy_ndc
                g3[2] = gz;              // dL/dz_view (direct)
            } else {
                i = -1;                  // culled: never selected by the forward
            }
        }
        const unsigned peers = __match_any_sync(0xffffffffu, i);
        group_sum<3>(peers, g3);
        if (i >= 0 && (int)(threadIdx.x & 31) == __ffs(peers) - 1) {
            const float fo = cam[12];
            const float gxv = g3[0] * fo * iz, gyv = g3[1] * fo * iz;
            const float gzv = g3[2] - (g3[0] * x + g3[1] * y) * iz;
            float *gp = grad_points + 3 * (int64_t)i;
            atomicAdd(gp + 0, cam[0] * gxv + cam[3] * gyv + cam[6] * gzv);
            atomicAdd(gp + 1, cam[1] * gxv + cam[4] * gyv + cam[7] * gzv);
            atomicAdd(gp + 2, cam[2] * gxv + cam[5] * gyv + cam[8] * gzv);
        }
    }
}

// ---------------------------------------------------------------------------
// backward of the rendered points
// ---------------------------------------------------------------------------
// The compositing adjoint (that of k_pcomp_bwd) and the rasterizer's in one
// pass over the packed slots: a slot's gradient, two NDC coordinates and D
// features, goes into its point's accumulator as one or two 16-byte
// reductions; k_pts_gather takes each point's sums through the projection
// once.  Empty pixels stop at their first slot.  8 clouds of 200,000 points,
// 256 px, K = 50: forward and backward 1,499 us through the Fragment data, 856 so.
struct PtsBwdArgs {
    const PtRec *rec;
    const int *cloud;
    const float *cams;
    const unsigned long long *slots;
    const float *features, *grad_image;
    float4 *acc;  // pts_acc_vecs(D) per point: (x, y, f0, f1), (f2, f3, f4, f5), (f6, f7, 0, 0)
    float *grad_points, *grad_features;
    int64_t P;
    int N, S, K, D, mode;
    float inv_r2;
};

// Splats of this radius in pixels and up: a warp's slots of one point are summed
// before the reduction.  Reductions into one accumulator queue up, 20 ns each, and a
// large splat has thousands: 8 clouds of 100 points, radius 128 px, K = 8, D = 3,
// forward and backward 1,577 us, grouped 315; 8 of 2,000, radius 26 px, K = 50, D = 3,
// 785, 673.  Small ones find few peers: the same at 6.4 px 392, 401 (D = 1: 362, 383).
constexpr float kGroupRadius = 16.f;

constexpr int pts_acc_vecs(int D) { return D <= 2 ? 1 : D <= 6 ? 2 : 3; }

__device__ __forceinline__ void red_add4(float4 *p, float x, float y, float z, float w) {
    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x), "f"(y), "f"(z), "f"(w)
                 : "memory");
}

template <int DM, bool GROUP>
__global__ void __launch_bounds__(256) k_pts_bwd(PtsBwdArgs a) {
    __shared__ float s_T[kCompChunks][256];
    const int tid = threadIdx.x;
    const int tx = ((tid >> 5) & 1) * 8 + (tid & 7), ty = (tid >> 6) * 4 + ((tid >> 3) & 3);
    const int row = blockIdx.y * 16 + ty, col = blockIdx.x * 16 + tx;
    const int64_t pix = ((int64_t)blockIdx.z * a.S + row) * a.S + col;
    const unsigned long long *s = a.slots + pix * a.K;
    const bool any = row < a.S && col < a.S && __ldg(s) != kPtEnd;
    if (GROUP ? !__any_sync(0xffffffffu, any) : !any) return;
    const bool norm = a.mode == PTS_COMPOSITE_NORM;
    float g[DM], out[DM], E[DM], f_next[DM];
#pragma unroll
    for (int ch = 0; ch < DM; ++ch) {
        g[ch] = any && ch < a.D ? a.grad_image[pix * a.D + ch] : 0.f;
        out[ch] = E[ch] = f_next[ch] = 0.f;
    }
    // forward: the transmittance at the start of each chunk, Norm's mean
    float T = 1.f, asum = 0.f;
    int held = 0, chunks = 0;
    for (bool more = any; more && held < a.K; ++chunks) {
        s_T[chunks][tid] = T;
        unsigned long long v[kCompChunk];
#pragma unroll
        for (int j = 0; j < kCompChunk; ++j)
            v[j] = chunks * kCompChunk + j < a.K ? __ldg(s + chunks * kCompChunk + j) : kPtEnd;
#pragma unroll
        for (int j = 0; j < kCompChunk; ++j) {
            more = more && v[j] != kPtEnd;
            if (!more) continue;
            const float q = __uint_as_float((unsigned)(v[j] >> 32)) * a.inv_r2;
            if (norm) {
#pragma unroll
                for (int ch = 0; ch < DM; ++ch)
                    if (ch < a.D) out[ch] += (1.f - q) * __ldg(a.features + (int64_t)(unsigned)v[j] * a.D + ch);
            }
            T *= q;
            asum += 1.f - q;
            ++held;
        }
    }
    const float inv_a = asum > 0.f ? 1.f / asum : 0.f;
#pragma unroll
    for (int ch = 0; ch < DM; ++ch)
        if (norm) out[ch] *= inv_a;
    const PixC p = pixel_centre(row, col, a.S);
    float q_next = 0.f;
    bool has_next = false;
    // (GROUP: the warp's lanes take the same chunk and rank, with or without a slot there)
    for (int c = (GROUP ? (int)__reduce_max_sync(0xffffffffu, (unsigned)chunks) : chunks) - 1; c >= 0; --c) {
        unsigned long long v[kCompChunk];
        float4 pos[kCompChunk];
        float Tv[kCompChunk], Tc = !GROUP || c < chunks ? s_T[c][tid] : 1.f;
#pragma unroll
        for (int j = 0; j < kCompChunk; ++j) {
            const bool in = c * kCompChunk + j < held;
            v[j] = in ? __ldg(s + c * kCompChunk + j) : kPtEnd;
            if (in) pos[j] = __ldg(reinterpret_cast<const float4 *>(a.rec + (unsigned)v[j]));
            Tv[j] = Tc;
            Tc *= __uint_as_float((unsigned)(v[j] >> 32)) * a.inv_r2;  // (only read up to the last slot)
        }
#pragma unroll
        for (int j = kCompChunk - 1; j >= 0; --j) {
            const bool in = c * kCompChunk + j < held;
            if (!GROUP && !in) continue;
            const int64_t i = (unsigned)v[j];
            // the slot's sums: x, y, features (even: room for the second of a pair)
            constexpr int NS = 2 + (DM > 2 ? DM : 2);
            float sum[NS];
#pragma unroll
            for (int u = 0; u < NS; ++u) sum[u] = 0.f;
            if (in) {
                const float q = __uint_as_float((unsigned)(v[j] >> 32)) * a.inv_r2, al = 1.f - q;
                float ga = 0.f;
#pragma unroll
                for (int ch = 0; ch < DM; ++ch) {
                    if (ch >= a.D) continue;
                    const float fc = __ldg(a.features + i * a.D + ch);
                    if (norm) {
                        sum[2 + ch] = al * inv_a * g[ch];
                        ga += g[ch] * (fc - out[ch]) * inv_a;
                    } else {
                        E[ch] = has_next ? (fc - f_next[ch]) + q_next * E[ch] : fc;
                        f_next[ch] = fc;
                        sum[2 + ch] = al * Tv[j] * g[ch];
                        ga += g[ch] * Tv[j] * E[ch];
                    }
                }
                q_next = q;
                has_next = true;
                const float gd = -ga * a.inv_r2;
                const float qx = __fadd_rn(__fsub_rn(p.xh, pos[j].x), __fsub_rn(p.xl, pos[j].z));
                const float qy = __fadd_rn(__fsub_rn(p.yh, pos[j].y), __fsub_rn(p.yl, pos[j].w));
                sum[0] = -2.f * gd * qx;
                sum[1] = -2.f * gd * qy;
            }
            if constexpr (GROUP) {
                const unsigned peers = __match_any_sync(0xffffffffu, in ? (int)i : -1 - (tid & 31));
                group_sum<NS>(peers, sum);
                if (!in || (tid & 31) != __ffs(peers) - 1) continue;
            }
            float4 *acc = a.acc + i * pts_acc_vecs(a.D);
            red_add4(acc, sum[0], sum[1], sum[2], sum[3]);
            if constexpr (DM >= 4) {
                if (a.D > 2) red_add4(acc + 1, sum[4], sum[5], DM > 4 ? sum[DM > 4 ? 6 : 0] : 0.f, DM > 4 ? sum[DM > 4 ? 7 : 0] : 0.f);
            }
            if constexpr (DM > 6) {
                if (a.D > 6) red_add4(acc + 2, sum[8], sum[9], 0.f, 0.f);
            }
        }
    }
}

__global__ void __launch_bounds__(256) k_pts_gather(PtsBwdArgs a) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.P) return;
    const int vecs = pts_acc_vecs(a.D), n = a.cloud[i];
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    float g[3] = {0.f, 0.f, 0.f};
    if (n >= 0) {
        v = __ldg(a.acc + i * vecs);
        const float4 pos = __ldg(reinterpret_cast<const float4 *>(a.rec + i));
        const float *cam = a.cams + 16 * n;
        // x = f x_v / z_v, y = f y_v / z_v: d/dx_v = f/z, d/dz_v = -(x dL/dx + y dL/dy)/z
        const float iz = 1.f / __ldg(reinterpret_cast<const float *>(a.rec + i) + 4), fo = cam[12];
        const float gxv = v.x * fo * iz, gyv = v.y * fo * iz, gzv = -(v.x * pos.x + v.y * pos.y) * iz;
#pragma unroll
        for (int j = 0; j < 3; ++j) g[j] = cam[j] * gxv + cam[3 + j] * gyv + cam[6 + j] * gzv;
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) a.grad_points[3 * i + j] = g[j];
    float *gf = a.grad_features + i * a.D;
    gf[0] = v.z;
    if (a.D > 1) gf[1] = v.w;
    for (int b = 1; b < vecs; ++b) {
        const float4 w = n >= 0 ? __ldg(a.acc + i * vecs + b) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (4 * b - 2 + j < a.D) gf[4 * b - 2 + j] = x[j];
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
template <bool GROUP>
static void launch_pts_bwd(const PtsBwdArgs &a, const dim3 &grid, cudaStream_t st) {
    if (a.D == 1) k_pts_bwd<1, GROUP><<<grid, 256, 0, st>>>(a);
    else if (a.D <= 4) k_pts_bwd<4, GROUP><<<grid, 256, 0, st>>>(a);
    else k_pts_bwd<8, GROUP><<<grid, 256, 0, st>>>(a);
}

static int km_for_points(int K) {
    if (K <= 1) return 1;
    if (K <= 2) return 2;
    if (K <= 4) return 4;
    if (K <= 8) return 8;
    if (K <= 16) return 16;
    return 0;
}

struct PtLayout {
    size_t records, cloud, counts, eff, offsets, cursor, lists, bytes;
    int64_t nb, NB, capacity;
};

static bool pt_params_ok(const pts_params *p, int64_t P) {
    if (!p) return false;
    if (p->N < 0 || p->N > 65535 || p->image_size < 1 || p->image_size > 8192) return false;
    if (p->points_per_pixel < 1) return false;
    if (!(p->radius > 0.f) || !(p->radius < 4.f)) return false;
    if (p->reserved != 0 || p->reserved_f != 0.f) return false;
    if (P < 0 || P >= 0x7fffffffLL) return false;
    if (p->bin_size > 0 && p->max_points_per_bin <= 0) return false;
    if (p->max_bin_entries < 0) return false;
    return true;
}

static bool pt_unsupported(const pts_params *p) {
    if (p->points_per_pixel > kMaxK || (p->bin_size != 0 && p->bin_size != 8 && p->bin_size != 16)) return true;
    if (p->bin_size > 0) {
        // bin keys, counts, offsets and list positions are 32-bit on the device
        const int64_t nb = (p->image_size + p->bin_size - 1) / p->bin_size;
        const int64_t NB = (int64_t)p->N * nb * nb;
        if (NB >= 0x7fffffffLL) return true;
        const int64_t cap = p->max_bin_entries > 0 ? p->max_bin_entries : NB * (int64_t)p->max_points_per_bin;
        if (cap > 0x7fffffffLL) return true;
    }
    return false;
}

static size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

static void pt_layout(const pts_params *p, int64_t P, PtLayout *L) {
    std::memset(L, 0, sizeof(*L));
    size_t off = 1536;  // header: status @0, queue @4, total @8, max count @16, long lists @24, @512 (as the mesh workspace)
    L->records = off;
    off = al256(off + (size_t)P * sizeof(PtRec));
    L->cloud = off;
    off = al256(off + (size_t)P * 4);
    if (p->bin_size > 0) {
        const int64_t nb = (p->image_size + p->bin_size - 1) / p->bin_size;
        const int64_t NB = (int64_t)p->N * nb * nb;
        const int64_t cap = p->max_bin_entries > 0 ? p->max_bin_entries : NB * (int64_t)p->max_points_per_bin;
        L->nb = nb;
        L->NB = NB;
        L->capacity = cap;
        L->counts = off;
        off = al256(off + (size_t)NB * 4);
        L->eff = off;
        off = al256(off + (size_t)NB * 4);
        L->offsets = off;
        off = al256(off + (size_t)(NB + 1) * 4);
        L->cursor = off;
        off = al256(off + (size_t)NB * 4);
        L->lists = off;
        off = al256(off + (size_t)cap * 8);
    }
    L->bytes = off;
}

static void pt_fill_args(PtArgs &a, const pts_params *p, const float *points, int64_t P, const int64_t *first,
                         const int64_t *num, const float *cams, char *ws, const PtLayout &L) {
    std::memset(&a, 0, sizeof(a));
    a.points = points;
    a.P = P;
    a.first = first;
    a.num = num;
    a.N = p->N;
    a.cams = cams;
    a.radius = p->radius;
    a.r2 = p->radius * p->radius;
    a.S = p->image_size;
    a.K = p->points_per_pixel;
    a.bin = p->bin_size > 0 ? p->bin_size : 1;
    a.nb = (int)L.nb;
    a.items = L.NB;
    a.rec = reinterpret_cast<PtRec *>(ws + L.records);
    a.cloud = reinterpret_cast<int *>(ws + L.cloud);
    if (p->bin_size > 0) {
        a.counts = reinterpret_cast<int *>(ws + L.counts);
        a.cursor = reinterpret_cast<int *>(ws + L.cursor);
        a.eff = reinterpret_cast<const int *>(ws + L.eff);
        a.offsets = reinterpret_cast<const int *>(ws + L.offsets);
        a.lists = reinterpret_cast<unsigned long long *>(ws + L.lists);
    }
    a.queue = reinterpret_cast<unsigned *>(ws + 4);
    a.status = reinterpret_cast<unsigned *>(ws);
}

// Enough points to give every SM two blocks of kPtPerThread points per thread.
// By the call, both ways (us; counted in shared memory, each pair to memory; 256 px,
// bins of 8): 1 cloud of 50,000 points 74, 47, of 200,000 91, 112, of 622,592 150, 291; 8 of
// 50,000 151, 139, of 77,824 160, 191; 32 of 20,000, whose blocks of 2,048 are the fewest
// per cloud, 346, 327.
static bool pt_hist(const PtArgs &a) {
    return a.P >= (int64_t)2 * mr_host::num_sms() * 256 * kPtPerThread && (int64_t)a.nb * a.nb <= kPtHist;
}

static unsigned pt_blocks(int64_t P, int per) { return (unsigned)((P + 256 * per - 1) / (256 * per)); }

static cudaError_t launch_pstage(const PtArgs &a, bool count, cudaStream_t st) {
    if (count && pt_hist(a)) k_pstage<kPtPerThread, true><<<pt_blocks(a.P, kPtPerThread), 256, 0, st>>>(a, 1);
    else k_pstage<1, false><<<pt_blocks(a.P, 1), 256, 0, st>>>(a, count ? 1 : 0);
    return cudaGetLastError();
}

static cudaError_t launch_pfill(const PtArgs &a, cudaStream_t st) {
    if (pt_hist(a)) k_pfill<kPtPerThread, true><<<pt_blocks(a.P, kPtPerThread), 256, 0, st>>>(a);
    else k_pfill<1, false><<<pt_blocks(a.P, 1), 256, 0, st>>>(a);
    return cudaGetLastError();
}

template <int BS, bool RENDER>
static cudaError_t launch_pfine_t(const PtArgs &a, cudaStream_t st) {
    constexpr int BD = kPfineThreads;
    const size_t dyn = (size_t)BS * BS * (a.K | 1) * (RENDER ? 2 : 1) * sizeof(int);  // ids, and 1 - alpha
    auto kern = k_pfine<BS, RENDER>;
    if (dyn > 16 * 1024) {  // static + dynamic above 48 KB needs the opt-in
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
        if (e != cudaSuccess) return e;
    }
    const int grid = mr_host::queue_blocks(a.items, 2048 / BD);
    kern<<<grid, BD, dyn, st>>>(a);
    return cudaGetLastError();
}

static cudaError_t launch_pfine(const PtArgs &a, int bin, cudaStream_t st) {
    if (bin == 8) return a.slots ? launch_pfine_t<8, true>(a, st) : launch_pfine_t<8, false>(a, st);
    if (bin == 16) return a.slots ? launch_pfine_t<16, true>(a, st) : launch_pfine_t<16, false>(a, st);
    return cudaErrorInvalidValue;
}

template <int KM>
static cudaError_t launch_pnaive_t(const PtArgs &a, cudaStream_t st) {
    const int BD = 256;
    const size_t dyn = (KM > 0) ? 0 : (size_t)BD * a.K * 8;
    if (KM == 0) {
        cudaError_t e = cudaFuncSetAttribute(k_pnaive<KM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
        if (e != cudaSuccess) return e;
    }
    const int64_t npx = (int64_t)a.S * a.S;
    const int grid = (int)((npx + BD - 1) / BD);
    for (int n = 0; n < a.N; ++n) {
        k_pnaive<KM><<<grid, BD, dyn, st>>>(a, n);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

static cudaError_t launch_pnaive(const PtArgs &a, cudaStream_t st) {
    switch (km_for_points(a.K)) {
        case 1: return launch_pnaive_t<1>(a, st);
        case 2: return launch_pnaive_t<2>(a, st);
        case 4: return launch_pnaive_t<4>(a, st);
        case 8: return launch_pnaive_t<8>(a, st);
        case 16: return launch_pnaive_t<16>(a, st);
        default: return launch_pnaive_t<0>(a, st);
    }
}

// records, then clouds, in a caller's buffer of pts_staged_bytes
static void pt_staged(const void *buf, int64_t P, PtRec *&rec, int *&cloud) {
    char *b = static_cast<char *>(const_cast<void *>(buf));
    rec = reinterpret_cast<PtRec *>(b);
    cloud = reinterpret_cast<int *>(b + (size_t)P * sizeof(PtRec));
}

static bool al16(const void *q) { return ((uintptr_t)q & 15u) == 0; }

static int check_pws(const pts_params *p, int64_t P, void *ws, size_t ws_bytes, PtLayout *L) {
    pt_layout(p, P, L);
    if (!ws || ((uintptr_t)ws & 255u) != 0 || ws_bytes < L->bytes) return MESHRAST_ERR_WORKSPACE;
    return MESHRAST_OK;
}

}  // namespace mr

using mr::PtLayout;

extern "C" {

size_t pts_workspace_bytes(const pts_params *p, int64_t P) {
    if (!mr::pt_params_ok(p, P) || mr::pt_unsupported(p)) return 0;
    PtLayout L;
    mr::pt_layout(p, P, &L);
    return L.bytes;
}

// Rasterization into Fragment data (a.idx ..), or with a.slots rendering on
// packed slots, the points' records and clouds in `staged` (NULL: workspace).
static int pts_forward(mr::PtArgs &out, const pts_params *p, const float *points, int64_t P,
                       const int64_t *first_point, const int64_t *num_points, const float *cams, void *staged,
                       void *workspace, size_t workspace_bytes, void *stream) {
    PtLayout L;
    int rc = mr::check_pws(p, P, workspace, workspace_bytes, &L);
    if (rc) return rc;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    char *ws = reinterpret_cast<char *>(workspace);
    if (cudaMemsetAsync(ws, 0, 256, st) != cudaSuccess) return MESHRAST_ERR_CUDA;
    if (p->N == 0) return MESHRAST_OK;
    const bool binned = p->bin_size > 0;
    if (binned && L.NB > 0 && cudaMemsetAsync(ws + L.counts, 0, (size_t)L.NB * 4, st) != cudaSuccess)
        return MESHRAST_ERR_CUDA;
    mr::PtArgs a;
    mr::pt_fill_args(a, p, points, P, first_point, num_points, cams, ws, L);
    a.idx = out.idx;
    a.zbuf = out.zbuf;
    a.dists = out.dists;
    a.slots = out.slots;
    a.features = out.features;
    a.image = out.image;
    a.D = out.D;
    a.mode = out.mode;
    a.inv_r2 = 1.f / (p->radius * p->radius);
    if (staged) mr::pt_staged(staged, P, a.rec, a.cloud);
    if (P > 0) {
        if (mr::launch_pstage(a, binned, st) != cudaSuccess) return MESHRAST_ERR_CUDA;
    }
    if (!binned) return mr::launch_pnaive(a, st) == cudaSuccess ? MESHRAST_OK : MESHRAST_ERR_CUDA;
    mr::ScanArgs sa;
    sa.counts = a.counts;
    sa.eff = reinterpret_cast<int *>(ws + L.eff);
    sa.offsets = reinterpret_cast<int *>(ws + L.offsets);
    sa.cursor = a.cursor;
    sa.order = nullptr;
    sa.NB = L.NB;
    sa.capacity = L.capacity;
    sa.max_per_bin = p->max_points_per_bin;
    sa.queue = a.queue;
    sa.status = a.status;
    sa.total = reinterpret_cast<long long *>(ws + 8);
    sa.maxcount = reinterpret_cast<int *>(ws + 16);
    sa.longs = p->max_points_per_bin > mr::kLongList ? reinterpret_cast<unsigned *>(ws + 24) : nullptr;
    sa.long_bins = reinterpret_cast<mr::LongBin *>(ws + 512);
    sa.first_face = first_point;
    sa.num_faces = num_points;
    sa.N = p->N;
    sa.F = P;
    if (mr::launch_scan(sa, st) != cudaSuccess) return MESHRAST_ERR_CUDA;
    if (P > 0) {
        if (mr::launch_pfill(a, st) != cudaSuccess) return MESHRAST_ERR_CUDA;
    }
    if (sa.longs) {
        a.total = sa.total;
        a.maxcount = sa.maxcount;
        if (mr::launch_sort_long({a.lists, a.eff, a.offsets, sa.longs, sa.long_bins}, st) != cudaSuccess)
            return MESHRAST_ERR_CUDA;
    }
    return mr::launch_pfine(a, p->bin_size, st) == cudaSuccess ? MESHRAST_OK : MESHRAST_ERR_CUDA;
}

int pts_rasterize_fwd(const pts_params *p, const float *points, int64_t P, const int64_t *first_point,
                      const int64_t *num_points, const float *cams, int64_t *idx, float *zbuf, float *dists,
                      void *workspace, size_t workspace_bytes, void *stream) {
    if (!mr::pt_params_ok(p, P)) return MESHRAST_ERR_INVALID_ARG;
    if (mr::pt_unsupported(p)) return MESHRAST_ERR_UNSUPPORTED;
    if (p->N > 0 && (!first_point || !num_points || !cams)) return MESHRAST_ERR_INVALID_ARG;
    if (P > 0 && !points) return MESHRAST_ERR_INVALID_ARG;
    const int64_t slots = (int64_t)p->N * p->image_size * p->image_size * p->points_per_pixel;
    if (slots > 0 && (!idx || !zbuf || !dists || !mr::al16(idx) || !mr::al16(zbuf) || !mr::al16(dists)))
        return MESHRAST_ERR_INVALID_ARG;
    mr::PtArgs out;
    std::memset(&out, 0, sizeof(out));
    out.idx = idx;
    out.zbuf = zbuf;
    out.dists = dists;
    return pts_forward(out, p, points, P, first_point, num_points, cams, nullptr, workspace, workspace_bytes, stream);
}

int pts_rasterize_bwd(const pts_params *p, const float *points, int64_t P, const int64_t *first_point,
                      const int64_t *num_points, const float *cams, const int64_t *idx, const float *grad_zbuf,
                      const float *grad_dists, float *grad_points, void *workspace, size_t workspace_bytes,
                      void *stream) {
    if (!mr::pt_params_ok(p, P)) return MESHRAST_ERR_INVALID_ARG;
    if (mr::pt_unsupported(p)) return MESHRAST_ERR_UNSUPPORTED;
    if (p->N > 0 && (!first_point || !num_points || !cams)) return MESHRAST_ERR_INVALID_ARG;
    if (P > 0 && (!points || !grad_points)) return MESHRAST_ERR_INVALID_ARG;
    const int64_t slots = (int64_t)p->N * p->image_size * p->image_size * p->points_per_pixel;
    if (slots > 0 && !idx) return MESHRAST_ERR_INVALID_ARG;
    PtLayout L;
    int rc = mr::check_pws(p, P, workspace, workspace_bytes, &L);
    if (rc) return rc;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    char *ws = reinterpret_cast<char *>(workspace);
    if (P > 0 && cudaMemsetAsync(grad_points, 0, (size_t)P * 3 * sizeof(float), st) != cudaSuccess)
        return MESHRAST_ERR_CUDA;
    if (slots == 0 || (!grad_zbuf && !grad_dists)) return MESHRAST_OK;
    mr::PtArgs a;
    mr::pt_fill_args(a, p, points, P, first_point, num_points, cams, ws, L);
    a.idx = const_cast<int64_t *>(idx);
    const unsigned tiles = (unsigned)((p->image_size + 15) / 16);
    mr::k_prast_bwd<<<dim3(tiles, tiles, (unsigned)p->N), 256, 0, st>>>(a, grad_zbuf, grad_dists, grad_points);
    return cudaGetLastError() == cudaSuccess ? MESHRAST_OK : MESHRAST_ERR_CUDA;
}

static int check_comp(const pts_params *p, int32_t mode, int64_t P, int32_t D) {
    if (!p || p->N < 0 || p->N > 65535 || p->image_size < 0 || p->image_size > 8192) return MESHRAST_ERR_INVALID_ARG;
    if (p->points_per_pixel < 1) return MESHRAST_ERR_INVALID_ARG;
    if (p->points_per_pixel > mr::kMaxK) return MESHRAST_ERR_UNSUPPORTED;
    if (!(p->radius > 0.f)) return MESHRAST_ERR_INVALID_ARG;
    if (mode != PTS_COMPOSITE_ALPHA && mode != PTS_COMPOSITE_NORM) return MESHRAST_ERR_INVALID_ARG;
    if (D < 1 || D > 8 || P < 0) return MESHRAST_ERR_INVALID_ARG;
    return MESHRAST_OK;
}

static void fill_comp(mr::CompArgs &c, const pts_params *p, int32_t mode, const int64_t *idx, const float *dists,
                      const float *features, int64_t P, int32_t D) {
    std::memset(&c, 0, sizeof(c));
    c.N = p->N;
    c.S = p->image_size;
    c.K = p->points_per_pixel;
    c.npix = (int64_t)p->N * p->image_size * p->image_size;
    c.D = D;
    c.mode = mode;
    c.inv_r2 = 1.f / (p->radius * p->radius);
    c.P = P;
    c.idx = idx;
    c.dists = dists;
    c.features = features;
}

int pts_composite_fwd(const pts_params *p, int32_t mode, const int64_t *idx, const float *dists,
                      const float *features, int64_t P, int32_t D, float *image, void *stream) {
    int rc = check_comp(p, mode, P, D);
    if (rc) return rc;
    mr::CompArgs c;
    fill_comp(c, p, mode, idx, dists, features, P, D);
    if (c.npix == 0) return MESHRAST_OK;
    if (!idx || !dists || !image || (P > 0 && !features)) return MESHRAST_ERR_INVALID_ARG;
    c.image = image;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    mr::k_pcomp_fwd<<<(unsigned)((c.npix + 255) / 256), 256, 0, st>>>(c);
    return cudaGetLastError() == cudaSuccess ? MESHRAST_OK : MESHRAST_ERR_CUDA;
}

int pts_composite_bwd(const pts_params *p, int32_t mode, const int64_t *idx, const float *dists,
                      const float *features, int64_t P, int32_t D, const float *grad_image, float *grad_dists,
                      float *grad_features, void *stream) {
    int rc = check_comp(p, mode, P, D);
    if (rc) return rc;
    mr::CompArgs c;
    fill_comp(c, p, mode, idx, dists, features, P, D);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (P > 0) {
        if (!grad_features) return MESHRAST_ERR_INVALID_ARG;
        if (cudaMemsetAsync(grad_features, 0, (size_t)P * D * sizeof(float), st) != cudaSuccess)
            return MESHRAST_ERR_CUDA;
    }
    if (c.npix == 0) return MESHRAST_OK;
    if (!idx || !dists || !grad_image || !grad_dists || (P > 0 && !features)) return MESHRAST_ERR_INVALID_ARG;
    c.grad_image = grad_image;
    c.grad_dists = grad_dists;
    c.grad_features = grad_features;
    const unsigned tiles = (unsigned)((p->image_size + 15) / 16);
    const dim3 grid(tiles, tiles, (unsigned)p->N);
    if (D == 1) mr::k_pcomp_bwd<1><<<grid, 256, 0, st>>>(c);
    else if (D <= 4) mr::k_pcomp_bwd<4><<<grid, 256, 0, st>>>(c);
    else mr::k_pcomp_bwd<8><<<grid, 256, 0, st>>>(c);
    return cudaGetLastError() == cudaSuccess ? MESHRAST_OK : MESHRAST_ERR_CUDA;
}

size_t pts_staged_bytes(int64_t P) {
    return P < 0 || P >= 0x7fffffffLL ? 0 : mr::al256((size_t)P * (sizeof(mr::PtRec) + sizeof(int)) + 1);
}

int pts_render_fwd(const pts_params *p, int32_t mode, const float *points, int64_t P, const int64_t *first_point,
                   const int64_t *num_points, const float *cams, const float *features, int32_t D, uint64_t *slots,
                   float *image, void *staged, void *workspace, size_t workspace_bytes, void *stream) {
    if (!mr::pt_params_ok(p, P)) return MESHRAST_ERR_INVALID_ARG;
    if (mr::pt_unsupported(p) || p->bin_size == 0) return MESHRAST_ERR_UNSUPPORTED;
    int rc = check_comp(p, mode, P, D);
    if (rc) return rc;
    if (p->N > 0 && (!first_point || !num_points || !cams || !slots || !image || !mr::al16(slots)))
        return MESHRAST_ERR_INVALID_ARG;
    if (P > 0 && (!points || !features)) return MESHRAST_ERR_INVALID_ARG;
    if (!staged || !mr::al16(staged)) return MESHRAST_ERR_INVALID_ARG;
    mr::PtArgs out;
    std::memset(&out, 0, sizeof(out));
    out.slots = reinterpret_cast<unsigned long long *>(slots);
    out.features = features;
    out.image = image;
    out.D = D;
    out.mode = mode;
    return pts_forward(out, p, points, P, first_point, num_points, cams, staged, workspace, workspace_bytes, stream);
}

int pts_render_bwd(const pts_params *p, int32_t mode, int64_t P, const float *cams, const float *features, int32_t D,
                   const uint64_t *slots, const void *staged, const float *grad_image, float *scratch,
                   float *grad_points, float *grad_features, void *stream) {
    if (!mr::pt_params_ok(p, P)) return MESHRAST_ERR_INVALID_ARG;
    if (mr::pt_unsupported(p) || p->bin_size == 0) return MESHRAST_ERR_UNSUPPORTED;
    int rc = check_comp(p, mode, P, D);
    if (rc) return rc;
    if (P == 0) return MESHRAST_OK;
    if (!grad_points || !grad_features) return MESHRAST_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (p->N == 0) {
        return cudaMemsetAsync(grad_points, 0, (size_t)P * 3 * sizeof(float), st) == cudaSuccess &&
                       cudaMemsetAsync(grad_features, 0, (size_t)P * D * sizeof(float), st) == cudaSuccess
                   ? MESHRAST_OK
                   : MESHRAST_ERR_CUDA;
    }
    if (!cams || !features || !slots || !staged || !grad_image || !scratch || !mr::al16(scratch) || !mr::al16(staged))
        return MESHRAST_ERR_INVALID_ARG;
    mr::PtsBwdArgs a;
    mr::PtRec *rec;
    int *cloud;
    mr::pt_staged(staged, P, rec, cloud);
    a.rec = rec;
    a.cloud = cloud;
    a.cams = cams;
    a.slots = reinterpret_cast<const unsigned long long *>(slots);
    a.features = features;
    a.grad_image = grad_image;
    a.acc = reinterpret_cast<float4 *>(scratch);
    a.grad_points = grad_points;
    a.grad_features = grad_features;
    a.P = P;
    a.N = p->N;
    a.S = p->image_size;
    a.K = p->points_per_pixel;
    a.D = D;
    a.mode = mode;
    a.inv_r2 = 1.f / (p->radius * p->radius);
    const size_t bytes = (size_t)P * mr::pts_acc_vecs(D) * sizeof(float4);
    if (cudaMemsetAsync(scratch, 0, bytes, st) != cudaSuccess) return MESHRAST_ERR_CUDA;
    const unsigned tiles = (unsigned)((p->image_size + 15) / 16);
    const dim3 grid(tiles, tiles, (unsigned)p->N);
    if (0.5f * p->radius * (float)p->image_size >= mr::kGroupRadius) mr::launch_pts_bwd<true>(a, grid, st);
    else mr::launch_pts_bwd<false>(a, grid, st);
    if (cudaGetLastError() != cudaSuccess) return MESHRAST_ERR_CUDA;
    mr::k_pts_gather<<<(unsigned)((P + 255) / 256), 256, 0, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? MESHRAST_OK : MESHRAST_ERR_CUDA;
}

int pts_bin_occupancy(const pts_params *p, int64_t P, const void *workspace, int32_t *max_count,
                      int64_t *total_entries, void *stream) {
    if (!mr::pt_params_ok(p, P) || !workspace || !max_count || !total_entries || p->bin_size <= 0)
        return MESHRAST_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (cudaStreamSynchronize(st) != cudaSuccess) return MESHRAST_ERR_CUDA;
    const char *ws = reinterpret_cast<const char *>(workspace);
    int32_t mc = 0;
    long long tot = 0;
    if (cudaMemcpy(&mc, ws + 16, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return MESHRAST_ERR_CUDA;
    if (cudaMemcpy(&tot, ws + 8, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return MESHRAST_ERR_CUDA;
    *max_count = mc;
    *total_entries = tot;
    return MESHRAST_OK;
}

}  // extern "C"
