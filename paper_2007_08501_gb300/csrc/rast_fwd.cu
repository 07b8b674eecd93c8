// Forward rasterization kernels for sm_103a.
//
// Section 3.2 of the paper ("Rasterizer"): camera transform to NDC, a
// two-pass approach that first assigns faces to image tiles (bins) and then
// finds, per pixel, the K nearest faces along z with a priority queue, and the
// Fragment data of those faces.  Launch sequence of one binned forward:
//   k_stage     one thread per face: double-float projection, 96-byte face
//               record, warp-aggregated bin counts
//   k_scan      one block: clamp counts to capacity, exclusive scan -> offsets;
//               finds the long lists
//   k_fill      one thread per face: warp-aggregated atomic append into lists
//   k_sort_long (sort_long.cu) where bins may hold more than kLongList entries:
//               long lists, where few are long
//   k_fine      persistent blocks pull (image, bin) items from a global queue,
//               walk each bin's faces front to back, keep a register-resident
//               top-K per pixel, write the fragments
// The plain form (bin_size 0) replaces scan/fill/fine by k_naive, every pixel
// against every face of its image.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>

#include "rast_common.cuh"
#include "rast_internal.h"
#include "blend_common.cuh"
#include "bin_common.cuh"
#include "sil.cuh"

namespace mr {

// ---------------------------------------------------------------------------
// staging
// ---------------------------------------------------------------------------
// A block's faces share most of their corners (256 faces of a mesh touch some
// 150 vertices, 768 corners): each distinct vertex is projected once, in
// double-float, found through a hash of its index in shared memory.  Bound by
// the loads of faces and vertices and by the barriers between the steps (48 %
// issue-active): 1.3M faces, an image of 1,024 px: 153 -> 133 us.
constexpr int kStageTable = 1024;  // > 3 x 256 corners
struct StageTable {
    int key[kStageTable];          // vertex, -1 free
    float x[6][kStageTable];       // X, Y, Z as hi, lo
    unsigned short list[3 * 256];  // occupied places
    unsigned char bad[kStageTable];
    int n;
};

__device__ __forceinline__ int stage_place(StageTable &t, int v) {
    unsigned h = ((unsigned)v * 2654435761u) >> 22;
    while (true) {
        const int seen = atomicCAS(&t.key[h], -1, v);
        if (seen == -1) t.list[atomicAdd(&t.n, 1)] = (unsigned short)h;
        if (seen == -1 || seen == v) return (int)h;
        h = (h + 1) & (kStageTable - 1);  // (at most 768 of 1,024 are taken)
    }
}

// Build the record of face f; returns the mesh index or -1 when culled.  Every
// thread of the block calls it; `block` is the image whose corners are shared.
__device__ int stage_face(const StageArgs &a, StageTable &t, int64_t f, int n, int block, FaceRec &R) {
    const float kInf = __int_as_float(0x7f800000);
    R.a = make_float4(0.f, 0.f, 0.f, 0.f);
    R.b = make_float4(0.f, 0.f, 0.f, 0.f);
    R.c = make_float4(kInf, -kInf, kInf, -kInf);
    R.d = make_float4(0.f, 1.f, 1.f, 1.f);
    R.e = make_float4(0.f, 0.f, 0.f, 0.f);
    R.h = make_float4(0.f, 0.f, 0.f, 0.f);
    reinterpret_cast<int4 *>(t.key)[threadIdx.x] = make_int4(-1, -1, -1, -1);
    if (threadIdx.x == 0) t.n = 0;
    __syncthreads();
    unsigned bad = 0;
    int64_t vi[3] = {0, 0, 0};
    int at[3] = {0, 0, 0};
    if (n >= 0) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            vi[i] = a.faces[3 * f + i];
            if (vi[i] < 0 || vi[i] >= a.V) bad |= MESHRAST_ST_BAD_INDEX;
        }
        if (!bad && n == block)
            for (int i = 0; i < 3; ++i) at[i] = stage_place(t, (int)vi[i]);
    }
    __syncthreads();
    for (int j = threadIdx.x; j < t.n; j += 256) {
        const int h = t.list[j];
        const float *v = a.verts + 3 * (int64_t)t.key[h];
        const float px = v[0], py = v[1], pz = v[2];
        t.bad[h] = !(isfinite(px) && isfinite(py) && isfinite(pz));
        df X, Y, Z;
        project_corner(a.cams + 16 * block, px, py, pz, X, Y, Z);
        t.x[0][h] = X.hi;
        t.x[1][h] = X.lo;
        t.x[2][h] = Y.hi;
        t.x[3][h] = Y.lo;
        t.x[4][h] = Z.hi;
        t.x[5][h] = Z.lo;
    }
    __syncthreads();
    if (n < 0) return -1;
    if (bad) { set_status(a.status, bad); return -1; }
    const float *cam = a.cams + 16 * n;
    df X[3], Y[3], Z[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        df x, y, z;
        if (n == block) {
            const int h = at[i];
            if (t.bad[h]) bad |= MESHRAST_ST_NONFINITE;
            x = {t.x[0][h], t.x[1][h]};
            y = {t.x[2][h], t.x[3][h]};
            z = {t.x[4][h], t.x[5][h]};
        } else {  // a block across two images
            const float *v = a.verts + 3 * vi[i];
            const float px = v[0], py = v[1], pz = v[2];
            if (!(isfinite(px) && isfinite(py) && isfinite(pz))) bad |= MESHRAST_ST_NONFINITE;
            project_corner(cam, px, py, pz, x, y, z);
        }
        X[i] = x;
        Y[i] = y;
        Z[i] = z;
    }
    if (bad) { set_status(a.status, bad); return -1; }
    const float znear = cam[13];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        // z < znear (as a double-float) culls the face
        if (Z[i].hi < znear || (Z[i].hi == znear && Z[i].lo < 0.f) || !isfinite(Z[i].hi)) return -1;
        if (!isfinite(X[i].hi) || !isfinite(Y[i].hi)) return -1;
    }
    df Ux = df_sub(X[1], X[0]), Uy = df_sub(Y[1], Y[0]);
    df Wx = df_sub(X[2], X[0]), Wy = df_sub(Y[2], Y[0]);
    // area in double-float (matches an FP64 evaluation to ~1e-14): culling and 1/A
    df Adf = df_sub(df_mul(Ux, Wy), df_mul(Uy, Wx));
    if (!(fabsf(Adf.hi) >= kCullArea)) return -1;
    const float A = __fadd_rn(Adf.hi, Adf.lo);
    float ux = Ux.hi, uy = Uy.hi, wx = Wx.hi, wy = Wy.hi;
    float r = (a.blur > 0.f) ? sqrtf(a.blur) : 0.f;
    df xmin = df_min(df_min(X[0], X[1]), X[2]), xmax = df_max(df_max(X[0], X[1]), X[2]);
    df ymin = df_min(df_min(Y[0], Y[1]), Y[2]), ymax = df_max(df_max(Y[0], Y[1]), Y[2]);
    R.a = make_float4(X[0].hi, Y[0].hi, X[0].lo, Y[0].lo);
    R.b = make_float4(ux, uy, wx, wy);
    R.c = make_float4(df_round_down(df_add(xmin, {-r, 0.f})), df_round_up(df_add(xmax, {r, 0.f})),
                      df_round_down(df_add(ymin, {-r, 0.f})), df_round_up(df_add(ymax, {r, 0.f})));
    R.d = make_float4(__fdiv_rn(1.f, A), __fdiv_rn(1.f, Z[0].hi), __fdiv_rn(1.f, Z[1].hi),
                      __fdiv_rn(1.f, Z[2].hi));
    R.e = make_float4(Ux.lo, Uy.lo, Wx.lo, Wy.lo);
    const float A2 = A * A;
    const float l0 = (wx - ux) * (wx - ux) + (wy - uy) * (wy - uy), l1 = wx * wx + wy * wy, l2 = ux * ux + uy * uy;
    R.h = make_float4(A2 / l0, A2 / l1, A2 / l2, 0.f);
    return n;
}

__global__ void __launch_bounds__(256) k_stage(StageArgs a) {
    const int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    __shared__ __align__(16) StageTable s_table;
    FaceRec R;
    int block;
    int64_t lo, hi;
    block_image(a.first_face, a.num_faces, a.N, a.F, (int64_t)blockIdx.x * blockDim.x, block, lo, hi);
    int n = f < a.F ? image_of(a.first_face, a.num_faces, a.N, f, block, lo, hi) : -1;
    n = stage_face(a, s_table, f, n, block, R);
    if (f < a.F) {
        float4 *dst = reinterpret_cast<float4 *>(a.rec + f);
        dst[kRecA] = R.a;
        dst[kRecB] = R.b;
        dst[kRecC] = R.c;
        dst[kRecD] = R.d;
        dst[kRecE] = R.e;
        dst[kRecH] = R.h;
        if (a.face_mesh) a.face_mesh[f] = n;
    }
    if (!a.do_count) return;
    int bx0 = 1, bx1 = 0, by0 = 1, by1 = 0;
    if (n >= 0) bin_rect(R, a.S, a.bin, bx0, bx1, by0, by1);
    count_bins(a.counts, n, a.nb, bx0, bx1, by0, by1);
}

// ---------------------------------------------------------------------------
// scan: one block; clamps counts, exclusive scan, resets cursors and queue, finds the long lists
// ---------------------------------------------------------------------------
// Bound by the latency of its rounds, so a thread takes four bins in each (16
// bytes at a time): 32,768 bins 56 -> 27 us.
constexpr int kScanBins = 4, kScanRound = 1024 * kScanBins;

// bins b .. b + 3 of an array of NB, 0 past its end (b a multiple of 4, the
// array 16-byte aligned)
__device__ __forceinline__ int4 load_bins(const int *a, int64_t b, int64_t NB) {
    if (b + 3 < NB) return *reinterpret_cast<const int4 *>(a + b);
    return make_int4(b < NB ? a[b] : 0, b + 1 < NB ? a[b + 1] : 0, b + 2 < NB ? a[b + 2] : 0, 0);
}
__device__ __forceinline__ void store_bins(int *a, int64_t b, int64_t NB, const int (&v)[kScanBins]) {
    if (b + 3 < NB) {
        *reinterpret_cast<int4 *>(a + b) = make_int4(v[0], v[1], v[2], v[3]);
        return;
    }
    for (int j = 0; j < 3; ++j)
        if (b + j < NB) a[b + j] = v[j];
}

__global__ void __launch_bounds__(1024) k_scan(ScanArgs a) {
    __shared__ long long warp_sums[32];
    __shared__ long long carry_s;   // running sum of the clamped counts (may exceed the capacity)
    __shared__ int maxc_s;
    __shared__ unsigned long long tot_s;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid == 0) {
        carry_s = 0;
        maxc_s = 0;
        tot_s = 0ull;
        *a.queue = 0u;
        // packed-layout validation of first_face / num_faces
        unsigned bad = 0;
        int64_t prev_end = 0;
        for (int n = 0; n < a.N; ++n) {
            int64_t lo = a.first_face[n], cnt = a.num_faces[n];
            if (lo < 0 || cnt < 0 || lo + cnt > a.F || lo < prev_end) bad |= MESHRAST_ST_BAD_MESH_RANGE;
            prev_end = lo + (cnt > 0 ? cnt : 0);
        }
        set_status(a.status, bad);
    }
    __syncthreads();
    bool overflow = false;
    int local_max = 0;
    unsigned long long local_tot = 0;
    for (int64_t base = 0; base < a.NB; base += kScanRound) {
        const int64_t b = base + tid * kScanBins;
        const int4 c4 = load_bins(a.counts, b, a.NB);
        const int c[kScanBins] = {c4.x, c4.y, c4.z, c4.w};
        int e[kScanBins], off[kScanBins], zero[kScanBins] = {0, 0, 0, 0};
        long long sum = 0;
#pragma unroll
        for (int j = 0; j < kScanBins; ++j) {
            local_max = max(local_max, c[j]);
            local_tot += (unsigned long long)c[j];
            e[j] = c[j];
            if (e[j] > a.max_per_bin) { e[j] = a.max_per_bin; overflow = true; }
            sum += e[j];
        }
        // block exclusive scan (64-bit: a round's counts may sum past 2^31)
        long long x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_sums[wid] = x;
        __syncthreads();
        if (wid == 0) {
            long long s = warp_sums[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                long long y = __shfl_up_sync(0xffffffffu, s, o);
                if (lane >= o) s += y;
            }
            warp_sums[lane] = s;
        }
        __syncthreads();
        const long long carry = carry_s;
        // 64-bit position; entries past the capacity are dropped (overflow bit)
        long long excl = carry + (wid ? warp_sums[wid - 1] : 0ll) + x - sum;
#pragma unroll
        for (int j = 0; j < kScanBins; ++j) {
            const long long next = excl + e[j], room = (long long)a.capacity - excl;
            if ((long long)e[j] > room) { e[j] = (int)max(0ll, room); overflow = overflow || b + j < a.NB; }
            off[j] = (int)min(excl, (long long)a.capacity);  // capacity < 2^31 (checked on the host)
            excl = next;
        }
        store_bins(a.offsets, b, a.NB, off);
        store_bins(a.eff, b, a.NB, e);
        store_bins(a.cursor, b, a.NB, zero);
        __syncthreads();
        if (tid == 1023) carry_s = carry + warp_sums[31];
        __syncthreads();
    }
    // block totals: warp reductions first, then one shared atomic per warp
    local_max = __reduce_max_sync(0xffffffffu, local_max);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) local_tot += __shfl_xor_sync(0xffffffffu, local_tot, o);
    if (lane == 0) {
        atomicMax(&maxc_s, local_max);
        atomicAdd(&tot_s, local_tot);
    }
    if (__any_sync(0xffffffffu, overflow) && lane == 0) set_status(a.status, MESHRAST_ST_BIN_OVERFLOW);
    __syncthreads();
    if (tid == 0) {
        a.offsets[a.NB] = (int)min(carry_s, (long long)a.capacity);
        *a.maxcount = maxc_s;
        *a.total = (long long)tot_s;
        if (a.longs) *a.longs = 0u;
    }
    if (a.longs) {
        const int from = long_list((long long)tot_s, maxc_s);
        if (from < maxc_s) {
            __syncthreads();
            for (int64_t b = tid; b < a.NB; b += 1024)
                if (a.eff[b] > from) a.long_bins[atomicAdd(a.longs, 1u)] = {(int)b, 0u};
        }
    }
    if (!a.order) return;
    // Queue order of the fine pass: bins by descending work class (the bit
    // length of the clamped count), a counting sort over 32 classes, so the
    // longest bins start first and the short ones fill the tail.  The order
    // within a class is whatever the atomics give: each bin's output depends
    // on that bin alone.
    __shared__ int cls_n[32];
    if (tid < 32) cls_n[tid] = 0;
    __syncthreads();
    auto bin_class = [&](const int4 &e, int j, int64_t b) {  // 0: empty bin; eff < 2^31
        const int v = j == 0 ? e.x : j == 1 ? e.y : j == 2 ? e.z : e.w;
        return b + j < a.NB ? 32 - __clz(v) : -1;
    };
    for (int64_t base = 0; base < a.NB; base += kScanRound) {  // every lane takes every round
        const int64_t b = base + tid * kScanBins;
        const int4 e = load_bins(a.eff, b, a.NB);
#pragma unroll
        for (int j = 0; j < kScanBins; ++j) {
            const int cls = bin_class(e, j, b);
            const unsigned grp = __match_any_sync(0xffffffffu, cls);
            if (cls >= 0 && lane == __ffs(grp) - 1) atomicAdd(&cls_n[cls], __popc(grp));
        }
    }
    __syncthreads();
    if (tid == 0) {
        int s = 0;
        for (int c = 31; c >= 0; --c) {
            const int n = cls_n[c];
            cls_n[c] = s;  // first position of class c
            s += n;
        }
    }
    __syncthreads();
    for (int64_t base = 0; base < a.NB; base += kScanRound) {
        const int64_t b = base + tid * kScanBins;
        const int4 e = load_bins(a.eff, b, a.NB);
#pragma unroll
        for (int j = 0; j < kScanBins; ++j) {
            const int cls = bin_class(e, j, b);
            const unsigned grp = __match_any_sync(0xffffffffu, cls);
            const int leader = __ffs(grp) - 1;
            int first = 0;
            if (cls >= 0 && lane == leader) first = atomicAdd(&cls_n[cls], __popc(grp));
            first = __shfl_sync(0xffffffffu, first, leader);
            if (cls >= 0) a.order[first + __popc(grp & ((1u << lane) - 1u))] = (int)(b + j);
        }
    }
}

// ---------------------------------------------------------------------------
// fill: warp-aggregated atomic append into the per-bin lists
// ---------------------------------------------------------------------------
// Lower bound on a face's depth at any pixel where it is a candidate (nearest
// corner), valid when the depth is a convex combination of the corner depths:
// with clipping, or without blur (inside pixels only).  Slightly reduced so
// that fp32 rounding of the key can never fall below it.
__device__ __forceinline__ float face_zmin(const FaceRec &R) {
    if (!(R.c.x <= R.c.y)) return __int_as_float(0x7f800000);  // culled
    return __fdividef(1.f, fmaxf(R.d.y, fmaxf(R.d.z, R.d.w))) * (1.f - 1e-6f);
}

// Bin-list entry: nearest-corner depth (a positive float, so its bits order
// like the value) in the high word, face id in the low word; sorting entries
// as integers orders a bin's faces front to back, ties by id.
__device__ __forceinline__ unsigned long long bin_entry(float zmin, int f) {
    return ((unsigned long long)__float_as_uint(zmin) << 32) | (unsigned)f;
}

__global__ void __launch_bounds__(256) k_fill(FillArgs a) {
    const int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int n = -1;
    FaceRec R;
    if (f < a.F) {
        n = a.face_mesh[f];
        if (n >= 0) {
            const float4 *src = reinterpret_cast<const float4 *>(a.rec + f);
            R.c = src[kRecC];
            R.d = src[kRecD];
        }
    }
    int bx0 = 1, bx1 = 0, by0 = 1, by1 = 0;
    if (n >= 0) bin_rect(R, a.S, a.bin, bx0, bx1, by0, by1);
    const unsigned long long entry = n >= 0 ? bin_entry(face_zmin(R), (int)f) : 0ull;
    fill_bins(a.lists, a.cursor, a.eff, a.offsets, entry, n, a.nb, bx0, bx1, by0, by1);
}

// ---------------------------------------------------------------------------
// output of one pixel's K fragments
// ---------------------------------------------------------------------------
template <int KM, bool BL>
__device__ __forceinline__ void write_pixel(const FineOut &o, int64_t pix, int K, const TopK<KM> &tk,
                                            const FaceRec *rec, const PixC &p, const EvalFlags &fl,
                                            const FineBlend &bl) {
    const int64_t s0 = pix * (int64_t)K;
    FwdBlend fb;
#pragma unroll
    for (int k = 0; k < KM; ++k) {
        if (k < KM - K) continue;
        const int64_t s = s0 + k - (KM - K);
        const int f = tk.f[k];
        const bool store = !BL || bl.frag;
        if (f == 0x7fffffff) {
            if (store) {
                o.pix_to_face[s] = -1;
                o.zbuf[s] = -1.f;
                o.bary[3 * s] = -1.f;
                o.bary[3 * s + 1] = -1.f;
                o.bary[3 * s + 2] = -1.f;
                o.dists[s] = -1.f;
            }
        } else {
            FaceRec R;
            const float4 *src = reinterpret_cast<const float4 *>(rec + f);
            R.a = __ldg(src + kRecA);
            R.b = __ldg(src + kRecB);
            R.c = __ldg(src + kRecC);
            R.d = __ldg(src + kRecD);
            R.e = __ldg(src + kRecE);
            float bp[3], d;
            face_fragment(R, p, fl, bp, d);
            if (store) {
                o.pix_to_face[s] = f;
                o.zbuf[s] = tk.z[k];
                o.bary[3 * s] = bp[0];
                o.bary[3 * s + 1] = bp[1];
                o.bary[3 * s + 2] = bp[2];
                o.dists[s] = d;
            }
            if constexpr (BL) fb.slot(bl, d);
        }
    }
    if constexpr (BL) fb.end(bl, pix);
}

// Fragments of one pixel's K winners written directly by the owning thread,
// 16-byte vector stores when K is a multiple of 4 (ids: K/2, depths and
// distances: K/4, barycentrics: 3K/4 stores per pixel).

template <int KM, bool BL>
__device__ __forceinline__ void write_pixel_vec(const FineOut &o, int64_t pix, int K, const TopK<KM> &tk,
                                                const FaceRec *rec, const PixC &p, const EvalFlags &fl,
                                                const FineBlend &bl) {
    if (K != KM || (KM % 4) != 0) {
        write_pixel<KM, BL>(o, pix, K, tk, rec, p, fl, bl);
        return;
    }
    FwdBlend fb;
    const bool store = !BL || bl.frag;
    const int64_t s0 = pix * KM;
    const unsigned long long pol = l2_keep_policy();
    longlong2 *ip = reinterpret_cast<longlong2 *>(o.pix_to_face + s0);
    float4 *zp = reinterpret_cast<float4 *>(o.zbuf + s0);
    float4 *dp = reinterpret_cast<float4 *>(o.dists + s0);
    float4 *bp = reinterpret_cast<float4 *>(o.bary + s0 * 3);
#pragma unroll
    for (int j = 0; j < KM / 2; ++j) {
        if (!store) break;
        longlong2 v;
        v.x = (tk.f[2 * j] == 0x7fffffff) ? -1ll : (long long)tk.f[2 * j];
        v.y = (tk.f[2 * j + 1] == 0x7fffffff) ? -1ll : (long long)tk.f[2 * j + 1];
        st_keep(ip + j, v, pol);
    }
    // four slots at a time: one float4 of depths, of distances, three of barycentrics
#pragma unroll
    for (int j = 0; j < KM / 4; ++j) {
        float bb[4][3], dd[4], zz[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int k = 4 * j + i;
            bb[i][0] = bb[i][1] = bb[i][2] = -1.f;
            dd[i] = -1.f;
            zz[i] = -1.f;
            if (tk.f[k] == 0x7fffffff) continue;
            FaceRec R;
            const float4 *src = reinterpret_cast<const float4 *>(rec + tk.f[k]);
            R.a = __ldg(src + kRecA);
            R.b = __ldg(src + kRecB);
            R.c = __ldg(src + kRecC);
            R.d = __ldg(src + kRecD);
            R.e = __ldg(src + kRecE);
            face_fragment(R, p, fl, bb[i], dd[i]);
            zz[i] = tk.z[k];
            if constexpr (BL) fb.slot(bl, dd[i]);
        }
        if (!store) continue;
        st_keep(zp + j, make_float4(zz[0], zz[1], zz[2], zz[3]), pol);
        st_keep(dp + j, make_float4(dd[0], dd[1], dd[2], dd[3]), pol);
        st_keep(bp + 3 * j, make_float4(bb[0][0], bb[0][1], bb[0][2], bb[1][0]), pol);
        st_keep(bp + 3 * j + 1, make_float4(bb[1][1], bb[1][2], bb[2][0], bb[2][1]), pol);
        st_keep(bp + 3 * j + 2, make_float4(bb[2][2], bb[3][0], bb[3][1], bb[3][2]), pol);
    }
    if constexpr (BL) fb.end(bl, pix);
}

// A pixel's packed silhouette slots, and Algorithm 1 on them (the arithmetic
// and order of FwdBlend).
template <int KM>
__device__ __forceinline__ void write_pixel_packed(const FineBlend &bl, int64_t pix, int K, const TopK<KM> &tk,
                                                   const FaceRec *rec, const PixC &p) {
    unsigned long long *out = bl.slots + pix * K;
    float keep = 1.f;
#pragma unroll
    for (int k = 0; k < KM; ++k) {
        if (k < KM - K) continue;
        const int f = tk.f[k], j = k - (KM - K);
        if (f == 0x7fffffff) {
            out[j] = kSilEnd;
            break;
        }
        FaceRec R;
        const float4 *src = reinterpret_cast<const float4 *>(rec + f);
        R.a = __ldg(src + kRecA);
        R.b = __ldg(src + kRecB);
        R.d = __ldg(src + kRecD);
        int edge;
        const float d = face_distance(R, p, edge);
        keep *= sigmoidf_(d / bl.sigma);
        out[j] = sil_pack(d, f, edge);
    }
    bl.keep[pix] = keep;
    reinterpret_cast<float4 *>(bl.image)[pix] = make_float4(0.f, 0.f, 0.f, 1.f - keep);
}

// ---------------------------------------------------------------------------
// fine pass: persistent blocks, one bin (bin x bin pixels = block) per item
// ---------------------------------------------------------------------------
// Two forms of a window.  0: what an early stop shortens; as many entries as fit the
// usual bin whole.  1: K > 16 without depth culling, where every face is met: an order
// only keeps the insertions short (unordered, 4 meshes of 81,920 faces, 256 px, K = 50:
// 7,008 us; ordered 4,673), and room for another block counts for more than long
// windows.  Shared memory of a block, besides the lists, and blocks per SM: form 0 48 KB
// (bins of 16) or 13 KB, limited by registers; form 1 27 or 11 KB, 3 blocks of bins of
// 16 at K = 24 (8 meshes of 5,120 faces, 256 px: 483 -> 421 us; bins of 8, K = 50: 663 ->
// 595).
constexpr int fine_window(int BS, int FORM) { return FORM ? (BS >= 16 ? 384 : 256) : BS >= 16 ? 1024 : 512; }
// Where the walk has a window's boxes from: the eight warps of a bin of 16 share them
// in shared memory (1.3M faces, K = 1: 382 us; with the records 402); the two warps of a
// bin of 8 bring them with the records, which leaves room for 16 blocks (8 meshes of
// 5,120 faces, 256 px, K = 4: 144 -> 132); form 1 reads them from L1.
enum { kBoxWindow, kBoxRecord, kBoxL1 };
constexpr int fine_boxes(int BS, int FORM) { return BS < 16 ? kBoxRecord : FORM ? kBoxL1 : kBoxWindow; }
// blocks per SM: 64, 80 and 128 registers hold the lists and the face test (K > 16: the
// lists in shared memory leave room for fewer)
constexpr int fine_blocks(int KM, int BS) { return (KM <= 4 ? 4 : KM == 8 ? 3 : 2) * 256 / (BS * BS); }

// OUT: 0 Fragment data, 1 with the silhouette blend, 2 packed silhouette slots with it
template <int KM, int BS, int OUT, int FORM>
__global__ void __launch_bounds__(BS *BS, fine_blocks(KM, BS)) k_fine(FineArgs a) {
    constexpr int BD = BS * BS;
    constexpr int WIN = fine_window(BS, FORM), BOX = fine_boxes(BS, FORM), NREC = BOX == kBoxRecord ? 6 : 5;
    __shared__ float4 s_box[BOX == kBoxWindow ? WIN : 1];  // the window's bboxes: lanes read them side by side
    __shared__ float4 s_rec[BD / 32][32][NREC];            // per warp: a, b, d, e, h (c) of the faces it walks next
    __shared__ WindowShared<WIN> s_win;
    __shared__ int s_item;
    // K > 16: the per-thread lists
    extern __shared__ unsigned long long s_lists[];
    const int tid = threadIdx.x;
    // K <= 16: each warp covers an 8 x 4 block of the bin (about as wide as
    // tall, like the inflated face bboxes it is culled against); K > 16: two
    // rows (the tile writer below walks slots in row order)
    const int ty = KM > 0 ? ((tid >> 5) / (BS / 8)) * 4 + ((tid & 31) >> 3) : tid / BS;
    const int tx = KM > 0 ? ((tid >> 5) % (BS / 8)) * 8 + (tid & 7) : tid % BS;
    EvalFlags fl = a.fl;
    const bool zcull = fl.clip || !(fl.blur > 0.f);
    const int nb2 = a.nb * a.nb;
    const int sorted_from = a.total ? long_list(*a.total, *a.maxcount) : 0x7fffffff;
    float4 (*const rec)[NREC] = s_rec[tid >> 5];
    while (true) {
        if (tid == 0) s_item = (int)atomicAdd(a.queue, 1u);
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= a.items) break;
        const int bin = a.order ? __ldg(a.order + item) : item;  // longest bins first
        const int n = bin / nb2, rem = bin - n * nb2;
        const int by = rem / a.nb, bx = rem - by * a.nb;
        const int r = by * BS + ty, c = bx * BS + tx;
        fl.znear = __ldg(a.cams + 16 * n + 13);
        const bool valid = (r < a.S) && (c < a.S);
        const PixC p = pixel_centre(r, c, a.S);
        // rectangle spanned by the centres of this warp's valid pixels (x and y
        // decrease with the column and row index); empty when no lane is valid
        const int lane = tid & 31;
        float wx0 = 1.f, wx1 = -1.f, wy0 = 1.f, wy1 = -1.f;
        {
            const unsigned cmin = __reduce_min_sync(0xffffffffu, valid ? (unsigned)c : 0xffffffffu);
            const unsigned cmax = __reduce_max_sync(0xffffffffu, valid ? (unsigned)c : 0u);
            const unsigned rmin = __reduce_min_sync(0xffffffffu, valid ? (unsigned)r : 0xffffffffu);
            const unsigned rmax = __reduce_max_sync(0xffffffffu, valid ? (unsigned)r : 0u);
            if (cmin <= cmax) {
                wx1 = pc_hi((int)cmin, a.S);
                wx0 = pc_hi((int)cmax, a.S);
                wy1 = pc_hi((int)rmin, a.S);
                wy0 = pc_hi((int)rmax, a.S);
            }
        }
        const int cnt = a.eff[bin];
        const int off = a.offsets[bin];
        TopK<(KM > 0 ? KM : 1)> tk;
        SmemTopK stk;
        if constexpr (KM > 0) {
            tk.init(a.K);
        } else {
            stk.z = reinterpret_cast<float *>(s_lists) + tid * a.K;
            stk.f = reinterpret_cast<int *>(s_lists) + BD * a.K + tid * a.K;
            stk.stride = 1;
            stk.K = a.K;
            stk.init();
        }
        auto kth = [&]() {
            if constexpr (KM > 0) return tk.z[KM - 1];
            else return stk.thr();
        };
        auto warp_kth = [&]() {
            return __int_as_float(__reduce_max_sync(0xffffffffu, valid ? __float_as_int(kth()) : 0));
        };
        // The bin's faces in front-to-back windows (two warps' worth is not
        // worth ordering; without depth culling the order only helps lists in
        // shared memory, which are inserted into from their ends).
        // Within a window the warps go their own way.  Faces are culled 32 at
        // a time for the whole warp: lane j tests face jb + j against the
        // rectangle spanned by the warp's pixel centres and against the warp's
        // largest K-th depth; one ballot names the faces the warp walks pixel
        // by pixel, and their lanes bring the records to the warp's own part
        // of shared memory.  A face is skipped
        // by a lane when its bbox misses the pixel or its nearest corner lies
        // behind the lane's K-th depth.  Once a warp's largest K-th depth
        // falls into a bucket in front of the next face's, the rest of the
        // window is behind all its lanes, and the block stops when everything
        // left is behind every warp.  (Staging the records for the block, 256
        // at a time, made all warps wait for the slowest at every 256: 700
        // against 633 us at 1.3M faces, 1024 px, K = 8, 225 against 176 for 5
        // meshes at 225 px; reading them from L1 one by one, 297 against 246
        // where few faces reach a warp: 1.3M faces, K = 1, no blur.)
        window_begin<BD>(s_win, a.lists + off, cnt, (zcull || KM == 0) && cnt > 64, cnt > sorted_from);
        while (const int m = window_next<BD>(s_win)) {
            if constexpr (BOX == kBoxWindow) {
                for (int i = tid; i < m; i += BD)
                    s_box[i] = __ldg(reinterpret_cast<const float4 *>(a.rec + (unsigned)s_win.ent[i]) + kRecC);
                __syncthreads();
            }
            for (int jb = 0; jb < m; jb += 32) {
                const float wthr = warp_kth();
                if (zcull && s_win.behind(entry_key(s_win.ent[jb]), wthr)) break;
                const int jl = jb + lane;
                bool hit = false;
                if (jl < m) {
                    const unsigned long long e = s_win.ent[jl];
                    const float4 bb =
                        BOX == kBoxWindow ? s_box[jl] : __ldg(reinterpret_cast<const float4 *>(a.rec + (unsigned)e) + kRecC);
                    hit = bb.x <= wx1 && bb.y >= wx0 && bb.z <= wy1 && bb.w >= wy0 && !(zcull && entry_key(e) > wthr);
                    if (hit) {
                        const float4 *src = reinterpret_cast<const float4 *>(a.rec + (unsigned)e);
                        rec[lane][0] = __ldg(src + kRecA);
                        rec[lane][1] = __ldg(src + kRecB);
                        rec[lane][2] = __ldg(src + kRecD);
                        rec[lane][3] = __ldg(src + kRecE);
                        rec[lane][4] = __ldg(src + kRecH);
                        if constexpr (BOX == kBoxRecord) rec[lane][5] = bb;
                    }
                }
                unsigned mask = __ballot_sync(0xffffffffu, hit);
                __syncwarp();
                while (mask) {
                    const int j = __ffs(mask) - 1, jj = jb + j;
                    mask &= mask - 1;
                    if (!valid) continue;
                    FaceRec R;
                    if constexpr (BOX == kBoxWindow) R.c = s_box[jj];
                    else if constexpr (BOX == kBoxRecord) R.c = rec[j][5];
                    else R.c = __ldg(reinterpret_cast<const float4 *>(a.rec + (unsigned)s_win.ent[jj]) + kRecC);
                    if (!in_bbox(R, p)) continue;
                    const unsigned long long e = s_win.ent[jj];
                    if (zcull && entry_key(e) > kth()) continue;
                    const int fid = (int)(unsigned)e;
                    R.a = rec[j][0];
                    R.b = rec[j][1];
                    R.d = rec[j][2];
                    R.e = rec[j][3];
                    R.h = rec[j][4];
                    float z;
                    if (face_key_nobbox(R, p, fl, z)) {
                        if constexpr (KM > 0) {
                            if (tk.admits(z, fid)) tk.insert(z, fid);
                        } else {
                            if (stk.admits(z, fid)) stk.insert(z, fid);
                        }
                    }
                }
                __syncwarp();
            }
            if (__syncthreads_and(zcull && s_win.rest_behind(warp_kth()))) break;
        }
        if constexpr (KM > 0) {
            const int64_t pix = ((int64_t)n * a.S + r) * a.S + c;
            if constexpr (OUT == 2) {
                if (valid) write_pixel_packed<KM>(a.blend, pix, a.K, tk, a.rec, p);
            } else {
                if (valid) write_pixel_vec<KM, OUT == 1>(a.out, pix, a.K, tk, a.rec, p, fl, a.blend);
            }
        } else {
            // K > 16: the block writes its tile slot by slot: consecutive
            // threads take consecutive output slots of a tile row (coalesced),
            // each recomputing its slot's barycentrics and distance
            int *const s_held = reinterpret_cast<int *>(s_win.ent);  // (the window is done)
            s_held[tid] = valid ? stk.n : 0;
            __syncthreads();
            const int K = a.K;
            const int rows = min(BS, a.S - by * BS), cols = min(BS, a.S - bx * BS);
            const int per_row = cols * K;
            const float *lz = reinterpret_cast<const float *>(s_lists);
            const int *lf = reinterpret_cast<const int *>(s_lists) + BD * K;
            for (int i = tid; i < rows * per_row; i += BD) {
                const int ry = i / per_row, rem = i - ry * per_row;
                const int cx = rem / K, k = rem - cx * K;
                const int t = ry * BS + cx;
                const int rr = by * BS + ry, cc = bx * BS + cx;
                const int64_t sl = (((int64_t)n * a.S + rr) * a.S + cc) * K + k;
                if (k < s_held[t]) {
                    const int f = lf[t * K + k];
                    FaceRec R;
                    const float4 *src = reinterpret_cast<const float4 *>(a.rec + f);
                    R.a = __ldg(src + kRecA);
                    R.b = __ldg(src + kRecB);
                    R.c = __ldg(src + kRecC);
                    R.d = __ldg(src + kRecD);
                    R.e = __ldg(src + kRecE);
                    float bp[3], d;
                    face_fragment(R, pixel_centre(rr, cc, a.S), fl, bp, d);
                    a.out.pix_to_face[sl] = f;
                    a.out.zbuf[sl] = lz[t * K + k];
                    a.out.bary[3 * sl] = bp[0];
                    a.out.bary[3 * sl + 1] = bp[1];
                    a.out.bary[3 * sl + 2] = bp[2];
                    a.out.dists[sl] = d;
                } else {
                    a.out.pix_to_face[sl] = -1;
                    a.out.zbuf[sl] = -1.f;
                    a.out.bary[3 * sl] = -1.f;
                    a.out.bary[3 * sl + 1] = -1.f;
                    a.out.bary[3 * sl + 2] = -1.f;
                    a.out.dists[sl] = -1.f;
                }
            }
            __syncthreads();
        }
    }
}

// ---------------------------------------------------------------------------
// plain form: every pixel against every face of its image, one launch
// ---------------------------------------------------------------------------
// A block takes 8 x 4 pixels, one per lane, and its eight warps share out the
// image's faces 32 at a time: lane j tests face j's box against the block's
// pixel centres and the warp walks the faces one ballot names.  (One thread
// per pixel over all faces left a 64 x 64 image with 16 blocks, each a serial
// chain of 1,280 record loads.)  The warps' sorted lists meet in shared
// memory: an entry's place among all eight is its place in its own list plus
// the entries before it in the others, and the thread that holds it writes
// that slot.  A call on 64 x 64 pixels and 1,280 faces, K = 1: 344 -> 53 us, what
// is left is the host's share.
constexpr int kPlainWarps = 8;

template <int KM>
__global__ void __launch_bounds__(kPlainWarps * 32) k_naive(NaiveArgs a) {
    extern __shared__ unsigned char s_dyn[];  // depths, then ids: [warp][K][lane]
    __shared__ int s_n[kPlainWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int n = blockIdx.y, K = a.K;
    const int bw = (a.S + 7) / 8;
    const int r = (int)(blockIdx.x / bw) * 4 + (lane >> 3), c = (int)(blockIdx.x % bw) * 8 + (lane & 7);
    const bool valid = r < a.S && c < a.S;
    const PixC p = pixel_centre(r, c, a.S);
    // the block's pixel centres (x and y decrease with the column and row)
    const int r0 = (int)(blockIdx.x / bw) * 4, c0 = (int)(blockIdx.x % bw) * 8;
    const float wx1 = pc_hi(c0, a.S), wx0 = pc_hi(min(c0 + 7, a.S - 1), a.S);
    const float wy1 = pc_hi(r0, a.S), wy0 = pc_hi(min(r0 + 3, a.S - 1), a.S);
    EvalFlags fl = a.fl;
    fl.znear = __ldg(a.cams + 16 * n + 13);
    const int64_t lo = max(a.first_face[n], (int64_t)0), hi = min(a.first_face[n] + a.num_faces[n], a.F);
    float *lz = reinterpret_cast<float *>(s_dyn) + (size_t)w * K * 32 + lane;
    int *lf = reinterpret_cast<int *>(s_dyn) + (size_t)(kPlainWarps + w) * K * 32 + lane;
    TopK<(KM > 0 ? KM : 1)> tk;
    SmemTopK stk;
    if constexpr (KM > 0) {
        tk.init(K);
    } else {
        stk.z = lz;
        stk.f = lf;
        stk.stride = 32;
        stk.K = K;
        stk.init();
    }
    for (int64_t fb = lo + 32 * w; fb < hi; fb += 32 * kPlainWarps) {
        bool hit = false;
        if (fb + lane < hi) {
            const float4 bb = __ldg(reinterpret_cast<const float4 *>(a.rec + fb + lane) + kRecC);
            hit = bb.x <= wx1 && bb.y >= wx0 && bb.z <= wy1 && bb.w >= wy0;
        }
        unsigned mask = __ballot_sync(0xffffffffu, hit);
        while (mask) {
            const int f = (int)fb + __ffs(mask) - 1;
            mask &= mask - 1;
            FaceRec R;
            const float4 *src = reinterpret_cast<const float4 *>(a.rec + f);
            R.a = __ldg(src + kRecA);
            R.b = __ldg(src + kRecB);
            R.c = __ldg(src + kRecC);
            R.d = __ldg(src + kRecD);
            R.e = __ldg(src + kRecE);
            R.h = __ldg(src + kRecH);
            float z;
            if (valid && face_key(R, p, fl, z)) {
                if constexpr (KM > 0) {
                    if (tk.admits(z, f)) tk.insert(z, f);
                } else {
                    if (stk.admits(z, f)) stk.insert(z, f);
                }
            }
        }
    }
    int held = 0;
    if constexpr (KM > 0) {
#pragma unroll
        for (int k = 0; k < KM; ++k) {
            if (tk.f[k] < 0 || tk.f[k] == 0x7fffffff) continue;  // unused or empty
            lz[held * 32] = tk.z[k];
            lf[held * 32] = tk.f[k];
            ++held;
        }
    } else {
        held = stk.n;
    }
    s_n[w][lane] = held;
    __syncthreads();
    if (!valid) return;
    const int64_t s0 = (((int64_t)n * a.S + r) * a.S + c) * K;
    int at[kPlainWarps], total = 0;  // entries of each list in front of the current one
#pragma unroll
    for (int v = 0; v < kPlainWarps; ++v) {
        at[v] = 0;
        total += s_n[v][lane];
    }
    for (int k = 0; k < held; ++k) {
        const float z = lz[k * 32];
        const int f = lf[k * 32];
        int rank = k;
#pragma unroll
        for (int v = 0; v < kPlainWarps; ++v) {
            if (v == w) continue;
            const float *oz = lz + (v - w) * K * 32;
            const int *of = lf + (v - w) * K * 32;
            while (at[v] < s_n[v][lane] && key_less(oz[at[v] * 32], of[at[v] * 32], z, f)) ++at[v];
            rank += at[v];
        }
        if (rank >= K) break;
        FaceRec R;
        const float4 *src = reinterpret_cast<const float4 *>(a.rec + f);
        R.a = __ldg(src + kRecA);
        R.b = __ldg(src + kRecB);
        R.d = __ldg(src + kRecD);
        R.e = __ldg(src + kRecE);
        float bp[3], d;
        face_fragment(R, p, fl, bp, d);
        const int64_t s = s0 + rank;
        a.out.pix_to_face[s] = f;
        a.out.zbuf[s] = z;
        a.out.bary[3 * s] = bp[0];
        a.out.bary[3 * s + 1] = bp[1];
        a.out.bary[3 * s + 2] = bp[2];
        a.out.dists[s] = d;
    }
    for (int k = total + w; k < K; k += kPlainWarps) {
        const int64_t s = s0 + k;
        a.out.pix_to_face[s] = -1;
        a.out.zbuf[s] = -1.f;
        a.out.bary[3 * s] = -1.f;
        a.out.bary[3 * s + 1] = -1.f;
        a.out.bary[3 * s + 2] = -1.f;
        a.out.dists[s] = -1.f;
    }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
static int km_for(int K) {
    if (K <= 1) return 1;
    if (K <= 2) return 2;
    if (K <= 4) return 4;
    if (K <= 8) return 8;
    if (K <= 16) return 16;
    return 0;  // shared-memory lists
}

template <int KM, int BS, int OUT, int FORM = 0>
static cudaError_t launch_fine_t(const FineArgs &a, cudaStream_t st) {
    constexpr int BD = BS * BS;
    const size_t dyn = (KM > 0) ? (size_t)0 : (size_t)BD * a.K * 8;
    auto kern = k_fine<KM, BS, OUT, FORM>;
    cudaError_t e = cudaSuccess;
    if (dyn > 0) {  // static + dynamic above 48 KB needs the opt-in
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
        if (e != cudaSuccess) return e;
    }
    const int grid = mr_host::queue_blocks(a.items, 2048 / BD);
    kern<<<grid, BD, dyn, st>>>(a);
    return cudaGetLastError();
}

// The silhouette blend runs inside the fine pass for K <= 16; the softmax
// blend does not (its colour gathers cost the fine pass more than the separate
// blend kernel's pass over the fragments).
bool fine_blends(int K, bool rgb) { return km_for(K) > 0 && !rgb; }

cudaError_t launch_fine(const FineArgs &a, int bin, cudaStream_t st) {
    const int km = km_for(a.K);
    const int out = a.blend.on ? (a.blend.slots ? 2 : 1) : 0;
#define MR_FINE(KM_, BS_)                                                              \
    if (km == KM_ && bin == BS_)                                                       \
        return out == 2   ? launch_fine_t<KM_, BS_, 2>(a, st)                          \
               : out == 1 ? launch_fine_t<KM_, BS_, 1>(a, st) : launch_fine_t<KM_, BS_, 0>(a, st);
    MR_FINE(1, 8) MR_FINE(2, 8) MR_FINE(4, 8) MR_FINE(8, 8) MR_FINE(16, 8)
    MR_FINE(1, 16) MR_FINE(2, 16) MR_FINE(4, 16) MR_FINE(8, 16) MR_FINE(16, 16)
#undef MR_FINE
    if (km == 0) {
        const bool zcull = a.fl.clip || !(a.fl.blur > 0.f);
        if (bin == 8) return zcull ? launch_fine_t<0, 8, 0>(a, st) : launch_fine_t<0, 8, 0, 1>(a, st);
        if (bin == 16) return zcull ? launch_fine_t<0, 16, 0>(a, st) : launch_fine_t<0, 16, 0, 1>(a, st);
    }
    return cudaErrorInvalidValue;
}

template <int KM>
static cudaError_t launch_naive_t(const NaiveArgs &a, int N, cudaStream_t st) {
    const size_t dyn = (size_t)kPlainWarps * a.K * 32 * 8;  // at most 128 KB
    auto kern = k_naive<KM>;
    if (dyn > 40 * 1024) {  // static + dynamic above 48 KB needs the opt-in
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
        if (e != cudaSuccess) return e;
    }
    const unsigned tiles = (unsigned)((a.S + 7) / 8) * (unsigned)((a.S + 3) / 4);
    kern<<<dim3(tiles, (unsigned)N), kPlainWarps * 32, dyn, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_naive(const NaiveArgs &a, int N, cudaStream_t st) {
    switch (km_for(a.K)) {
        case 1: return launch_naive_t<1>(a, N, st);
        case 2: return launch_naive_t<2>(a, N, st);
        case 4: return launch_naive_t<4>(a, N, st);
        case 8: return launch_naive_t<8>(a, N, st);
        case 16: return launch_naive_t<16>(a, N, st);
        default: return launch_naive_t<0>(a, N, st);
    }
}

cudaError_t launch_stage(const StageArgs &a, cudaStream_t st) {
    if (a.F <= 0) return cudaSuccess;
    const int grid = (int)((a.F + 255) / 256);
    k_stage<<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_scan(const ScanArgs &a, cudaStream_t st) {
    k_scan<<<1, 1024, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_fill(const FillArgs &a, cudaStream_t st) {
    if (a.F <= 0) return cudaSuccess;
    const int grid = (int)((a.F + 255) / 256);
    k_fill<<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace mr
