// Device helpers shared by the mesh and point rasterizers: camera projection
// in double-float, binning rectangles, the front-to-back sort of a bin's
// entries and the shared-memory K-nearest lists.
#pragma once

#include "rast_common.cuh"

namespace mr {

__device__ __forceinline__ int find_mesh(const int64_t *first_face, int N, int64_t f) {
    int lo = 0, hi = N - 1, ans = -1;
    while (lo <= hi) {
        int mid = (lo + hi) >> 1;
        if (first_face[mid] <= f) { ans = mid; lo = mid + 1; } else { hi = mid - 1; }
    }
    return ans;
}

// Image of a block's first element i0 of a packed batch (ranges first[n] ..
// first[n] + num[n]) and that image's range; -1 and an empty range past the
// end.  Thread 0 looks it up; every thread of the block must call it (it
// synchronises the block).
__device__ __forceinline__ void block_image(const int64_t *first, const int64_t *num, int N, int64_t count,
                                            int64_t i0, int &block, int64_t &lo, int64_t &hi) {
    __shared__ int s_n;
    __shared__ long long s_lo, s_hi;
    if (threadIdx.x == 0) {
        const int n0 = i0 < count ? find_mesh(first, N, i0) : -1;
        s_n = n0;
        s_lo = n0 >= 0 ? first[n0] : 0;
        s_hi = n0 >= 0 ? first[n0] + num[n0] : 0;
    }
    __syncthreads();
    block = s_n;
    lo = s_lo;
    hi = s_hi;
}

// Image of element i, or -1: the block's when i lies in its range, else by search.
__device__ __forceinline__ int image_of(const int64_t *first, const int64_t *num, int N, int64_t i, int block,
                                        int64_t lo, int64_t hi) {
    if (block >= 0 && i >= lo && i < hi) return block;
    const int n = find_mesh(first, N, i);
    return (n >= 0 && i < first[n] + num[n]) ? n : -1;
}

// world -> view -> NDC of one corner, in double-float arithmetic
__device__ __forceinline__ void project_corner(const float *cam, float px, float py, float pz, df &X, df &Y,
                                               df &Z) {
    df d0 = two_sum(px, -cam[9]), d1 = two_sum(py, -cam[10]), d2 = two_sum(pz, -cam[11]);
    df x = df_add(df_add(df_mul_f(d0, cam[0]), df_mul_f(d1, cam[1])), df_mul_f(d2, cam[2]));
    df y = df_add(df_add(df_mul_f(d0, cam[3]), df_mul_f(d1, cam[4])), df_mul_f(d2, cam[5]));
    df z = df_add(df_add(df_mul_f(d0, cam[6]), df_mul_f(d1, cam[7])), df_mul_f(d2, cam[8]));
    float f = cam[12];
    X = df_div(df_mul_f(x, f), z);
    Y = df_div(df_mul_f(y, f), z);
    Z = z;
}

__device__ __forceinline__ df df_min(df a, df b) { return (a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo)) ? a : b; }
__device__ __forceinline__ df df_max(df a, df b) { return (a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo)) ? a : b; }

// Columns (or rows) whose fp32 pixel centre lies in [lo, hi]: first index
// with centre <= hi, last index with centre >= lo (centres decrease with the
// index).  Exactly the comparisons the fine pass makes.
__device__ __forceinline__ float pc_hi(int i, int S) {
    float h, l;
    pix_coord(i, S, h, l);
    return h;
}
__device__ __forceinline__ void centre_range(float lo, float hi, int S, int &i0, int &i1) {
    float Sf = (float)S;
    int a = (int)ceilf(fminf(fmaxf(((Sf - 1.f) - hi * Sf) * 0.5f, -1.f), Sf));
    a = max(0, min(a, S));
    while (a > 0 && pc_hi(a - 1, S) <= hi) --a;
    while (a < S && pc_hi(a, S) > hi) ++a;
    int b = (int)floorf(fminf(fmaxf(((Sf - 1.f) - lo * Sf) * 0.5f, -1.f), Sf));
    b = max(-1, min(b, S - 1));
    while (b < S - 1 && pc_hi(b + 1, S) >= lo) ++b;
    while (b >= 0 && pc_hi(b, S) < lo) --b;
    i0 = a;
    i1 = b;
}

// Bins (bx0..bx1, by0..by1) whose pixel-centre span meets the box (xmin,
// xmax, ymin, ymax).  Empty when bx0 > bx1 or by0 > by1.
__device__ __forceinline__ void bin_rect_box(const float4 &box, int S, int bin, int &bx0, int &bx1, int &by0,
                                             int &by1) {
    if (!(box.x <= box.y) || !(box.z <= box.w)) { bx0 = 1; bx1 = 0; by0 = 1; by1 = 0; return; }
    int c0, c1, r0, r1;
    centre_range(box.x, box.y, S, c0, c1);
    centre_range(box.z, box.w, S, r0, r1);
    if (c0 > S - 1 || c1 < 0 || r0 > S - 1 || r1 < 0) { bx0 = 1; bx1 = 0; by0 = 1; by1 = 0; return; }
    bx0 = c0 / bin;
    bx1 = c1 / bin;
    by0 = r0 / bin;
    by1 = r1 / bin;
}

// Bins of a face: the bin's pixel-centre span meets the inflated bbox.
__device__ __forceinline__ void bin_rect(const FaceRec &R, int S, int bin, int &bx0, int &bx1, int &by0,
                                         int &by1) {
    bin_rect_box(R.c, S, bin, bx0, bx1, by0, by1);
}

// The warp's (element, bin) pairs, one bin per lane and step: f(key) with key -1
// for lanes whose rectangle is done.  Every lane of the warp calls it.
template <class F>
__device__ __forceinline__ void for_bins(int n, int nb, int bx0, int bx1, int by0, int by1, const F &f) {
    const int cnt = max(0, bx1 - bx0 + 1) * max(0, by1 - by0 + 1);
    const int wmax = __reduce_max_sync(0xffffffffu, cnt);
    int bx = bx0, row = (n * nb + by0) * nb;
    for (int i = 0; i < wmax; ++i) {
        f(i < cnt ? row + bx : -1);
        if (++bx > bx1) { bx = bx0; row += nb; }
    }
}

// Adds the warp's pairs to the bins' counts, equal bins of a step as one.
__device__ __forceinline__ void count_bins(int *counts, int n, int nb, int bx0, int bx1, int by0, int by1) {
    const int lane = threadIdx.x & 31;
    for_bins(n, nb, bx0, bx1, by0, by1, [&](int key) {
        const unsigned grp = __match_any_sync(0xffffffffu, key);
        if (key >= 0 && lane == __ffs(grp) - 1) atomicAdd(counts + key, __popc(grp));
    });
}

// Appends `entry` to the lists of the element's bins (up to eff entries each
// from offsets), four steps' cursor additions in flight at a time: one at a
// time, each waited for its round trip to L2 (1.3M faces in 14M pairs: 107
// -> 94 us).
__device__ __forceinline__ void fill_bins(unsigned long long *lists, int *cursor, const int *eff, const int *offsets,
                                          unsigned long long entry, int n, int nb, int bx0, int bx1, int by0, int by1) {
    constexpr int U = 4;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int cnt = max(0, bx1 - bx0 + 1) * max(0, by1 - by0 + 1);
    const int wmax = __reduce_max_sync(0xffffffffu, cnt);
    int bx = bx0, row = (n * nb + by0) * nb;
    for (int i = 0; i < wmax; i += U) {
        int key[U], base[U], room[U], off[U];
        unsigned grp[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            key[u] = i + u < cnt ? row + bx : -1;
            if (++bx > bx1) { bx = bx0; row += nb; }
            grp[u] = __match_any_sync(0xffffffffu, key[u]);
            base[u] = room[u] = off[u] = 0;
            if (key[u] >= 0) {
                if (lane == __ffs(grp[u]) - 1) base[u] = atomicAdd(cursor + key[u], __popc(grp[u]));
                room[u] = eff[key[u]];
                off[u] = offsets[key[u]];
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int slot = __shfl_sync(0xffffffffu, base[u], __ffs(grp[u]) - 1) + __popc(grp[u] & lt);
            if (key[u] >= 0 && slot < room[u]) lists[off[u] + slot] = entry;
        }
    }
}

// Bitonic sort of N2 = BD * E entries, E consecutive entries per thread in
// registers: stages whose partner is in the same thread (distance < E) run in
// registers, stages whose partner is in the same warp (distance < 32 E) go
// through lane shuffles, and only the few wider ones through shared memory
// (two barriers each).  Padding entries (all ones) sort last.
template <int E, int J>
__device__ __forceinline__ void sort_stage_local(unsigned long long (&v)[E], int k2, int tid) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
        if (e & J) continue;
        const int i = tid * E + e;
        const unsigned long long x = v[e], y = v[e + J];
        const bool asc = (i & k2) == 0;
        const unsigned long long lo = x < y ? x : y, hi = x < y ? y : x;
        v[e] = asc ? lo : hi;
        v[e + J] = asc ? hi : lo;
    }
}

// From k_first = N2: only the last merge, of a sequence that is bitonic already.
template <int BD, int E>
__device__ __forceinline__ void sort_entries_regs(unsigned long long *s_sort, const unsigned long long *src, int m,
                                                  int k_first = 2) {
    constexpr int N2 = BD * E;
    const int tid = threadIdx.x;
    unsigned long long v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = tid * E + e;
        v[e] = i < m ? src[i] : ~0ull;
    }
#pragma unroll 1
    for (int k2 = k_first; k2 <= N2; k2 <<= 1) {
#pragma unroll 1
        for (int j2 = k2 >> 1; j2 > 0; j2 >>= 1) {
            if (j2 < E) {
                if constexpr (E > 4) { if (j2 == 4) { sort_stage_local<E, (E > 4 ? 4 : 1)>(v, k2, tid); continue; } }
                if constexpr (E > 2) { if (j2 == 2) { sort_stage_local<E, (E > 2 ? 2 : 1)>(v, k2, tid); continue; } }
                sort_stage_local<E, 1>(v, k2, tid);
                continue;
            }
            if (j2 < 32 * E) {
                const int lm = j2 / E;  // partner lane distance
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int i = tid * E + e;
                    const unsigned long long o = __shfl_xor_sync(0xffffffffu, v[e], lm);
                    const bool keep_min = ((i & j2) == 0) == ((i & k2) == 0);
                    v[e] = keep_min ? (o < v[e] ? o : v[e]) : (o > v[e] ? o : v[e]);
                }
                continue;
            }
            // (entries e of the threads side by side: no bank conflicts)
#pragma unroll
            for (int e = 0; e < E; ++e) s_sort[e * BD + tid] = v[e];
            __syncthreads();
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int i = tid * E + e;
                const unsigned long long o = s_sort[e * BD + (tid ^ (j2 / E))];
                const bool keep_min = ((i & j2) == 0) == ((i & k2) == 0);
                v[e] = keep_min ? (o < v[e] ? o : v[e]) : (o > v[e] ? o : v[e]);
            }
            __syncthreads();
        }
    }
#pragma unroll
    for (int e = 0; e < E; ++e) s_sort[tid * E + e] = v[e];
    __syncthreads();
}

// Bitonic sort of n2 (a power of two) entries in shared memory.
template <int BD>
__device__ __forceinline__ void bitonic_shared(unsigned long long *s_sort, int n2) {
    const int tid = threadIdx.x;
#pragma unroll 1
    for (int k2 = 2; k2 <= n2; k2 <<= 1) {
#pragma unroll 1
        for (int j2 = k2 >> 1; j2 > 0; j2 >>= 1) {
            for (int i = tid; i < (n2 >> 1); i += BD) {
                const int lo = ((i & ~(j2 - 1)) << 1) | (i & (j2 - 1));
                const int hi = lo + j2;
                const unsigned long long x = s_sort[lo], y = s_sort[hi];
                if ((x > y) == ((lo & k2) == 0)) {
                    s_sort[lo] = y;
                    s_sort[hi] = x;
                }
            }
            __syncthreads();
        }
    }
}

// Sorts m <= sort-buffer bin entries (64-bit keys) from src into s_sort,
// ascending; every thread of the block (BD threads) must call it.  A segment
// that fits one entry per thread sorts in registers: partners closer than 32
// trade through shuffles, farther ones through shared memory.  Up to eight per
// thread sort likewise, larger ones in shared memory.  Padding entries (all ones) sort last.
template <int BD>
__device__ __forceinline__ void sort_entries(unsigned long long *s_sort, const unsigned long long *src, int m) {
    const int tid = threadIdx.x;
    int n2 = 32;
    while (n2 < m) n2 <<= 1;
    if (n2 <= BD) {
        // one entry per thread: partners closer than 32 trade through
        // shuffles, farther ones through shared memory
        unsigned long long v = tid < m ? src[tid] : ~0ull;
#pragma unroll 1
        for (int k2 = 2; k2 <= n2; k2 <<= 1) {
#pragma unroll 1
            for (int j2 = k2 >> 1; j2 > 0; j2 >>= 1) {
                unsigned long long o;
                if (j2 >= 32) {
                    s_sort[tid] = v;
                    __syncthreads();
                    o = s_sort[tid ^ j2];
                    __syncthreads();
                } else {
                    o = __shfl_xor_sync(0xffffffffu, v, j2);
                }
                const bool keep_min = ((tid & j2) == 0) == ((tid & k2) == 0);
                v = keep_min ? (o < v ? o : v) : (o > v ? o : v);
            }
        }
        s_sort[tid] = v;
        __syncthreads();
        return;
    }
    // two to eight entries per thread in registers and shuffles (far fewer barriers)
    if (n2 == 2 * BD) { sort_entries_regs<BD, 2>(s_sort, src, m); return; }
    if (n2 == 4 * BD) { sort_entries_regs<BD, 4>(s_sort, src, m); return; }
    if (n2 == 8 * BD) { sort_entries_regs<BD, 8>(s_sort, src, m); return; }
    for (int i = tid; i < n2; i += BD) s_sort[i] = i < m ? src[i] : ~0ull;
    __syncthreads();
    bitonic_shared<BD>(s_sort, n2);
}

// ---------------------------------------------------------------------------
// A bin's list in front-to-back windows, for the fine passes.
//
// What a fine pass keeps (the K nearest by depth and id) does not depend on the
// order it meets the candidates in; order only buys the early stop once every
// pixel's K-th depth lies in front of what is left.  So the list is not sorted
// but dealt into 256 depth buckets (linear in the key between the bin's
// smallest and largest) and handed out in windows of consecutive buckets that
// fit WIN entries of shared memory: one pass for the range, one for the
// counts, one per window to fetch its entries, about six barriers for a bin of
// up to WIN entries where a bitonic sort of 1,024 takes 55 exchange stages.
// A bucket that does not fit is dealt into 256 buckets of its own; what does
// not fit then (entries at nearly one depth) is handed out in pieces of the
// list, in whatever order it has.
//
// The bucket of a key is monotone in the key (a rounded subtraction, a rounded
// product, a truncation), so if bucket(x) < bucket(key), then x < key: comparing
// the bucket of a pixel's K-th depth with a window's buckets decides, without
// knowing any window's smallest key, that everything from there on is behind.
// ---------------------------------------------------------------------------
//
// Every window reads the whole list for its entries.  Where few lists are long, they
// are sorted in place before the fine pass (sort_long.cu) and handed out as they lie:
// 1.6M points on 16 px, K = 1, bins of 8: dealt 307 ms, sorted 7.0; 200,000 on 64 px, bins
// of 16: 1,696 us, 386; 1.3M faces on 16 px, K = 8, soft, bins of 8: 378 ms, 40.0; on 64 px,
// hard, bins of 16: 29.9, 14.7.  Where many are, they fill the GPU as they are and most
// stop after a few windows: 1.3M faces on 1,024 px (1,600 lists of 8,000 to 20,000), K = 8:
// 972 us dealt, 1,764 with all of them sorted.  The line: some list has more than 16,384
// entries and a 64th of all bins' entries; then all of half that length are sorted, so
// that the pass does not wait for those just below.  (With T / 48: 4 meshes of 328k faces
// on 48 px, K = 8, bins of 8: 4,726 us against 3,688; with 24,576: 2 of them on 64 px, K = 1,
// bins of 16: 2,140 against 1,928, dealt 1,818.)
constexpr int kBuckets = 256;

struct KeyMap {
    float lo, scale;
    // NaN (0 x inf) converts to 0, values past the int range saturate
    __device__ __forceinline__ int operator()(float key) const {
        return min(kBuckets - 1, __float2int_rz(__fmul_rn(__fsub_rn(key, lo), scale)));
    }
};

__device__ __forceinline__ float entry_key(unsigned long long e) { return __uint_as_float((unsigned)(e >> 32)); }

// Keys of either sign (points where znear is below 0) are kept in the order of
// their values: the sign bit set on positive ones, all bits turned on negative.
__device__ __forceinline__ unsigned signed_key_bits(float z) {
    const unsigned u = __float_as_uint(z);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
template <bool SIGNED>
__device__ __forceinline__ float key_of_bits(unsigned u) {
    if (SIGNED) u = (u & 0x80000000u) ? (u ^ 0x80000000u) : ~u;
    return __uint_as_float(u);
}

// Where a block is in its bin's list; the same in every thread.
struct WindowState {
    const unsigned long long *list;
    int cnt;
    KeyMap map[2];
    int b0, b1;      // next bucket of level 0; of level 1 while `deep`
    int seg;         // >= 0: next piece of the list (as it lies, or a level-1 bucket that does not fit)
    int deep, plain;
    int ascending;   // plain, and the list is sorted
    int sorted;      // level whose buckets order the current window, -1: none
    int base;        // entries of that level in front of the current window
};

template <int WIN, bool SIGNED = false>
struct WindowShared {
    static __device__ __forceinline__ float key(unsigned long long e) {
        return key_of_bits<SIGNED>((unsigned)(e >> 32));
    }
    unsigned long long ent[WIN];      // the current window
    int pre[2][kBuckets + 1];         // entries before each bucket, per level
    int cur[kBuckets];
    int wsum[8];
    unsigned lo, hi;
    int n;
    WindowState st;

    // bucket that orders the current window (constant when nothing does)
    __device__ __forceinline__ int rank(float key) const { return st.sorted < 0 ? 0 : st.map[st.sorted](key); }

    // whether the key and all that follow it in the current window lie behind depth z
    __device__ __forceinline__ bool behind(float key, float z) const {
        return st.ascending ? z < key : rank(z) < rank(key);
    }

    // whether every entry not yet handed out lies behind depth z
    __device__ __forceinline__ bool rest_behind(float z) const {
        if (st.plain) return st.ascending && (st.seg >= st.cnt || z < WindowShared::key(__ldg(st.list + st.seg)));
        const int k = st.map[0](z);
        return k < st.b0 || (st.deep && k == st.b0 && st.map[1](z) < st.b1);
    }
};

template <int BD, int WIN, bool SIGNED>
struct WindowLoader : WindowState {
    using Shared = WindowShared<WIN, SIGNED>;
    Shared &s;
    __device__ __forceinline__ WindowLoader(Shared &sh) : WindowState(sh.st), s(sh) {}

    __device__ __forceinline__ bool mine(float key, int level) const { return level == 0 || map[0](key) == b0; }

    // f on every entry of the list, several loads in flight per thread (one at a
    // time, 64 threads wait for 128 round trips to L2 on a list of 8,192)
    template <class F>
    __device__ __forceinline__ void for_list(const F &f) const {
        constexpr int U = WIN / BD < 4 ? 4 : WIN / BD;
        for (int i = threadIdx.x; i < cnt; i += U * BD) {
            unsigned long long e[U];
#pragma unroll
            for (int u = 0; u < U; ++u) e[u] = i + u * BD < cnt ? __ldg(list + i + u * BD) : 0ull;
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i + u * BD < cnt) f(e[u]);
        }
    }

    // ranges and counts of the buckets of a level
    template <int level>
    __device__ __forceinline__ void deal() {
        const int tid = threadIdx.x;
        __syncthreads();
        if (tid == 0) { s.lo = 0xffffffffu; s.hi = 0u; }
        for (int b = tid; b < kBuckets; b += BD) s.cur[b] = 0;
        __syncthreads();
        unsigned lo = 0xffffffffu, hi = 0u;  // the bits order like the values
        for_list([&](unsigned long long e) {
            if (!mine(Shared::key(e), level)) return;
            lo = min(lo, (unsigned)(e >> 32));
            hi = max(hi, (unsigned)(e >> 32));
        });
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if ((tid & 31) == 0) { atomicMin(&s.lo, lo); atomicMax(&s.hi, hi); }
        __syncthreads();
        KeyMap m;
        m.lo = key_of_bits<SIGNED>(s.lo);
        const float d = key_of_bits<SIGNED>(s.hi) - m.lo;
        m.scale = d > 0.f ? __fdiv_rn((float)kBuckets, d) : 0.f;
        map[level] = m;
        for_list([&](unsigned long long e) {
            const float key = Shared::key(e);
            if (mine(key, level)) atomicAdd(&s.cur[m(key)], 1);
        });
        __syncthreads();
        // exclusive prefix of the counts: kBuckets / BD consecutive buckets per thread
        constexpr int E = kBuckets / BD;
        int v[E], sum = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) { v[e] = s.cur[tid * E + e]; sum += v[e]; }
        int x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if ((tid & 31) >= o) x += y;
        }
        if ((tid & 31) == 31) s.wsum[tid >> 5] = x;
        __syncthreads();
        int base = x - sum;
        for (int w = 0; w < (tid >> 5); ++w) base += s.wsum[w];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            s.pre[level][tid * E + e] = base;
            base += v[e];
        }
        if (tid == BD - 1) s.pre[level][kBuckets] = base;
        for (int b = tid; b < kBuckets; b += BD) s.cur[b] = 0;
        __syncthreads();
    }

    // one past the last bucket of the longest run from b that fits WIN entries
    __device__ __forceinline__ int run_end(int level, int b) const {
        const int *p = s.pre[level];
        const int lim = p[b] + WIN;
        int lo = b, hi = kBuckets;  // p[lo] <= lim
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (p[mid] <= lim) lo = mid;
            else hi = mid - 1;
        }
        return lo;
    }

    // entries of buckets [b, e) of a level, in bucket order
    template <int level>
    __device__ __forceinline__ int fetch(int b, int e) {
        const int n = s.pre[level][e] - s.pre[level][b];
        if (n > 0) {
            const KeyMap m = map[level];
            for_list([&](unsigned long long v) {
                const float key = Shared::key(v);
                if (!mine(key, level)) return;
                const int k = m(key);
                if (k < b || k >= e) return;
                s.ent[s.pre[level][k] - s.pre[level][b] + atomicAdd(&s.cur[k], 1)] = v;
            });
            __syncthreads();
        }
        sorted = level;
        base = s.pre[level][b];
        return n;
    }

    // the next window's size; 0 at the end
    __device__ __forceinline__ int next() {
        while (cnt > 0) {
            if (plain) {
                const int m = min(WIN, cnt - seg);
                if (m <= 0) return 0;
                for (int i = threadIdx.x; i < m; i += BD) s.ent[i] = __ldg(list + seg + i);
                seg += m;
                __syncthreads();
                return m;
            }
            if (seg >= 0) {
                if (seg >= cnt) { seg = -1; ++b1; continue; }
                if (threadIdx.x == 0) s.n = 0;
                __syncthreads();
                const int m = min(WIN, cnt - seg);
                for (int i = threadIdx.x; i < m; i += BD) {
                    const unsigned long long v = __ldg(list + seg + i);
                    const float key = Shared::key(v);
                    if (map[0](key) == b0 && map[1](key) == b1) s.ent[atomicAdd(&s.n, 1)] = v;
                }
                seg += m;
                sorted = -1;
                __syncthreads();
                const int n = s.n;
                __syncthreads();  // s.n is reset by the next piece
                if (n == 0) continue;
                return n;
            }
            if (deep) {
                if (b1 >= kBuckets) {
                    deep = false;
                    ++b0;
                    for (int b = threadIdx.x; b < kBuckets; b += BD) s.cur[b] = 0;
                    __syncthreads();
                    continue;
                }
                const int e = run_end(1, b1);
                if (e == b1) { seg = 0; continue; }
                const int n = fetch<1>(b1, e);
                b1 = e;
                if (n > 0) return n;
                continue;
            }
            if (b0 >= kBuckets) return 0;
            const int e = run_end(0, b0);
            if (e == b0) { deal<1>(); deep = true; b1 = 0; continue; }
            const int n = fetch<0>(b0, e);
            b0 = e;
            if (n > 0) return n;
        }
        return 0;
    }
};

// Starts on a list; `ordered` false hands it out as it is, `ascending` says that
// it is sorted.  Every thread of the block calls this and window_next.
template <int BD, int WIN, bool SIGNED>
__device__ __forceinline__ void window_begin(WindowShared<WIN, SIGNED> &s, const unsigned long long *list, int cnt,
                                             bool ordered, bool ascending) {
    ordered = ordered && !ascending;
    __syncthreads();
    if (threadIdx.x == 0) {
        s.st.list = list;
        s.st.cnt = cnt;
        s.st.b0 = ordered ? -1 : 0;
        s.st.b1 = 0;
        s.st.seg = ordered ? -1 : 0;
        s.st.deep = 0;
        s.st.plain = !ordered;
        s.st.ascending = ascending;
        s.st.sorted = -1;
        s.st.base = 0;
    }
    __syncthreads();
}

// Loads the next window into s.ent and returns its size; 0 at the end.  Every
// thread must be done with the last window.  Not inlined: the walk between two
// windows keeps its registers.
template <int BD, int WIN, bool SIGNED>
static __device__ __noinline__ int window_next(WindowShared<WIN, SIGNED> &s) {
    WindowLoader<BD, WIN, SIGNED> w(s);
    if (w.cnt <= 0) return 0;
    if (w.b0 < 0) {
        w.template deal<0>();
        w.b0 = 0;
    }
    const int n = w.next();
    __syncthreads();
    if (threadIdx.x == 0) s.st = w;
    __syncthreads();
    return n;
}

// large-K variant: per-thread sorted lists in shared memory; element k of a
// thread's list sits at z[k * stride], f[k * stride]
struct SmemTopK {
    float *z;
    int *f;
    int stride, K;
    int n;  // entries held (< K while the list is not full)
    __device__ __forceinline__ void init() { n = 0; }
    // K-th smallest depth so far (infinite until K candidates were kept)
    __device__ __forceinline__ float thr() const {
        return n < K ? __int_as_float(0x7f800000) : z[(K - 1) * stride];
    }
    __device__ __forceinline__ bool admits(float zz, int ff) const {
        return n < K || key_less(zz, ff, z[(K - 1) * stride], f[(K - 1) * stride]);
    }
    // insertion from the end of the held entries: candidates arrive nearly in
    // depth order, so most insertions are appends
    __device__ __forceinline__ void insert(float zz, int ff) {
        int k = n < K ? n : K - 1;
        while (k > 0) {
            float zp = z[(k - 1) * stride];
            int fp = f[(k - 1) * stride];
            if (!key_less(zz, ff, zp, fp)) break;
            z[k * stride] = zp;
            f[k * stride] = fp;
            --k;
        }
        z[k * stride] = zz;
        f[k * stride] = ff;
        if (n < K) ++n;
    }
};

}  // namespace mr
