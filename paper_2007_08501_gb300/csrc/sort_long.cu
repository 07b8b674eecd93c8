// Long bin lists put in order before the fine pass (sm_103a).
//
// A fine pass fetches its windows from the list it has, so a list of n entries
// that no early stop shortens costs it n^2 / window loads.  Lists beyond
// long_list entries are therefore sorted in place first: runs of 8,192, each by
// a block of its own, in registers and shared memory; then one block per list
// merges them in global memory (L2) down to runs, the rest of each merge in
// shared memory again.  The network sorts ascending throughout (each merge
// starts by comparing mirrored places), so the places past the list's end,
// thought of as holding the largest entry, need neither storage nor padding.
// Bound by the latency of one block's loads; n log^2 n, where what it replaces
// grew as n^2 (figures in bin_common.cuh).
#include <cuda_runtime.h>

#include <cstdint>

#include "bin_common.cuh"
#include "rast_common.cuh"
#include "rast_internal.h"

namespace mr {

constexpr int kSortThreads = 1024, kSortEach = 8, kSortRun = kSortThreads * kSortEach;

// One stage over the whole list: pair p's lower place and its partner from
// `place`; four pairs' loads in flight per thread.
template <class Place>
__device__ __forceinline__ void sort_stage_global(unsigned long long *list, unsigned n, unsigned pairs,
                                                  const Place &place) {
    constexpr int U = 4;
    for (unsigned base = threadIdx.x; base < pairs; base += U * kSortThreads) {
        unsigned i[U], j[U];
        unsigned long long x[U], y[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            i[u] = j[u] = n;
            if (base + u * kSortThreads < pairs) place(base + u * kSortThreads, i[u], j[u]);
            if (j[u] < n) {
                x[u] = list[i[u]];
                y[u] = list[j[u]];
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (j[u] < n && x[u] > y[u]) {
                list[i[u]] = y[u];
                list[j[u]] = x[u];
            }
    }
    __syncthreads();
}

// Run `at` of the list, kSortRun entries: sorted from any order, or (merge) from
// the order the wider stages leave.
__device__ __forceinline__ void sort_run(unsigned long long *s_sort, unsigned long long *list, unsigned n, unsigned at,
                                         bool merge) {
    const int m = (int)min(n - at, (unsigned)kSortRun);
    sort_entries_regs<kSortThreads, kSortEach>(s_sort, list + at, m, merge ? kSortRun : 2);
    for (int i = threadIdx.x; i < m; i += kSortThreads) list[at + i] = s_sort[i];
    __syncthreads();
}

// f(list, entries) on the long lists of block column blockIdx.x, whose bins lie
// gridDim.x apart (long lists are neighbours).
template <class F>
__device__ __forceinline__ void for_long(const SortLongArgs &a, const F &f) {
    __shared__ int s_bins[kSortThreads];
    __shared__ int s_n;
    const int from = long_list(*a.total);
    if (*a.maxcount <= from) return;
    for (int64_t base = blockIdx.x; base < a.items; base += (int64_t)gridDim.x * kSortThreads) {
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        const int64_t b = base + (int64_t)threadIdx.x * gridDim.x;
        if (b < a.items && a.eff[b] > from) s_bins[atomicAdd(&s_n, 1)] = (int)b;
        __syncthreads();
        for (int q = 0; q < s_n; ++q) f(a.lists + a.offsets[s_bins[q]], (unsigned)a.eff[s_bins[q]]);
        __syncthreads();
    }
}

// the runs of a list shared out over gridDim.y blocks
__global__ void __launch_bounds__(kSortThreads) k_sort_runs(SortLongArgs a) {
    extern __shared__ unsigned long long s_sort[];  // kSortRun
    for_long(a, [&](unsigned long long *list, unsigned n) {
        for (unsigned at = blockIdx.y * kSortRun; at < n; at += gridDim.y * kSortRun) sort_run(s_sort, list, n, at, false);
    });
}

__global__ void __launch_bounds__(kSortThreads) k_merge_runs(SortLongArgs a) {
    extern __shared__ unsigned long long s_sort[];
    for_long(a, [&](unsigned long long *list, unsigned n) {
        for (uint64_t width = 2 * kSortRun; (width >> 1) < n; width <<= 1) {  // (n < 2^31)
            const unsigned k = (unsigned)width, half = k >> 1;
            const int lg = 31 - __clz((int)half);
            const unsigned pairs = ((n + k - 1) / k) << lg;
            sort_stage_global(list, n, pairs, [&](unsigned p, unsigned &i, unsigned &j) {
                const unsigned start = (p >> lg) * k, off = p & (half - 1);
                i = start + off;
                j = start + k - 1 - off;
            });
            for (unsigned d = half >> 1; d >= (unsigned)kSortRun; d >>= 1)
                sort_stage_global(list, n, pairs, [&](unsigned p, unsigned &i, unsigned &j) {
                    i = ((p & ~(d - 1)) << 1) | (p & (d - 1));
                    j = i + d;
                });
            for (unsigned at = 0; at < n; at += kSortRun) sort_run(s_sort, list, n, at, true);
        }
    });
}

cudaError_t launch_sort_long(const SortLongArgs &a, cudaStream_t st) {
    const size_t dyn = (size_t)kSortRun * sizeof(unsigned long long);  // 64 KB
    cudaError_t e = cudaFuncSetAttribute(k_sort_runs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_merge_runs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    if (e != cudaSuccess) return e;
    const int lists = (int)(a.items < 64 ? a.items : 64);  // (fewer than 64 are long)
    k_sort_runs<<<dim3((unsigned)lists, 8), kSortThreads, dyn, st>>>(a);
    k_merge_runs<<<lists, kSortThreads, dyn, st>>>(a);
    return cudaGetLastError();
}

}  // namespace mr
