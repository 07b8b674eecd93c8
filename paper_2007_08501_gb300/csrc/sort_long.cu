// Long bin lists put in order before the fine pass (sm_103a).
//
// A fine pass fetches its windows from the list it has, so a list of n entries
// that no early stop shortens costs it n^2 / window loads.  Long lists are
// therefore sorted in place first (k_scan finds them): runs of 8,192, each by a
// block, in registers and shared memory; then one block per list merges in global
// memory (L2) down to runs, the rest of each merge in shared memory again.  The
// network sorts ascending throughout (each merge starts by comparing mirrored
// places), so the places past the list's end, thought of as holding the largest
// entry, need neither storage nor padding.
// Bound by the latency of one block's loads; n log^2 n, where what it replaces
// grew as n^2 (figures in bin_common.cuh).
#include <cuda_runtime.h>

#include <cstdint>

#include "bin_common.cuh"
#include "rast_common.cuh"
#include "rast_internal.h"

namespace mr {

constexpr int kSortThreads = 1024, kSortEach = 8, kSortRun = kSortThreads * kSortEach;
__device__ __forceinline__ unsigned sort_runs(unsigned n) { return (n + kSortRun - 1) / kSortRun; }

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

// A list's runs in one, by one block.
__device__ __forceinline__ void merge_runs(unsigned long long *s_sort, unsigned long long *list, unsigned n) {
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
}

// The runs of all long lists are shared out over the blocks; a block that has no
// runs left merges lists whose runs are all sorted until it sees none.  No block
// waits for another: who ends a list's last run looks for lists after that.  One
// launch, because most calls that could have long lists have none: 1.3M faces on
// 1,024 px, K = 8: 973 us without, 978 with it, 983 with two.
__global__ void __launch_bounds__(kSortThreads) k_sort_long(SortLongArgs a) {
    extern __shared__ unsigned long long s_sort[];  // kSortRun
    __shared__ int s_pick;
    const unsigned lists = *a.n;
    constexpr unsigned kTaken = 0xffffffffu;
    for (unsigned q = 0, turn = blockIdx.x; q < lists; ++q) {  // turn: the block's next run, counted from list q
        const int bin = a.long_bins[q].bin;
        const unsigned n = (unsigned)a.eff[bin], runs = sort_runs(n);
        for (; turn < runs; turn += gridDim.x) {
            sort_run(s_sort, a.lists + a.offsets[bin], n, turn * kSortRun, false);
            if (threadIdx.x == 0) {
                __threadfence();
                atomicAdd(&a.long_bins[q].runs, 1u);
            }
        }
        turn -= runs;
    }
    while (lists) {  // (every turn takes a list, loses one to another block or is the last)
        if (threadIdx.x == 0) s_pick = kMaxLong;
        __syncthreads();
        if (threadIdx.x < lists) {  // each block looks from a list of its own on
            const unsigned q = (threadIdx.x + blockIdx.x) % lists;
            const LongBin *const l = a.long_bins + q;
            if (*(const volatile unsigned *)&l->runs == sort_runs((unsigned)a.eff[l->bin]))
                atomicMin(&s_pick, (int)threadIdx.x);
        }
        __syncthreads();
        const unsigned pick = (unsigned)s_pick;
        __syncthreads();
        if (pick == kMaxLong) break;
        LongBin *const l = a.long_bins + (pick + blockIdx.x) % lists;
        const unsigned n = (unsigned)a.eff[l->bin], runs = sort_runs(n);
        if (threadIdx.x == 0) s_pick = atomicCAS(&l->runs, runs, kTaken) == runs;
        __syncthreads();
        const bool mine = s_pick != 0;
        __threadfence();
        __syncthreads();
        if (mine) merge_runs(s_sort, a.lists + a.offsets[l->bin], n);
    }
}

cudaError_t launch_sort_long(const SortLongArgs &a, cudaStream_t st) {
    const size_t dyn = (size_t)kSortRun * sizeof(unsigned long long);  // 64 KB
    const cudaError_t e = cudaFuncSetAttribute(k_sort_long, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    if (e != cudaSuccess) return e;
    k_sort_long<<<mr_host::num_sms(), kSortThreads, dyn, st>>>(a);
    return cudaGetLastError();
}

}  // namespace mr
