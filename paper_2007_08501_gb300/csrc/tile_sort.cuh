// A tile's slots brought together by face, for the backward kernels that
// scatter per-slot gradients to vertices.
//
// Neighbouring pixels hold a face at different ranks, so at any one rank few of
// a warp's 32 pixels share one: grouping them there (match, a tree of shuffles
// over up to 27 sums, one lane per face adding) runs at three to four lanes per
// group and a round trip per group.  Here the up to 8 slots of the block's 256
// pixels are dealt into 1,024 buckets by a hash of the face (a counting sort in
// shared memory, ~30 instructions per slot); consecutive lanes then hold slots
// of one face, records and vertices come as broadcasts, empty slots take no
// lane, and a segmented sum leaves one addition per face and warp.
#pragma once

#include <cstddef>

#include "rast_common.cuh"

namespace mr {

constexpr int kTileSlots = 8;  // slots per pixel dealt at a time
constexpr int kTileBuckets = 1024;

struct __align__(16) TileSort {  // (start is read four at a time)
    unsigned short order[kTileSlots * 256];  // slot << 8 | thread whose pixel it is
    int start[kTileBuckets];
    int wsum[8];
    int n;
};
static_assert(offsetof(TileSort, start) % 16 == 0 && alignof(TileSort) == 16, "int4 loads of start");

// key(k) for k < kTileSlots: the face of slot k of this thread's pixel, -1 for
// none.  Returns the number of slots in s.order.  Blocks of 256 threads; every
// thread calls it, and again only after a barrier.
template <class Key>
__device__ __forceinline__ int tile_sort(TileSort &s, const Key &key) {
    const int tid = threadIdx.x, lane = tid & 31;
    reinterpret_cast<int4 *>(s.start)[tid] = make_int4(0, 0, 0, 0);
    __syncthreads();
    int at[kTileSlots];
#pragma unroll
    for (int k = 0; k < kTileSlots; ++k) {
        const int f = key(k);
        at[k] = -1;
        if (f >= 0) {
            const unsigned b = ((unsigned)f * 2654435761u) >> 22;
            at[k] = (int)(b << 16) | atomicAdd(&s.start[b], 1);  // at most 2,048 in a bucket
        }
    }
    __syncthreads();
    const int4 v = reinterpret_cast<int4 *>(s.start)[tid];
    const int sum = v.x + v.y + v.z + v.w;
    int x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s.wsum[tid >> 5] = x;
    __syncthreads();
    int base = x - sum;
    for (int w = 0; w < (tid >> 5); ++w) base += s.wsum[w];
    reinterpret_cast<int4 *>(s.start)[tid] = make_int4(base, base + v.x, base + v.x + v.y, base + v.x + v.y + v.z);
    if (tid == 255) s.n = base + sum;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kTileSlots; ++k)
        if (at[k] >= 0) s.order[s.start[at[k] >> 16] + (at[k] & 0xffff)] = (unsigned short)(k << 8 | tid);
    __syncthreads();
    return s.n;
}

// Pixel of thread t in a 16 x 16 tile: each warp covers an 8 x 4 block.
__device__ __forceinline__ void tile_xy(int t, int &tx, int &ty) {
    tx = ((t >> 5) & 1) * 8 + (t & 7);
    ty = (t >> 6) * 4 + ((t >> 3) & 3);
}

// Sums of x over runs of lanes with equal keys, left in each run's first lane;
// returns whether this lane is one.  Every lane of the warp calls it.
template <int NV>
__device__ __forceinline__ bool run_sum(int key, float (&x)[NV]) {
    const int lane = threadIdx.x & 31;
    const int prev = __shfl_up_sync(0xffffffffu, key, 1);
    const bool head = lane == 0 || prev != key;
    const unsigned rest = __ballot_sync(0xffffffffu, head) & ~((2u << lane) - 1u);
    const int last = rest ? __ffs(rest) - 2 : 31;
    const int longest = __reduce_max_sync(0xffffffffu, head ? last - lane + 1 : 0);
    for (int o = 1; o < longest; o <<= 1) {
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            const float t = __shfl_down_sync(0xffffffffu, x[j], o);
            if (lane + o <= last) x[j] += t;
        }
    }
    return head;
}

}  // namespace mr
