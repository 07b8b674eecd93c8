// Tiles of a batch of query clouds: one launch covers a heterogeneous batch
// without a host round trip.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace mr {

// Exclusive prefix over the clouds of ceil(len / per) into tiles (N + 1 words,
// the last one the total).  One block of BD threads.
template <int BD>
__device__ __forceinline__ void plan_tiles(const int64_t *len, int N, int per, long long *tiles) {
    __shared__ long long s_warp[BD / 32];
    __shared__ long long s_carry;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int base = 0; base < N; base += BD) {
        const int i = base + threadIdx.x;
        long long v = 0;
        if (i < N) {
            const long long n = len[i];
            v = n > 0 ? (n + per - 1) / per : 0;
        }
        long long x = v;   // inclusive scan within the warp
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[w] = x;
        __syncthreads();
        if (w == 0) {
            long long t = lane < BD / 32 ? s_warp[lane] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long y = __shfl_up_sync(0xffffffffu, t, o);
                if (lane >= o) t += y;
            }
            if (lane < BD / 32) s_warp[lane] = t;   // inclusive over warps
        }
        __syncthreads();
        const long long carry = s_carry;
        const long long before = carry + (w > 0 ? s_warp[w - 1] : 0) + x - v;
        if (i < N) tiles[i] = before;
        __syncthreads();
        if (threadIdx.x == 0) s_carry = carry + s_warp[BD / 32 - 1];
        __syncthreads();
    }
    if (threadIdx.x == 0) tiles[N] = s_carry;
}

// Cloud of tile b of that plan: the last i with tiles[i] <= b (tiles[0] = 0 <= b < tiles[N]).
__device__ __forceinline__ int planned_cloud(const long long *tiles, int N, long long b) {
    int lo = 0, hi = N;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (tiles[mid] <= b) lo = mid; else hi = mid;
    }
    return lo;
}

}  // namespace mr
