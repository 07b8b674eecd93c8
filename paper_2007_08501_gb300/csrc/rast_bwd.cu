// Backward rasterization for sm_103a.
//
// Section 3.2 of the paper: the backward pass reuses the Fragment data (the
// face id of each slot) instead of recomputing face-pixel intersections.  For
// every non-empty slot this kernel recomputes the fragment of that face at
// that pixel from the staged face record and pulls dL/d(bary, zbuf, dists)
// back through clipping, perspective correction, the edge functions and the
// nearest-segment distance to the three NDC corners, then through the
// projection Jacobian and R^T to world-space vertices (atomic scatter).
#include <cuda_runtime.h>

#include "rast_common.cuh"
#include "rast_internal.h"
#include "rast_adjoint.cuh"
#include "tile_sort.cuh"

namespace mr {

// One block = a 16 x 16 pixel tile of one image, kTileSlots slots per pixel at
// a time, by face over the tile (tile_sort.cuh).  Bound by instructions (the
// adjoint itself, ~700 per slot).  8 meshes of 5,120 faces, 256 px, K = 8: 110 -> 105
// us.
__global__ void __launch_bounds__(256) k_rast_bwd(RastBwdArgs a) {
    const int n = blockIdx.z;
    int tx, ty;
    tile_xy(threadIdx.x, tx, ty);
    const int row = blockIdx.y * 16 + ty, col = blockIdx.x * 16 + tx;
    const int64_t s0 = row < a.S && col < a.S ? (((int64_t)n * a.S + row) * a.S + col) * a.K : -1;
    __shared__ TileSort s_sorted;
    __shared__ RareSlot s_rare[kRareCap];
    __shared__ int s_nrare;
    if (threadIdx.x == 0) s_nrare = 0;
    const RareQueue rq{s_rare, &s_nrare};
    const bool pairs = ((uintptr_t)a.grad_verts & 7u) == 0;
    for (int kb = 0; kb < a.K; kb += kTileSlots) {
        const int cnt = tile_sort(s_sorted, [&](int k) {
            const int64_t f = s0 >= 0 && kb + k < a.K ? __ldg(a.pix_to_face + s0 + kb + k) : -1;
            return f >= 0 && f < a.F ? (int)f : -1;  // an id outside the batch contributes nothing
        });
        for (int i = threadIdx.x; i < ((cnt + 31) & ~31); i += 256) {
            int key = -1, nf = -1;
            float g[9];
#pragma unroll
            for (int j = 0; j < 9; ++j) g[j] = 0.f;
            FaceRec R;
            if (i < cnt) {
                const int e = s_sorted.order[i];
                int px, py;
                tile_xy(e & 255, px, py);
                const int r = blockIdx.y * 16 + py, c = blockIdx.x * 16 + px;
                const int64_t s = (((int64_t)n * a.S + r) * a.S + c) * a.K + kb + (e >> 8);
                const int f = (int)__ldg(a.pix_to_face + s);
                nf = __ldg(a.face_mesh + f);
                const float gz = a.grad_zbuf ? __ldg(a.grad_zbuf + s) : 0.f;
                const float gd = a.grad_dists ? __ldg(a.grad_dists + s) : 0.f;
                float gb0 = 0.f, gb1 = 0.f, gb2 = 0.f;
                if (a.grad_bary) {
                    gb0 = __ldg(a.grad_bary + 3 * s);
                    gb1 = __ldg(a.grad_bary + 3 * s + 1);
                    gb2 = __ldg(a.grad_bary + 3 * s + 2);
                }
                if (nf >= 0 && (gz != 0.f || gd != 0.f || gb0 != 0.f || gb1 != 0.f || gb2 != 0.f)) {
                    key = f;
                    const float4 *src = reinterpret_cast<const float4 *>(a.rec + f);
                    R.a = __ldg(src + kRecA);
                    R.b = __ldg(src + kRecB);
                    R.d = __ldg(src + kRecD);
                    R.e = __ldg(src + kRecE);
                    slot_corner_grads(R, pixel_centre(r, c, a.S), a.fl, gz, gd, gb0, gb1, gb2, g, rq, f, nf,
                                      (py << 4) | px);
                }
            }
            if (run_sum<9>(key, g) && key >= 0)
                scatter_corner_grads(R, a.cams + 16 * nf, a.faces, key, g, a.grad_verts, pairs);
        }
        __syncthreads();
    }
    flush_rare_slots(rq, a.rec, a.cams, a.faces, a.grad_verts, a.S, a.fl);
}

cudaError_t launch_rast_bwd(const RastBwdArgs &a, int N, cudaStream_t st) {
    if (a.slots <= 0 || N <= 0) return cudaSuccess;
    const unsigned tiles = (unsigned)((a.S + 15) / 16);
    k_rast_bwd<<<dim3(tiles, tiles, (unsigned)N), 256, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace mr
