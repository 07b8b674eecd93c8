// Backward of the packed silhouette for sm_103a: dL/d(image alpha) through
// Algorithm 1 and the distance to the nearest edge to the vertices.
//
// A slot moves the x, y of its nearest edge's two corners, nothing else, so a
// slot's whole gradient is one 16-byte vector reduction into its face's
// accumulator for that edge (48 bytes per face, in L2); k_sil_gather then takes
// each face's three accumulators through the projection Jacobian and R^T once.
// Grouping the warp's lanes by face at every slot first (match, a shuffle tree
// of six sums, Jacobian and nine scalar reductions by one lane per face) costs
// several times the slot's own arithmetic: neighbouring pixels hold a face at
// different ranks, so few lanes share one.  The distance, its sign and the
// edge come with the slot; only the edge's parameter t is formed again.  Fused
// backward of 20 views, 512 px, K = 50: 4.04 -> 1.09 ms; 1.3M faces, 1024 px, K =
// 8: 113 -> 66 us.
#include <cuda_runtime.h>

#include "blend_common.cuh"
#include "rast_adjoint.cuh"
#include "rast_common.cuh"
#include "rast_internal.h"
#include "sil.cuh"

namespace mr {

__device__ __forceinline__ void red_add4(float4 *p, float x, float y, float z, float w) {
    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x), "f"(y), "f"(z), "f"(w)
                 : "memory");
}

__global__ void __launch_bounds__(256) k_sil_bwd(SilBwdArgs a) {
    // one thread per pixel; each warp covers an 8 x 4 block of the 16 x 16 tile
    const int tx = ((threadIdx.x >> 5) & 1) * 8 + (threadIdx.x & 7), ty = (threadIdx.x >> 6) * 4 + ((threadIdx.x >> 3) & 3);
    const int row = blockIdx.y * 16 + ty, col = blockIdx.x * 16 + tx;
    if (row >= a.S || col >= a.S) return;
    const int64_t pix = ((int64_t)blockIdx.z * a.S + row) * a.S + col;
    const unsigned long long *s = a.slots + pix * a.K;
    unsigned long long next = __ldg(s);
    if (next == kSilEnd) return;
    const PixC p = pixel_centre(row, col, a.S);
    const float isg = __frcp_rn(a.sigma);
    // d alpha / d d_k = -prob_k * prod_j (1 - prob_j) / sigma
    const float sil = -a.grad_image[4 * pix + 3] * a.keep[pix] / a.sigma;
    for (int k = 0; k < a.K && next != kSilEnd; ++k) {
        const unsigned long long v = next;
        if (k + 1 < a.K) next = __ldg(s + k + 1);
        const float d = __uint_as_float((unsigned)(v >> 32));
        const int f = (int)((unsigned)v & 0x3fffffffu), edge = (int)((unsigned)v >> 30);
        const float gd = sil * sigmoidf_(-d * isg);
        const float gs = signbit(d) ? -gd : gd;
        if (gs == 0.f) continue;
        const float4 *src = reinterpret_cast<const float4 *>(a.rec + f);
        FaceRec R;
        R.a = __ldg(src + kRecA);
        R.b = __ldg(src + kRecB);
        R.e = __ldg(src + kRecE);
        float qx, qy, t;
        local_q(R, p, qx, qy);
        const float ux = R.b.x, uy = R.b.y, wx = R.b.z, wy = R.b.w;
        const float ax = edge == 0 ? 0.f : edge == 1 ? ux : wx, ay = edge == 0 ? 0.f : edge == 1 ? uy : wy;
        const float ex = edge == 0 ? ux : edge == 1 ? __fsub_rn(wx, ux) : -wx;
        const float ey = edge == 0 ? uy : edge == 1 ? __fsub_rn(wy, uy) : -wy;
        (void)seg_dist2(ax, ay, ex, ey, qx, qy, t);
        float rx, ry;
        edge_residual(R, p, edge, t, rx, ry);
        const float wa = -2.f * gs * (1.f - t), wb = -2.f * gs * t;
        red_add4(a.acc + 3 * (int64_t)f + edge, wa * rx, wa * ry, wb * rx, wb * ry);
    }
}

__global__ void __launch_bounds__(256) k_sil_gather(SilBwdArgs a, int pairs) {
    const int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= a.F) return;
    const float4 e0 = __ldg(a.acc + 3 * f), e1 = __ldg(a.acc + 3 * f + 1), e2 = __ldg(a.acc + 3 * f + 2);
    const float gx[3] = {e0.x + e2.z, e0.z + e1.x, e1.z + e2.x}, gy[3] = {e0.y + e2.w, e0.w + e1.y, e1.w + e2.y};
    if (gx[0] == 0.f && gy[0] == 0.f && gx[1] == 0.f && gy[1] == 0.f && gx[2] == 0.f && gy[2] == 0.f) return;
    const int n = a.face_mesh[f];
    if (n < 0) return;
    const float4 *src = reinterpret_cast<const float4 *>(a.rec + f);
    const float4 ra = __ldg(src + kRecA), rb = __ldg(src + kRecB), rd = __ldg(src + kRecD);
    const float *cam = a.cams + 16 * n;
    const float fo = cam[12], v0x = ra.x + ra.z, v0y = ra.y + ra.w;
    const float Px[3] = {0.f, rb.x, rb.z}, Py[3] = {0.f, rb.y, rb.w}, iz[3] = {rd.y, rd.z, rd.w};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (gx[i] == 0.f && gy[i] == 0.f) continue;
        // x = f x_v / z_v, y = f y_v / z_v: d/dx_v = f/z, d/dz_v = -(x dL/dx + y dL/dy)/z
        const float xn = v0x + Px[i], yn = v0y + Py[i];
        const float gxv = gx[i] * fo * iz[i], gyv = gy[i] * fo * iz[i];
        const float gzv = -(gx[i] * xn + gy[i] * yn) * iz[i];
        const float g[3] = {cam[0] * gxv + cam[3] * gyv + cam[6] * gzv, cam[1] * gxv + cam[4] * gyv + cam[7] * gzv,
                            cam[2] * gxv + cam[5] * gyv + cam[8] * gzv};
        red_add_row<3>(a.grad_verts, __ldg(a.faces + 3 * f + i), g, pairs != 0);
    }
}

cudaError_t launch_sil_bwd(const SilBwdArgs &a, cudaStream_t st) {
    if (a.N <= 0 || a.F <= 0) return cudaSuccess;
    const unsigned tiles = (unsigned)((a.S + 15) / 16);
    k_sil_bwd<<<dim3(tiles, tiles, (unsigned)a.N), 256, 0, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int pairs = ((uintptr_t)a.grad_verts & 7u) == 0;
    k_sil_gather<<<(unsigned)((a.F + 255) / 256), 256, 0, st>>>(a, pairs);
    return cudaGetLastError();
}

}  // namespace mr
