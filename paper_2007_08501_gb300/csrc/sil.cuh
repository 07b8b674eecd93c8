// Packed silhouette slots: what the silhouette blend's backward needs of a
// fragment, in 8 bytes instead of the 28 of the Fragment data.
//
//   high word  the signed squared distance (the sign bit tells inside)
//   low word   face id (30 bits), nearest edge (2 bits: 0 v0v1, 1 v1v2, 2 v2v0)
//
// A pixel's slots ascend by (depth, id) and end at the first kSilEnd (or after
// K); what follows is never written nor read, so pixels without faces, most of
// an image, cost one slot.
#pragma once

#include "rast_common.cuh"

namespace mr {

constexpr unsigned long long kSilEnd = ~0ull;  // not a distance: its high word is a NaN
constexpr int64_t kSilMaxFaces = 1ll << 30;

__device__ __forceinline__ unsigned long long sil_pack(float d, int f, int edge) {
    return ((unsigned long long)__float_as_uint(d) << 32) | (unsigned)f | ((unsigned)edge << 30);
}

// Signed squared distance of a candidate and its nearest edge: face_fragment's
// distance, bit for bit.
__device__ __forceinline__ float face_distance(const FaceRec &r, const PixC &p, int &edge) {
    float qx, qy, b0, b1, b2, t;
    local_q(r, p, qx, qy);
    screen_bary(r, qx, qy, b0, b1, b2);
    const bool inside = (b0 >= 0.f) && (b1 >= 0.f) && (b2 >= 0.f);
    const float s = nearest_edge(r, qx, qy, edge, t);
    return inside ? -s : s;
}

}  // namespace mr
