// The certificate of the binary32 codeword ranking, shared by the kernels of the write path.
#pragma once

#include "novakv_internal.cuh"

// What the binary32 evaluation can have moved a squared distance by: the coefficient vector of the group
// is off by at most delta in norm, the eight operations of the distance add a relative 6 * 2^-24.
// |d32 - d| <= 2 sqrt(d) delta + delta^2 + 6 * 2^-24 d; the test below uses twice the bound at the larger of the two
// distances (both have moved) with some slack on the constants.  key_rel: what the caller's packing of the distances
// has cut from either of them, relative.
__device__ __forceinline__ bool needs_exact_search(float best, float second, float delta, float key_rel = 0.f) {
    float root;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(root) : "f"(second));          // (the slack covers its error)
    const float thr = 4.5f * root * delta + 2.5f * delta * delta + (9.6e-7f + 2.f * key_rel) * second;     // 9.6e-7 > 16 * 2^-24
    return !(second - best > thr);
}
