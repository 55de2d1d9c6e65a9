// sp_crossing.cuh -- the winding test of one lattice edge.
#pragma once
#include <cuda_runtime.h>

namespace sp {

// Signed crossing of the positive real axis by the segment u -> v: +1 upward
// when cross(u, v) >= 0, -1 downward when cross(u, v) <= 0, else 0; a vertex
// on the axis counts as above it.  FP64 products of FP32 values are exact, so
// the sign is.
__device__ __forceinline__ int crossing(float2 u, float2 v)
{
    const bool ua = u.y >= 0.0f, va = v.y >= 0.0f;
    if (ua == va) return 0;
    const double cr = __dsub_rn(__dmul_rn((double)u.x, (double)v.y), __dmul_rn((double)u.y, (double)v.x));
    return va ? (cr >= 0.0 ? 1 : 0) : (cr <= 0.0 ? -1 : 0);
}

// The same from FP32 products where they tell: rounding is monotone, so two
// rounded products that differ are ordered as the exact ones are.  unsure is
// set when they do not (a tie or a NaN on an edge that changes sides): the
// caller then asks crossing().
__device__ __forceinline__ int crossing_fp32(float2 u, float2 v, bool &unsure)
{
    const int ua = u.y >= 0.0f, va = v.y >= 0.0f;
    const float p = __fmul_rn(u.x, v.y), q = __fmul_rn(u.y, v.x);
    const bool up = p > q, down = p < q;
    unsure = unsure || (ua != va && !up && !down);
    return (va ? up : down) ? va - ua : 0;
}

}  // namespace sp
