// starlet_math.cuh -- the B3-spline filter (taps 1, 4, 6, 4, 1) on fp32 scalars,
// vectors and packed pairs, all with the same rounding (starlet.cu, small.cu).
#pragma once

#include "common.cuh"

namespace fm {

__device__ __forceinline__ float4 f4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void sf4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
__device__ __forceinline__ float tap5(float a, float b, float c, float d, float e)
{
    // (a + e) + 4 (b + d) + 6 c
    return fmaf(6.f, c, fmaf(4.f, b + d, a + e));
}
__device__ __forceinline__ float4 tap5(float4 a, float4 b, float4 c, float4 d, float4 e)
{
    return make_float4(tap5(a.x, b.x, c.x, d.x, e.x), tap5(a.y, b.y, c.y, d.y, e.y), tap5(a.z, b.z, c.z, d.z, e.z),
                       tap5(a.w, b.w, c.w, d.w, e.w));
}
struct Pair4 {  // four columns as two packed pairs
    float2 a, b;
};
__device__ __forceinline__ Pair4 p4(const float *p)
{
    const float4 v = f4(p);
    return Pair4{make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
// (a + e) + 4 (b + d) + 6 c on packed pairs, the rounding of tap5
__device__ __forceinline__ float2 tap5(float2 a, float2 b, float2 c, float2 d, float2 e)
{
    return __ffma2_rn(make_float2(6.f, 6.f), c, __ffma2_rn(make_float2(4.f, 4.f), __fadd2_rn(b, d), __fadd2_rn(a, e)));
}
__device__ __forceinline__ Pair4 tap5(const Pair4 &a, const Pair4 &b, const Pair4 &c, const Pair4 &d, const Pair4 &e)
{
    return Pair4{tap5(a.a, b.a, c.a, d.a, e.a), tap5(a.b, b.b, c.b, d.b, e.b)};
}

}  // namespace fm
