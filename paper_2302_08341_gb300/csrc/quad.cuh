// A lane's four neighbouring cells as two FP32 pairs, the operands of the
// two-wide instructions.
#pragma once

#include <cuda_runtime.h>

namespace flood {

struct Quad {
    float2 a, b;
};

__device__ __forceinline__ Quad ld_quad(const float* p)
{
    const float4 t = *reinterpret_cast<const float4*>(p);
    return Quad{make_float2(t.x, t.y), make_float2(t.z, t.w)};
}
__device__ __forceinline__ void st_quad(float* p, const Quad& v)
{
    *reinterpret_cast<float4*>(p) = make_float4(v.a.x, v.a.y, v.b.x, v.b.y);
}
__device__ __forceinline__ float& quad_at(Quad& v, int j)
{
    return j == 0 ? v.a.x : j == 1 ? v.a.y : j == 2 ? v.b.x : v.b.y;
}
__device__ __forceinline__ const float& quad_at(const Quad& v, int j)
{
    return j == 0 ? v.a.x : j == 1 ? v.a.y : j == 2 ? v.b.x : v.b.y;
}
__device__ __forceinline__ Quad quad_of(float x) { return Quad{make_float2(x, x), make_float2(x, x)}; }

}  // namespace flood
