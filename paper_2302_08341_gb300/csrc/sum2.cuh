// Sums in two FP32 words.
#pragma once

namespace flood {

// A sum kept in two FP32 words (hi + lo, about 2^-46 relative): Knuth's
// error-free addition, the errors added up beside the sum.  The FP64 pipe
// takes 64 cycles a warp instruction and a division fifteen of them, so what
// every warp sums stays off it and one lane widens the total at the end: a
// warp's five-round FP64 sum over its lanes cost a strip some 2400 cycles.
struct Sum2 {
    float hi = 0.0f, lo = 0.0f;
    __device__ __forceinline__ void add(float x)
    {
        const float s = __fadd_rn(hi, x), b = __fsub_rn(s, hi);
        lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(x, b)));
        hi = s;
    }
    __device__ __forceinline__ bool zero() const { return hi == 0.0f && lo == 0.0f; }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
    // x times the sum of two words
    __device__ __forceinline__ void add_product(float x, float2 y)
    {
        const float p = __fmul_rn(x, y.x);
        add(p);
        lo = __fadd_rn(lo, __fmaf_rn(x, y.y, __fmaf_rn(x, y.x, -p)));
    }
    __device__ __forceinline__ void merge(float h, float l)
    {
        add(h);
        lo = __fadd_rn(lo, l);
    }
    __device__ __forceinline__ void warp_sum()
    {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const float h = __shfl_xor_sync(0xffffffffu, hi, off), l = __shfl_xor_sync(0xffffffffu, lo, off);
            merge(h, l);
        }
    }
};

}  // namespace flood
