// Unevaluated sums hi + lo of two FP32 numbers (about 48 bits), by the
// error-free transformations of floating-point arithmetic: the two-sum of Knuth
// (The Art of Computer Programming 2, 4.2.2) and the two-product with a fused
// multiply-add.
#pragma once

#include "lbm_internal.cuh"

namespace lbm {

struct Pair32 {
    float hi, lo;
};

// hi + lo = a + b exactly
__device__ __forceinline__ Pair32 two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float t = __fadd_rn(s, -a);
    return {s, __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -t)), __fadd_rn(b, -t))};
}
__device__ __forceinline__ Pair32 operator+(Pair32 a, Pair32 b)
{
    const Pair32 s = two_sum(a.hi, b.hi);
    return {s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo))};
}
__device__ __forceinline__ Pair32 operator-(Pair32 a, Pair32 b) { return a + Pair32{-b.hi, -b.lo}; }
// (without lo^2: added here, it would be rounded away more often than not)
__device__ __forceinline__ Pair32 square(Pair32 a)
{
    const float p = __fmul_rn(a.hi, a.hi);
    return {p, __fmaf_rn(2.f * a.hi, a.lo, __fmaf_rn(a.hi, a.hi, -p))};
}
__device__ __forceinline__ Pair32 operator*(Pair32 a, Pair32 b)
{
    const float p = __fmul_rn(a.hi, b.hi);
    return {p, __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.hi, b.hi, -p)))};
}
__device__ __forceinline__ double value(Pair32 a) { return (double)a.hi + (double)a.lo; }

}  // namespace lbm
