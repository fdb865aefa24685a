// Arithmetic on unevaluated sums h + l of two floats (about 48 bits), by the
// error-free transformations of Knuth and Dekker, beside the same operations on
// doubles: for results that need more than FP32 on the way and are rounded to
// FP32 in the end, the pairs run on the FP32 pipe, 64 times as wide as GB300's
// FP64 pipe.
#pragma once

#include <cuda_runtime.h>

namespace les {

template <typename real> struct Num;
template <> struct Num<double> {
    typedef double T;
    static __device__ __forceinline__ T of(double v) { return v; }
    static __device__ __forceinline__ T mul(double a, T b) { return a * b; }
    static __device__ __forceinline__ T mulp(T a, T b) { return a * b; }
    static __device__ __forceinline__ T add(T a, T b) { return a + b; }
    static __device__ __forceinline__ T sub(T a, T b) { return a - b; }
    static __device__ __forceinline__ float out(T a) { return (float)a; }
};
struct FloatPair {
    float h, l;
};
template <> struct Num<float> {
    typedef FloatPair T;
    static __device__ __forceinline__ T of(double v)
    {
        const float h = (float)v;
        return {h, (float)(v - (double)h)};
    }
    static __device__ __forceinline__ T quick(float a, float b) // |a| >= |b|
    {
        const float s = __fadd_rn(a, b);
        return {s, __fsub_rn(b, __fsub_rn(s, a))};
    }
    static __device__ __forceinline__ T mul(float a, T b)
    {
        const float p = __fmul_rn(a, b.h);
        return quick(p, __fmaf_rn(a, b.l, __fmaf_rn(a, b.h, -p)));
    }
    static __device__ __forceinline__ T mulp(T a, T b)
    {
        const float p = __fmul_rn(a.h, b.h);
        return quick(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
    }
    static __device__ __forceinline__ T add(T a, T b)
    {
        const float s = __fadd_rn(a.h, b.h), v = __fsub_rn(s, a.h);
        const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, v)), __fsub_rn(b.h, v));
        return quick(s, __fadd_rn(e, __fadd_rn(a.l, b.l)));
    }
    static __device__ __forceinline__ T sub(T a, T b) { return add(a, T{-b.h, -b.l}); }
    static __device__ __forceinline__ float out(T a) { return __fadd_rn(a.h, a.l); }
};

} // namespace les
