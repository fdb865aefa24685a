// FP64 building blocks of the stage kernels, chosen to issue few FP64
// instructions: GB300's FP64 pipe takes two lanes per clock and SM.
//
// Reciprocals and square roots refine the hardware's approximate seeds (about 20
// bits) by one step of a power series in the seed's error.  With e = 1 - b y0
// (exact to 2^-73 by the fused multiply-add), 1/b = y0 (1 + e + e^2 + ...) cut
// after e^2 leaves e^3 ~ 2^-60: three operations.  With e = 1 - x y0^2, the
// binomial series (1 - e)^(-1/2) = 1 + e/2 + 3 e^2/8 + ... cut after e^2 gives
// x^(-1/2), within about an ulp.  The square root takes the same series on the
// residual: t = x y0 rounded, r = x - t^2 (exact but for its last bit), sqrt(x) =
// t + r y0 (1/2 + 3 e/8), so that the rounding of t does not reach the result:
// six operations, within 0.53 ulp.  (As t (1 + e/2 + 3 e^2/8), five operations,
// it was off by up to 0.76 ulp; the sixth operation costs ten FP64 steps 28 us of
// 3120 on 48x32x32 and 0.27 ms of 34.3 on the polar 200x75x40.)
// Comparisons of non-negative numbers go to the integer pipe.
#pragma once

#include <cuda_runtime.h>

namespace les {

__device__ __forceinline__ double rcp_seed64(double b)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(b));
    return r;
}
__device__ __forceinline__ double rsqrt_seed64(double b)
{
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(b));
    return r;
}
// 1/b, b positive and normal
__device__ __forceinline__ double rcp64(double b)
{
    const double r = rcp_seed64(b);
    const double e = fma(-b, r, 1.0);
    return fma(r, fma(e, e, e), r);
}
// 1/b to a relative 1e-12 or so: for factors whose error the residual damps
// (pressure sensor, Sutherland law)
__device__ __forceinline__ double rcp64_1(double b)
{
    const double r = rcp_seed64(b);
    return fma(r, fma(-b, r, 1.0), r);
}
// x^-1/2, x positive and normal
__device__ __forceinline__ double rsqrt64(double x)
{
    const double y = rsqrt_seed64(x);
    const double e = fma(-(x * y), y, 1.0);
    return fma(y, e * fma(0.375, e, 0.5), y);
}
// y 2^E, y and the result normal
template <int E> __device__ __forceinline__ double scaled64(double y)
{
    return E != 0 ? __hiloint2double(__double2hiint(y) + E * (1 << 20), __double2loint(y)) : y;
}
// x^1/2 times 2^E, x >= 0; 0 below the normal range, infinity from infinity (and
// NaN from x < 0)
template <int E> __device__ __forceinline__ double sqrt64_scaled(double x)
{
    const double y = rsqrt_seed64(x), t = x * y;
    const double e = fma(-t, y, 1.0), r = fma(-t, t, x);
    const double s = fma(r * scaled64<E>(y), fma(0.375, e, 0.5), scaled64<E>(t));
    const int h = __double2hiint(x), m = h & 0x7fffffff;
    if (m < 0x00100000) return 0.0;
    return h == 0x7ff00000 ? x : s; // (NaN stays NaN: s is one)
}
__device__ __forceinline__ double sqrt64(double x) { return sqrt64_scaled<0>(x); }
__device__ __forceinline__ double twice_sqrt64(double x) { return sqrt64_scaled<1>(x); }
__device__ __forceinline__ double half_sqrt64(double x) { return sqrt64_scaled<-1>(x); }
// max of two non-negative numbers (their bit patterns order as integers)
__device__ __forceinline__ double max_nn(double a, double b)
{
    return __longlong_as_double(max(__double_as_longlong(a), __double_as_longlong(b)));
}
// max(x, 0) by the sign bit
__device__ __forceinline__ double clamp0(double x) { return __double2hiint(x) < 0 ? 0.0 : x; }

} // namespace les
