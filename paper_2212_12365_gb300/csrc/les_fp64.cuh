// FP64 building blocks of the stage kernels, chosen to issue few FP64
// instructions: GB300's FP64 pipe takes two lanes per clock and SM.
//
// Reciprocals and square roots iterate from the hardware's approximate seeds
// (about 20 bits).  With e = 1 - b y0, the series 1/b = y0 (1 + e + e^2 + ...)
// cut after e^2 leaves e^3 ~ 2^-60: three operations (two Newton steps take
// four).  For the square root, with t = x y0, e = 1 - t y0, sqrt(x) =
// t (1 + e/2 + 3 e^2/8 + ...): five operations, against eight of the
// library's sqrt; both round to within about an ulp.  Comparisons of
// non-negative numbers go to the integer pipe.
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
// x^1/2, x >= 0; 0 below the normal range
template <int E> // times 2^E
__device__ __forceinline__ double sqrt64_scaled(double x)
{
    const double y = rsqrt_seed64(x);
    const double t0 = x * y;
    const double e = fma(-t0, y, 1.0);
    const double t = E != 0 ? __hiloint2double(__double2hiint(t0) + E * (1 << 20), __double2loint(t0)) : t0;
    const double s = fma(t, e * fma(0.375, e, 0.5), t);
    return __double2hiint(x) < 0x00100000 && __double2hiint(x) >= 0 ? 0.0 : s;
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
