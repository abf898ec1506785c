// gp2s_kernel_math.cuh -- device evaluation of the kernel pieces shared by the assembly, value and
// adjoint kernels: the Wendland taper (Eq. 3 and the "C2" reading) and its derivative.
#pragma once

#include <cuda_runtime.h>

namespace gp2s {

// phi(t) for t = |xi - xj| / r; zero for t >= 1 (strict support, Eq. 3).
//   kind 1 (Eq. 3):        (1-t)^8 (32 t^3 + 25 t^2 + 8 t + 1)
//   kind 0, d <= 3 (C2 reading):  (1-t)^4 (4 t + 1)
//   kind 0, d == 4 (C2 reading):  (1-t)^5 (5 t + 1)
template <class T>
__device__ __forceinline__ T wendland(int kind, int d, T t)
{
    if constexpr (sizeof(T) == 8) {
        // read off the high word: an FP64 comparison costs as much as an addition.  NaN is outside the
        // support whatever its sign (inf - inf has the sign bit set)
        const int hi = __double2hiint((double)t);
        if (hi >= 0x3ff00000 || (unsigned)hi > 0xfff00000u) return T(0);
        if (hi < 0) t = T(0);
    } else {
        if (!(t < T(1))) return T(0);
        if (t < T(0)) t = T(0);
    }
    const T u = T(1) - t;
    const T u2 = u * u;
    if (kind == 1) {
        const T u4 = u2 * u2;
        return (u4 * u4) * (((T(32) * t + T(25)) * t + T(8)) * t + T(1));
    }
    if (d <= 3) return (u2 * u2) * (T(4) * t + T(1));
    return (u2 * u2 * u) * (T(5) * t + T(1));
}

// d phi / d t.
template <class T>
__device__ __forceinline__ T wendland_dt(int kind, int d, T t)
{
    if (!(t < T(1))) return T(0);
    if (t < T(0)) t = T(0);
    const T u = T(1) - t;
    const T u2 = u * u;
    if (kind == 1) {
        const T u7 = u2 * u2 * u2 * u;
        return T(-22) * t * u7 * ((T(16) * t + T(7)) * t + T(1));
    }
    if (d <= 3) return T(-20) * t * (u2 * u);
    return T(-30) * t * (u2 * u2);
}

// phi'(t) / t, finite at t = 0 (each form's derivative carries a factor t).
template <class T>
__device__ __forceinline__ T wendland_dt_over_t(int kind, int d, T t)
{
    if (!(t < T(1))) return T(0);
    if (t < T(0)) t = T(0);
    const T u = T(1) - t;
    const T u2 = u * u;
    if (kind == 1) {
        const T u7 = u2 * u2 * u2 * u;
        return T(-22) * u7 * ((T(16) * t + T(7)) * t + T(1));
    }
    if (d <= 3) return T(-20) * (u2 * u);
    return T(-30) * (u2 * u2);
}

#ifdef __CUDACC__
// Square root of q >= 0 in six FP64 operations: the FP32 reciprocal root y of q (its exponent and upper
// mantissa bits moved to FP32 and back by integer operations, since conversions are FP64 work), one coupled
// Newton step for g ~ sqrt(q) and h ~ 1 / (2 sqrt(q)) (Goldschmidt's iteration), and the residual
// correction g + (q - g^2) h.  y is off by less than 2^-21, g and h by 2^-42, so before its last rounding
// the result is off by less than 2^-80: it is the correctly rounded root unless that root lies
// within 2^-80 of the middle between two doubles (one q in 2^26), and then it may be its neighbour.  Zero, and
// values outside 2^-100 .. 2^100, take sqrt().
__device__ __forceinline__ double sqrt_pos(double q)
{
    const int hi = __double2hiint(q), lo = __double2loint(q);
    if (hi < ((1023 - 100) << 20) || hi >= ((1023 + 100) << 20)) return sqrt(q);
    const float f = __int_as_float(((hi - ((1023 - 127) << 20)) << 3) | (int)((unsigned)lo >> 29));
    const int yb = __float_as_int(rsqrtf(f));
    const int yhi = (yb >> 3) + ((1023 - 127) << 20);
    const double y = __hiloint2double(yhi, yb << 29), h0 = __hiloint2double(yhi - (1 << 20), yb << 29);
    const double g0 = q * y;
    const double e = fma(-g0, h0, 0.5);
    const double g = fma(g0, e, g0), h = fma(h0, e, h0);
    return fma(fma(-g, g, q), h, g);
}

// 1 / d for a positive finite d in three dependent FP64 operations instead of a full division's chain: the
// FP32 reciprocal r (the same bit moves; 1 - d r = e below 2^-22) and one step of Chebyshev's third-order
// iteration, r (1 + e + e^2).  Off by less than 2^-65 before the last rounding: within an ulp of the
// quotient, and equal to it but for one d in some thousands.  Outside 2^-100 .. 2^100 the division itself.
__device__ __forceinline__ double rcp_pos(double d)
{
    const int hi = __double2hiint(d), lo = __double2loint(d);
    if (hi < ((1023 - 100) << 20) || hi >= ((1023 + 100) << 20)) return 1.0 / d;
    const float f = __int_as_float(((hi - ((1023 - 127) << 20)) << 3) | (int)((unsigned)lo >> 29));
    const int rf = __float_as_int(1.0f / f);
    const double r = __hiloint2double((rf >> 3) + ((1023 - 127) << 20), rf << 29);
    const double e = fma(-d, r, 1.0);
    return fma(r, fma(e, e, e), r);
}
#endif

}  // namespace gp2s
