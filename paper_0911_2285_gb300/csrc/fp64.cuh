// FP64 helpers for a GPU whose FP64 pipe is scarce (measured on GB300: 2 lanes per
// clock per SM and 64 cycles of latency for every FP64 instruction, conversions to
// and from FP32 included; FP32 and integer instructions issue 32 to 64 times as
// fast): conversions on the integer pipe, and reciprocals and square roots from
// FP32 seeds, whose library forms are serial chains of dozens of FP64 steps.
#pragma once
#include "common.cuh"

namespace lqcd {

// a positive and inside [2^-99, 2^99): squares and Newton seeds stay in FP32's
// normal range. On the high word: an FP64 comparison costs the FP64 pipe's latency.
__device__ __forceinline__ bool mid_range(double a) { return ((unsigned)__double2hiint(a) >> 20) - 924u < 198u; }

// FP32 <-> FP64 of a positive number inside FP32's normal range; to FP32 by
// truncation, which is good enough for the Newton seeds below.
__device__ __forceinline__ float seed_f32(double a) {
    return __uint_as_float((unsigned)(((__double2hiint(a) - (896 << 20)) << 3) | ((unsigned)__double2loint(a) >> 29)));
}
__device__ __forceinline__ double exact_f64(float a) {
    const unsigned b = __float_as_uint(a);
    return __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29));
}

// FP32 to FP64, exact (infinities and NaNs kept); subnormals (below 1.2e-38) give
// zero. Without the conversion instruction even as a rare branch: the compiler
// would turn the branch into a select and issue it always.
__device__ __forceinline__ double widen(float a) {
    const unsigned b = __float_as_uint(a), m = b & 0x7fffffffu;
    const unsigned up = m >= 0x7f800000u ? (1792u << 20) : (896u << 20);
    const bool zero = m < 0x00800000u;
    return __hiloint2double((int)((b & 0x80000000u) | (zero ? 0u : (m >> 3) + up)), zero ? 0 : (int)(b << 29));
}
// FP64 to FP32, to nearest (ties away from zero); below 2^-126 zero, from FP32's
// largest number up infinity, NaN kept.
__device__ __forceinline__ float narrow(double a) {
    const unsigned hi = (unsigned)__double2hiint(a), lo = (unsigned)__double2loint(a), sign = hi & 0x80000000u;
    const unsigned l2 = lo + 0x10000000u;                       // half a unit of FP32's last place
    const unsigned h2 = (hi & 0x7fffffffu) + (l2 < lo ? 1u : 0u);
    unsigned r = ((h2 - (896u << 20)) << 3) | (l2 >> 29);
    if (h2 < (897u << 20)) r = 0u;
    if (h2 >= (1151u << 20)) r = 0x7f800000u;
    if ((hi & 0x7fffffffu) + (lo != 0u ? 1u : 0u) > 0x7ff00000u) r = 0x7fffffffu;   // NaN
    return __uint_as_float(sign | r);
}
__device__ __forceinline__ float2 narrow(double2 a) { return make_float2(narrow(a.x), narrow(a.y)); }
__device__ __forceinline__ double2 widen(float2 a) { return make_double2(widen(a.x), widen(a.y)); }

// 1/sqrt(a) for a > 0 in FP64: inside FP32's normal range an FP32 reciprocal
// square root y (relative error about 2^-21) and one step of third order: with
// e = 1 - a y^2, 1/sqrt(a) = y (1 + e/2 + 3 e^2/8 + O(e^3)). Outside: 1 / sqrt(a).
__device__ __forceinline__ double rsqrt_fp64(double a) {
    if (!mid_range(a)) return 1.0 / sqrt(a);
    const double y = exact_f64(rsqrtf(seed_f32(a)));
    const double e = fma(-(a * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// 1/a in FP64 the same way: FP32 reciprocal seed y, e = 1 - a y,
// 1/a = y (1 + e + e^2 + O(e^3)). Outside FP32's normal range: 1 / a.
__device__ __forceinline__ double rcp_fp64(double a) {
    const double m = fabs(a);
    if (!mid_range(m)) return 1.0 / a;
    const double y = copysign(exact_f64(__frcp_rn(seed_f32(m))), a);
    const double e = fma(-a, y, 1.0);
    return fma(y * e, 1.0 + e, y);
}

// sqrt(a) for a >= 0: a / sqrt(a) and one correction of the product's rounding.
__device__ __forceinline__ double sqrt_fp64(double a) {
    if (!mid_range(a)) return sqrt(a);
    const double r = rsqrt_fp64(a), s = a * r;
    return fma(0.5 * r, fma(-s, s, a), s);
}

}  // namespace lqcd
