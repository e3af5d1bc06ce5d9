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

// FP32 to FP64, exact over FP32's whole range (subnormals scaled up first). Without
// the conversion instruction even as a rare branch: the compiler would turn the
// branch into a select and issue it always.
__device__ __forceinline__ double widen(float a) {
    const unsigned ma = __float_as_uint(a) & 0x7fffffffu;
    const bool sub = ma < 0x00800000u;
    const unsigned b = __float_as_uint(sub ? a * 16777216.f : a), m = b & 0x7fffffffu;
    const unsigned up = ma >= 0x7f800000u ? (1792u << 20) : sub ? (872u << 20) : (896u << 20);
    const bool zero = m == 0u;
    return __hiloint2double((int)((b & 0x80000000u) | (zero ? 0u : (m >> 3) + up)), zero ? 0 : (int)(b << 29));
}
// The bits below FP32's normal range, |a| < 2^-126 (m: high word of |a|): a whole number of
// 2^-149. A call: inlined, its 64-bit shifts are issued for every conversion (deflation of
// 8 guesses on 16^3 x 32 0.98 -> 1.03 ms).
static __device__ __noinline__ unsigned narrow_small(unsigned m, unsigned lo) {
    const unsigned sh = 926u - (m >> 20);   // places of the 53-bit mantissa below 2^-149: 30 and more
    const unsigned long long v = ((unsigned long long)((m & 0xfffffu) | 0x100000u) << 32) | lo;
    return sh > 54u ? 0u : (unsigned)((v + ((1ull << (sh - 1u)) - 1ull) + ((v >> sh) & 1ull)) >> sh);
}
// FP64 to FP32, to nearest over FP32's whole range; EVEN: ties to even, as the conversion
// instruction rounds, else away from zero. From FP32's largest number up infinity, NaN kept.
template <bool EVEN> __device__ __forceinline__ float narrow_to(double a) {
    const unsigned hi = (unsigned)__double2hiint(a), lo = (unsigned)__double2loint(a), m = hi & 0x7fffffffu;
    const unsigned l2 = lo + (EVEN ? 0x0fffffffu + ((lo >> 29) & 1u) : 0x10000000u);   // half a unit of FP32's last place
    const unsigned h2 = m + (l2 < lo ? 1u : 0u);
    unsigned r = ((h2 - (896u << 20)) << 3) | (l2 >> 29);
    if (h2 >= (1151u << 20)) r = 0x7f800000u;
    if (m < (897u << 20)) r = (m | lo) == 0u ? 0u : narrow_small(m, lo);
    if (m + (lo != 0u ? 1u : 0u) > 0x7ff00000u) r = 0x7fffffffu;   // NaN
    return __uint_as_float((hi & 0x80000000u) | r);
}
__device__ __forceinline__ float narrow(double a) { return narrow_to<true>(a); }
__device__ __forceinline__ float2 narrow(double2 a) { return make_float2(narrow(a.x), narrow(a.y)); }
__device__ __forceinline__ double2 widen(float2 a) { return make_double2(widen(a.x), widen(a.y)); }
// FP64 to storage precision S and back.
template <typename S> __device__ __forceinline__ cplx<S> nar(double2 a) {
    if constexpr (sizeof(S) == 4) return narrow(a);
    else return a;
}
__device__ __forceinline__ double2 wid(float2 a) { return widen(a); }
__device__ __forceinline__ double2 wid(double2 a) { return a; }

// 2^e with the exponent field f = e + 1023, 0 < f < 2047; a times 2^e by its exponent.
__device__ __forceinline__ double pow2_field(int f) { return __hiloint2double(f << 20, 0); }
__device__ __forceinline__ double shift_exp(double a, int e) {
    return __hiloint2double(__double2hiint(a) + e * (1 << 20), __double2loint(a));
}
// a positive with an exponent that the routines below may move by half or negate.
__device__ __forceinline__ bool wide_range(double a) { return ((unsigned)__double2hiint(a) >> 20) - 64u < 1918u; }

// 1/sqrt(a) for a > 0 in FP64: a scaled by 4^k into [1, 4), an FP32 reciprocal
// square root y (relative error about 2^-21) and one step of third order: with
// e = 1 - a y^2, 1/sqrt(a) = y (1 + e/2 + 3 e^2/8 + O(e^3)). Near the ends of
// FP64's range: 1 / sqrt(a).
__device__ __forceinline__ double rsqrt_fp64(double a) {
    if (!wide_range(a)) return 1.0 / sqrt(a);
    const int k = ((__double2hiint(a) >> 20) - 1023) & ~1;
    const double m = shift_exp(a, -k);
    const double y = exact_f64(rsqrtf(seed_f32(m)));
    const double e = fma(-(m * y), y, 1.0);
    return shift_exp(fma(y * e, fma(0.375, e, 0.5), y), -(k / 2));
}

// 1/a in FP64 the same way: mantissa in [1, 2), FP32 reciprocal seed y, e = 1 - a y,
// 1/a = y (1 + e + e^2 + O(e^3)).
__device__ __forceinline__ double rcp_fp64(double a) {
    const double p = fabs(a);
    if (!wide_range(p)) return 1.0 / a;
    const int k = (__double2hiint(p) >> 20) - 1023;
    const double m = shift_exp(p, -k);
    const double y = exact_f64(__frcp_rn(seed_f32(m)));
    const double e = fma(-m, y, 1.0);
    return copysign(shift_exp(fma(y * e, 1.0 + e, y), -k), a);
}

// sqrt(a) for a >= 0: a / sqrt(a) and one correction of the product's rounding.
__device__ __forceinline__ double sqrt_fp64(double a) {
    if (!wide_range(a)) return sqrt(a);
    const double r = rsqrt_fp64(a), s = a * r;
    return fma(0.5 * r, fma(-s, s, a), s);
}

// a / b: the larger part of b scaled to [1, 2), one reciprocal of |b|^2 (Smith's
// division takes three dependent FP64 divisions). Near the ends of the range: Smith.
__device__ __forceinline__ double2 cdiv_fp64(double2 a, double2 b) {
    const int f = max(__double2hiint(b.x) & 0x7ff00000, __double2hiint(b.y) & 0x7ff00000) >> 20;
    if (f < 64 || f > 1982) return cdiv(a, b);
    const double up = pow2_field(2046 - f);   // 2^(1023 - f)
    const double2 s = make_double2(up * b.x, up * b.y);
    const double r = rcp_fp64(fma(s.y, s.y, s.x * s.x)) * up;
    const double2 t = make_double2(r * s.x, -(r * s.y));
    return make_double2(fma(-a.y, t.y, a.x * t.x), fma(a.y, t.x, a.x * t.y));
}

// |z| >= tol s1 s2 (s1, s2 >= 0); false for NaN. On squares where both sides' stay in
// FP64's range (exponents within +-480), else by hypot.
static __device__ __noinline__ bool abs_at_least_far(double2 z, double t) { return cabs_(z) >= t; }
__device__ __forceinline__ bool abs_at_least(double2 z, double tol, double s1, double s2) {
    const double t = tol * s1 * s2;
    const unsigned fx = (unsigned)__double2hiint(z.x) & 0x7fffffffu, fy = (unsigned)__double2hiint(z.y) & 0x7fffffffu;
    const unsigned fz = max(fx, fy) >> 20, ft = (unsigned)__double2hiint(t) >> 20;
    if (fz - 543u < 961u && ft - 543u < 961u) return fma(z.y, z.y, z.x * z.x) >= t * t;
    return abs_at_least_far(z, t);
}

}  // namespace lqcd
