// Double-FP32 ("double-float") arithmetic for the reliable-update residual.
//
// FP64 runs at a small fraction of the FP32 rate on this GPU, so the in-iteration
// reliable updates evaluate A x in pairs of FP32 numbers: a value is the
// unevaluated sum h + l (|l| <= ulp(h)/2), about 48 significant bits. Sums use
// Knuth's two-sum, products Dekker's two-product through the fused multiply-add,
// and the SU(3) row sums are compensated dot products (Ogita, Rump and Oishi,
// "Accurate sum and dot product", SIAM J. Sci. Comput. 26 (2005), Dot2 with the
// cross terms of the low parts). The convergence certificate of a solve is
// still the native FP64 residual.
#pragma once
#include "fp64.cuh"

namespace lqcd {

struct dfl { float h, l; };
struct dfc { dfl x, y; };   // complex: x = real part, y = imaginary part

__device__ __forceinline__ dfl operator-(dfl a) { return {-a.h, -a.l}; }
__device__ __forceinline__ dfl operator+(dfl a, dfl b) {
    const float s = a.h + b.h, v = s - a.h;
    float e = (a.h - (s - v)) + (b.h - v);
    e += a.l + b.l;
    const float h = s + e;
    return {h, e - (h - s)};
}
__device__ __forceinline__ dfl operator-(dfl a, dfl b) { return a + (-b); }
// a + f b, f = +-1
__device__ __forceinline__ dfl df_axpy(dfl a, float f, dfl b) {
    const float s = fmaf(f, b.h, a.h), v = s - a.h;
    float e = (a.h - (s - v)) + fmaf(f, b.h, -v);
    e += fmaf(f, b.l, a.l);
    const float h = s + e;
    return {h, e - (h - s)};
}
__device__ __forceinline__ dfc operator+(dfc a, dfc b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ dfc operator-(dfc a, dfc b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ dfc operator-(dfc a) { return {-a.x, -a.y}; }

// One FP64 instruction each (the conversions run on the integer pipe). In a split the side
// that a tie goes to costs nothing: l holds the rest of h exactly, and is off by half a unit
// of its own either way.
__device__ __forceinline__ dfl df_split(double v) {
    const float h = narrow_to<false>(v);
    return {h, narrow_to<false>(v - widen(h))};
}
__device__ __forceinline__ double df_value(dfl a) { return widen(a.h) + widen(a.l); }

// Compensated sum of products a_i b_i: s + c, c collecting every rounding error.
struct Dot2 {
    float s, c;
    __device__ __forceinline__ void first(dfl a, dfl b) {
        s = a.h * b.h;
        float e = fmaf(a.h, b.h, -s);
        e = fmaf(a.h, b.l, e);
        c = fmaf(a.l, b.h, e);
    }
    __device__ __forceinline__ void add(dfl a, dfl b) {
        const float p = a.h * b.h;
        float e = fmaf(a.h, b.h, -p);
        e = fmaf(a.h, b.l, e);
        e = fmaf(a.l, b.h, e);
        const float s2 = s + p, bp = s2 - s;
        const float q = (s - (s2 - bp)) + (p - bp);
        s = s2;
        c += q + e;
    }
    // + (h + l), exact product signs folded in by the caller
    __device__ __forceinline__ void plus(float h, float l) {
        const float s2 = s + h, bp = s2 - s;
        c += ((s - (s2 - bp)) + (h - bp)) + l;
        s = s2;
    }
    // + f (h + l), f = +-1: the same two-sum with the sign in the multiply-adds
    __device__ __forceinline__ void plus(float f, float h, float l) {
        const float s2 = fmaf(f, h, s), bp = s2 - s;
        c += fmaf(f, l, (s - (s2 - bp)) + fmaf(f, h, -bp));
        s = s2;
    }
    __device__ __forceinline__ dfl done() const {
        const float h = s + c;
        return {h, c - (h - s)};
    }
};

}  // namespace lqcd
