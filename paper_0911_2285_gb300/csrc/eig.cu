// Small dense FP64 complex algebra on the device, one CTA per problem:
//  * eig with right and left eigenvectors ([zr, zl, D] = eig(C), paper Sec. 1
//    notation), eigenvalues ordered by smallest |lambda| (Sec. 2);
//  * the coefficient-space part of Algorithm BiCG-eigen (Sec. 2);
//  * final Ritz pairs of an eigBiCG window (Algorithm eigBiCG, step 4);
//  * LU factorisation / solves for H = U_l^H A U_r (Algorithm Incremental).
//
// Eigen-solver: Householder reduction to Hessenberg form, complex single-shift
// (Wilkinson) implicit QR to Schur form T = Q^H C Q (Golub & Van Loan,
// "Matrix Computations", Sec. 7.4-7.5), eigenvectors of T by back / forward
// substitution, mapped back with Q. Conventions: right vectors have unit
// 2-norm with their largest-modulus entry real positive; left vectors satisfy
// z^H y = 1.
//
// What bounds it: one problem lives on one SM, and a QR sweep is a chain of
// rotations (about 2500 of them for a 40 x 40 window matrix, 5500 for 60 x 60)
// that cannot overlap, so the time is rotations x the latency of one: form it,
// apply it to two rows, apply it to two columns. FP64 instructions take 64
// cycles each and issue at 2 lanes per clock per SM (measured), so the scalars
// that one thread used to form with the FP64 library (square roots, hypot,
// divisions: thousands of cycles each, the other warps waiting) were most of
// it. Here warp 0 forms the next rotation while the other warps are still
// applying the last one to their rows, two half-warps share each pair (one
// output each), a rotation costs two barriers, and shifts, deflation scans,
// norms, pivot searches and substitutions run across the lanes of a warp.
// Measured: restart coefficients (both eigen-solves and the FP64 finish) 60 x 60
// 20.2 -> 5.0 ms, 40 x 40 10.9 -> 2.7 ms; FP64 eigen-solve 60 x 60 18.2 -> 10.9 ms.
#include <mutex>

#include "../../include/lqcd.h"
#include "dfloat.cuh"
#include "fp64.cuh"
#include "kernels.cuh"

namespace lqcd {
namespace {

constexpr int ET = 256;          // threads per eigen CTA
constexpr int EW = ET / 32;      // warps
constexpr double EPS = 2.220446049250313e-16;
constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ double2 czero() { return make_double2(0.0, 0.0); }
__device__ __forceinline__ double2 cone() { return make_double2(1.0, 0.0); }

// |re| + |im|: the modulus surrogate used for negligibility tests (no sqrt).
__device__ __forceinline__ double cabs1(double2 a) { return fabs(a.x) + fabs(a.y); }

// ------------------------------------------------------ double-float numbers
// The restart's eigen-solves of H^(m) and H^(m-1) run the reduction in
// double-float arithmetic (pairs of FP32 numbers, about 48 significant bits;
// Knuth's two-sum and Dekker's FMA two-product, as for the reliable-update
// residual): the FP32 pipe issues 64 times faster than FP64 on this GPU.
__device__ __forceinline__ dfl df_mul(dfl a, dfl b) {
    const float p = a.h * b.h;
    float e = fmaf(a.h, b.h, -p);
    e = fmaf(a.h, b.l, e);
    e = fmaf(a.l, b.h, e);
    const float h = p + e;
    return {h, e - (h - p)};
}
__device__ __forceinline__ dfc dc_from(double2 a) { return {df_split(a.x), df_split(a.y)}; }
__device__ __forceinline__ double2 dc_to(dfc a) { return make_double2(df_value(a.x), df_value(a.y)); }
__device__ __forceinline__ dfl df_scale(dfl a, float s) { return {a.h * s, a.l * s}; }   // s a power of two
__device__ __forceinline__ dfl df_fast_sum(float h, float l) {   // |l| small against |h|
    const float s = h + l;
    return {s, l - (s - h)};
}
// 1/sqrt(a), a.h inside [1e-28, 1e28], to about 2^-49: FP32 seed y and one
// third-order step. e = 1 - a y^2 is kept as an exact part d (1 minus the rounded
// a.h y^2) and the small rest, and y d/2 with its rounding error: one FP32 number
// for e would leave 2^-47, which the thousands of rotations of a solve add up.
__device__ __forceinline__ dfl df_rsqrt(dfl a) {
    const float y = rsqrtf(a.h);
    const float t = y * y, tl = fmaf(y, y, -t);
    const float p = a.h * t, pl = fmaf(a.h, t, -p);
    const float d = 1.f - p;   // exact: p is within 2^-20 of 1
    const float rest = -fmaf(a.h, tl, fmaf(a.l, t, pl));
    const float hd = 0.5f * d, m = y * hd, ml = fmaf(y, hd, -m);
    const float e = d + rest;
    const float low = fmaf(y, fmaf(0.375f * e, e, 0.5f * rest), ml);
    const float h = y + m;
    return df_fast_sum(h, (m - (h - y)) + low);
}
// 1/a the same way.
__device__ __forceinline__ dfl df_rcp(dfl a) {
    const float y = __frcp_rn(a.h);
    float e = fmaf(-a.h, y, 1.f);
    e = fmaf(-a.l, y, e);
    return df_fast_sum(y, y * fmaf(e, e, e));
}
__device__ __forceinline__ bool df_seed_ok(float h) { return h > 1e-28f && h < 1e28f; }

// ------------------------------------------------------- number types
// What the reduction needs of a complex number type C: u a + v b, c - a b,
// running sums of products, the rotation, the shift and the negligibility test.
struct NumD {
    using C = double2;
    using R = double;
    static constexpr bool WIDE = true;   // squares may leave FP64's range
    static __device__ __forceinline__ C zero() { return czero(); }
    static __device__ __forceinline__ C one() { return cone(); }
    static __device__ __forceinline__ C from(double2 a) { return a; }
    static __device__ __forceinline__ double2 to(C a) { return a; }
    static __device__ __forceinline__ C lin2(C u, C a, C v, C b) {
        return make_double2(fma(-v.y, b.y, fma(v.x, b.x, fma(-u.y, a.y, u.x * a.x))),
                            fma(v.y, b.x, fma(v.x, b.y, fma(u.y, a.x, u.x * a.y))));
    }
    static __device__ __forceinline__ C fms(C c, C a, C b) {
        return make_double2(fma(a.y, b.y, fma(-a.x, b.x, c.x)), fma(-a.y, b.x, fma(-a.x, b.y, c.y)));
    }
    static __device__ __forceinline__ C scale(R s, C a) { return s * a; }
    struct Sum {
        C s = czero();
        __device__ __forceinline__ void add(C a, C b) {
            s = make_double2(fma(-a.y, b.y, fma(a.x, b.x, s.x)), fma(a.y, b.x, fma(a.x, b.y, s.y)));
        }
        __device__ __forceinline__ C value() const { return s; }
    };
    static __device__ __forceinline__ R abs2(C a) { return fma(a.y, a.y, a.x * a.x); }
    static __device__ __forceinline__ R rfrom(double a) { return a; }
    static __device__ __forceinline__ bool is_zero(C a) { return a.x == 0.0 && a.y == 0.0; }
    static __device__ __forceinline__ bool negligible(C sub, C d0, C d1, double anorm) {
        double t = cabs1(d0) + cabs1(d1);
        if (t == 0.0) t = anorm;
        return cabs1(sub) <= EPS * t;
    }
    static __device__ __forceinline__ double wide_abs2(C a) { return abs2(a); }
    // G = [[cx, cy], [-conj(cy), conj(cx)]] with G [x; y] = [n; 0], cx = conj(x)/n,
    // cy = conj(y)/n, n = sqrt(|x|^2 + |y|^2).
    static __device__ __forceinline__ void givens(C x, C y, C& cx, C& cy) {
        const double n2 = abs2(x) + abs2(y);
        if (!wide_range(n2) && n2 == 0.0) { cx = one(); cy = zero(); return; }
        const double inv = rsqrt_fp64(n2);
        cx = make_double2(inv * x.x, -(inv * x.y));
        cy = make_double2(inv * y.x, -(inv * y.y));
    }
};

struct NumF {
    using C = dfc;
    using R = dfl;
    static constexpr bool WIDE = false;
    static __device__ __forceinline__ C zero() { return {{0.f, 0.f}, {0.f, 0.f}}; }
    static __device__ __forceinline__ C one() { return {{1.f, 0.f}, {0.f, 0.f}}; }
    static __device__ __forceinline__ C from(double2 a) { return dc_from(a); }
    static __device__ __forceinline__ double2 to(C a) { return dc_to(a); }
    // Every product and sum normalised: running (s, c) sums would take 30 % fewer
    // instructions, but cost half a bit in the residuals of the small eigenpairs.
    static __device__ __forceinline__ C mul(C a, C b) {
        return {df_mul(a.x, b.x) - df_mul(a.y, b.y), df_mul(a.x, b.y) + df_mul(a.y, b.x)};
    }
    static __device__ __forceinline__ C lin2(C u, C a, C v, C b) { return mul(u, a) + mul(v, b); }
    static __device__ __forceinline__ C fms(C c, C a, C b) { return c - mul(a, b); }
    static __device__ __forceinline__ C scale(R s, C a) { return {df_mul(s, a.x), df_mul(s, a.y)}; }
    struct Sum {
        C s = {{0.f, 0.f}, {0.f, 0.f}};
        __device__ __forceinline__ void add(C a, C b) { s = s + mul(a, b); }
        __device__ __forceinline__ C value() const { return s; }
    };
    static __device__ __forceinline__ R abs2(C a) {
        Dot2 s;
        s.first(a.x, a.x);
        s.add(a.y, a.y);
        return s.done();
    }
    static __device__ __forceinline__ R rfrom(double a) { return df_split(a); }
    static __device__ __forceinline__ bool is_zero(C a) { return a.x.h == 0.f && a.y.h == 0.f; }
    static constexpr float EPS_DF = 1.4e-14f;   // about four units of double-float rounding
    static __device__ __forceinline__ float abs1(C a) { return fabsf(a.x.h) + fabsf(a.y.h); }
    static __device__ __forceinline__ bool negligible(C sub, C d0, C d1, double anorm) {
        float t = abs1(d0) + abs1(d1);
        if (t == 0.f) t = (float)anorm;
        return abs1(sub) <= EPS_DF * t;
    }
    static __device__ __forceinline__ double wide_abs2(C a) { return NumD::abs2(dc_to(a)); }
    static __device__ __forceinline__ void givens(C x, C y, C& cx, C& cy) {
        Dot2 s;
        s.first(x.x, x.x); s.add(x.y, x.y); s.add(y.x, y.x); s.add(y.y, y.y);
        const dfl n2 = s.done();
        if (!df_seed_ok(n2.h)) {   // squares near the ends of FP32's range: in FP64
            double2 dx, dy;
            NumD::givens(dc_to(x), dc_to(y), dx, dy);
            cx = dc_from(dx);
            cy = dc_from(dy);
            return;
        }
        const dfl inv = df_rsqrt(n2);
        cx = {df_mul(inv, x.x), -df_mul(inv, x.y)};
        cy = {df_mul(inv, y.x), -df_mul(inv, y.y)};
    }
};

// Wilkinson shift of [[a, b], [c, d]]: the eigenvalue nearer d is d - corr with
// corr = b c / (t + sqrt(t^2 + b c)), t = (a - d)/2, with the larger denominator.
// A shift only steers the convergence, so double-float arithmetic serves both
// number types, on entries scaled by a power of two (max |entry| near 1), so that
// FP32's exponent range does not matter. Returns corr of the scaled entries.
__device__ __forceinline__ dfc shift_correction(dfc a, dfc b, dfc c, dfc d) {
    const dfc t = {df_scale(a.x - d.x, 0.5f), df_scale(a.y - d.y, 0.5f)};
    const dfc bc = NumF::mul(b, c);
    const dfc q = NumF::lin2(t, t, b, c);   // t^2 + b c
    const dfl m2 = NumF::abs2(q);
    dfc s = NumF::zero();   // sqrt(q), principal branch
    if (m2.h > 1e-36f) {    // |entries| <= 2, so no upper bound is needed
        const dfl m = df_mul(m2, df_rsqrt(m2));
        // the larger of |Re s|, |Im s| from (|q| + |Re q|)/2, the other from Im q
        const bool pos = q.x.h >= 0.f;
        const dfl w = df_scale(m + (pos ? q.x : -q.x), 0.5f);
        const dfl iw = df_rsqrt(w), big = df_mul(w, iw), small = df_scale(df_mul(q.y, iw), 0.5f);
        if (pos) s = {big, small};
        else s = q.y.h < 0.f ? dfc{-small, -big} : dfc{small, big};
    }
    const dfc p = t + s, n = t - s;
    const dfl ap = NumF::abs2(p), an = NumF::abs2(n);
    const bool plus = ap.h >= an.h;
    const dfc den = plus ? p : n;
    const dfl d2 = plus ? ap : an;
    if (!df_seed_ok(d2.h)) return NumF::zero();
    const dfc num = NumF::mul(bc, {den.x, -den.y});
    const dfl r = df_rcp(d2);
    return {df_mul(num.x, r), df_mul(num.y, r)};
}
// An FP64 number in FP32's exponent range (or zero) as h + l, both parts truncated:
// one FP64 instruction instead of four (conversions run on the FP64 pipe).
__device__ __forceinline__ dfl quick_split(double v) {
    const double m = fabs(v);
    if (!mid_range(m)) return {0.f, 0.f};
    const float h = seed_f32(m);
    const double r = m - exact_f64(h);   // >= 0, exact
    const float l = mid_range(r) ? seed_f32(r) : 0.f;
    return v < 0.0 ? dfl{-h, -l} : dfl{h, l};
}
__device__ double2 wilkinson_shift(double2 a, double2 b, double2 c, double2 d) {
    const unsigned hw[8] = {(unsigned)__double2hiint(a.x), (unsigned)__double2hiint(a.y), (unsigned)__double2hiint(b.x),
                            (unsigned)__double2hiint(b.y), (unsigned)__double2hiint(c.x), (unsigned)__double2hiint(c.y),
                            (unsigned)__double2hiint(d.x), (unsigned)__double2hiint(d.y)};
    unsigned ex = 0;   // largest exponent field
#pragma unroll
    for (int i = 0; i < 8; ++i) ex = max(ex, (hw[i] >> 20) & 0x7ffu);
    if (ex < 64u || ex > 1982u) return d;   // zero, non-finite or near the ends of FP64's range
    const double up = __hiloint2double((int)(2046u - ex) << 20, 0), down = __hiloint2double((int)ex << 20, 0);
    auto in = [&](double2 v) { return dfc{quick_split(up * v.x), quick_split(up * v.y)}; };   // 2^(1023-ex) v
    return d - down * dc_to(shift_correction(in(a), in(b), in(c), in(d)));
}
__device__ dfc wilkinson_shift(dfc a, dfc b, dfc c, dfc d) {
    float mx = fmaxf(fmaxf(NumF::abs1(a), NumF::abs1(b)), fmaxf(NumF::abs1(c), NumF::abs1(d)));
    if (!(mx > 1e-30f && mx < 1e30f)) return d;
    const unsigned ex = __float_as_uint(mx) & 0x7f800000u;
    const float up = __uint_as_float(0x7f000000u - ex), down = __uint_as_float(ex);   // 2^(127-e), 2^(e-127)
    auto in = [&](dfc v) { return dfc{df_scale(v.x, up), df_scale(v.y, up)}; };
    const dfc r = shift_correction(in(a), in(b), in(c), in(d));
    return d - dfc{df_scale(r.x, down), df_scale(r.y, down)};
}
__device__ __forceinline__ double2 exceptional_shift(double2 c, double2 d) { return d + make_double2(0.75 * cabs1(c), 0.0); }
__device__ __forceinline__ dfc exceptional_shift(dfc c, dfc d) { return d + dfc{{0.75f * NumF::abs1(c), 0.f}, {0.f, 0.f}}; }

// ---------------------------------------------------------------------------
// Block-cooperative reduction of A (n x n, row stride lda, shared memory, numbers
// of type M::C in 16-byte slots) to Schur form: on return A holds T and Q the
// Schur vectors, both in FP64. Returns 0 on success, 1 if QR failed to
// converge. v: n slots; sh: 8 doubles (sh[4] = Frobenius norm of the Hessenberg
// form on return). lda is odd, so that a column is read without bank conflicts.
//
// Half-warps share each pair of a rotation: lanes 0-15 form the first output of
// 16 pairs, lanes 16-31 the second, after both have read the pair.
template <class M>
__device__ int schur(double2* A64, double2* Q64, int n, int lda, double2* v64, double* sh) {
    using C = typename M::C;
    using R = typename M::R;
    static_assert(sizeof(C) == sizeof(double2), "numbers are converted in place");
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    C* A = reinterpret_cast<C*>(A64);
    C* Q = reinterpret_cast<C*>(Q64);
    C* v = reinterpret_cast<C*>(v64);
    __shared__ C s_cx[2], s_cy[2];
    __shared__ R s_tau;
    __shared__ int s_len, s_l, s_hi, s_fail;
    for (int e = tid; e < n * lda; e += ET) {   // in place: each thread converts its own slots
        const int i = e / lda, j = e % lda;
        if (j < n) {
            const double2 a = A64[e];
            A[e] = M::from(a);
        }
        Q[e] = i == j ? M::one() : M::zero();
    }
    __syncthreads();
    // Householder reduction to upper Hessenberg. A column with nothing below its
    // subdiagonal is skipped, and a reflection spans only the rows up to the
    // column's last nonzero: the projected matrices of eigBiCG are tridiagonal,
    // or after a restart diagonal + coupling arrow + tridiagonal, so most
    // columns need no work. Warp 0 forms the reflection, a column element per lane.
    for (int k = 0; k + 2 < n; ++k) {
        if (warp == 0) {
            int last = k + 1;
            for (int i = k + 1 + lane; i < n; i += 32)
                if (!M::is_zero(A[i * lda + k])) last = i;
            last = __reduce_max_sync(FULL, last);
            const bool work = last > k + 1;
            if (work) {   // v = x + e^{i theta} ||x|| e1, tau = 2/||v||^2
                // The norm in FP64: squares of small entries leave FP32's range. Where they
                // would leave FP64's as well, v is formed from the column times a power of
                // two (its length does not matter).
                bool far = false;
                double up = 1.0;
                if constexpr (M::WIDE) {
                    unsigned f = 0;   // largest exponent field of the column
                    for (int i = k + 1 + lane; i <= last; i += 32) {
                        const double2 x = M::to(A[i * lda + k]);
                        f = max(f, max((unsigned)__double2hiint(x.x) & 0x7ff00000u, (unsigned)__double2hiint(x.y) & 0x7ff00000u) >> 20);
                    }
                    f = __reduce_max_sync(FULL, f);
                    far = f - 543u > 960u;
                    if (far) up = pow2_field(max(2046 - (int)f, 1));
                }
                auto entry = [&](int i) {
                    const double2 x = M::to(A[i * lda + k]);
                    return far ? up * x : x;
                };
                double nrm2 = 0.0;
                for (int i = k + 1 + lane; i <= last; i += 32) nrm2 += NumD::abs2(entry(i));
                nrm2 = warp_sum(nrm2);
                const double alpha = sqrt_fp64(nrm2);
                const double2 x0 = entry(k + 1);
                const double a0 = NumD::abs2(x0);
                double2 ph = cone();
                double ax0 = 0.0;
                if (a0 > 0.0) {
                    const double r0 = rsqrt_fp64(a0);
                    ax0 = a0 * r0;
                    ph = r0 * x0;
                }
                for (int i = k + 1 + lane; i <= last; i += 32) {
                    C x = A[i * lda + k];
                    if (far) x = M::from(entry(i));
                    if (i == k + 1) x = M::from(x0 + alpha * ph);
                    v[i - k - 1] = x;
                }
                if (lane == 0) s_tau = M::rfrom(rcp_fp64(alpha * (alpha + ax0)));
            }
            if (lane == 0) s_len = work ? last - k : 0;
        }
        __syncthreads();
        const int len = s_len;
        if (len == 0) { __syncthreads(); continue; }
        const R tau = s_tau;
        // rows k+1..last of A: A -= tau v (v^H A), columns k..n-1
        for (int j = k + tid; j < n; j += ET) {
            typename M::Sum w;
            for (int i = 0; i < len; ++i) w.add(conj_(v[i]), A[(k + 1 + i) * lda + j]);
            const C tw = M::scale(tau, w.value());
            for (int i = 0; i < len; ++i) A[(k + 1 + i) * lda + j] = M::fms(A[(k + 1 + i) * lda + j], v[i], tw);
        }
        __syncthreads();
        // columns k+1..last of A (all rows) and of Q: X -= tau (X v) v^H; column k below the subdiagonal is zero
        for (int i = tid; i < 2 * n; i += ET) {
            C* row = (i < n ? A + i * lda : Q + (i - n) * lda) + k + 1;
            typename M::Sum u;
            for (int l = 0; l < len; ++l) u.add(row[l], v[l]);
            const C tu = M::scale(tau, u.value());
            for (int l = 0; l < len; ++l) row[l] = M::fms(row[l], tu, conj_(v[l]));
            if (i >= k + 2 && i <= k + len) A[i * lda + k] = M::zero();
        }
        __syncthreads();
    }
    // Frobenius norm for the negligibility tests.
    {
        double f = 0.0;
        for (int e = tid; e < n * n; e += ET) {
            const int i = e / n, j = e % n;
            if (j + 1 >= i) f += M::wide_abs2(A[i * lda + j]);
        }
        f = warp_sum(f);
        __shared__ double s_f[EW];
        if (lane == 0) s_f[warp] = f;
        __syncthreads();
        if (tid == 0) {
            double t = 0.0;
            for (int w = 0; w < EW; ++w) t += s_f[w];
            sh[4] = sqrt(t);
            s_fail = 0;
        }
        __syncthreads();
    }
    const double anorm = sh[4] > 0.0 ? sh[4] : 1.0;
    // Single-shift implicit QR with deflation from the bottom. Warp 0 steers: it
    // scans the subdiagonal (one entry per lane), forms the shift and the first
    // rotation of a sweep, and each next rotation as soon as its own rows of the
    // column update are done.
    const int half = lane >> 4;
    int hi = n - 1, iters = 0, total = 0;   // warp 0 only
    while (true) {
        if (warp == 0) {
            int l = 0;
            bool fail = false;
            while (hi > 0) {
                l = 0;
                for (int base = hi & ~31; base >= 0; base -= 32) {
                    const int i = base + lane;
                    const bool neg = i > 0 && i <= hi &&
                                     M::negligible(A[i * lda + i - 1], A[(i - 1) * lda + i - 1], A[i * lda + i], anorm);
                    const unsigned b = __ballot_sync(FULL, neg);
                    if (b) { l = base + 31 - __clz(b); break; }
                }
                if (l < hi) break;
                --hi;
                iters = 0;
            }
            if (hi > 0) {
                ++iters; ++total;
                fail = iters > 60 || total > 60 * n;
                if (!fail) {
                    const C c = A[hi * lda + hi - 1], d = A[hi * lda + hi];
                    const C mu = iters % 11 == 10 ? exceptional_shift(c, d)
                                                  : wilkinson_shift(A[(hi - 1) * lda + hi - 1], A[(hi - 1) * lda + hi], c, d);
                    C cx, cy;
                    M::givens(A[l * lda + l] - mu, A[(l + 1) * lda + l], cx, cy);
                    __syncwarp();
                    if (lane == 0) {
                        if (l > 0) A[l * lda + l - 1] = M::zero();
                        s_cx[l & 1] = cx;
                        s_cy[l & 1] = cy;
                    }
                }
            }
            if (lane == 0) {
                s_l = l;
                s_hi = fail ? 0 : hi;
                if (fail) s_fail = 1;
            }
        }
        __syncthreads();
        const int l = s_l, h = s_hi;
        if (h <= 0) break;
        for (int k = l; k < h; ++k) {
            const C cx = s_cx[k & 1], cy = s_cy[k & 1];
            // rows k, k+1:  [a; b] <- G [a; b]
            {
                const int j0 = k == l ? l : k - 1;
                const C u = half ? conj_(cx) : cx, w = half ? -conj_(cy) : cy;
                C* row = A + (k + half) * lda;
                const C* oth = A + (k + 1 - half) * lda;
                for (int base = j0 + (warp << 4); base < n; base += 16 * EW) {
                    const int j = base + (lane & 15), jc = min(j, n - 1);
                    C out = M::lin2(u, row[jc], w, oth[jc]);
                    if (half && j < k) out = M::zero();   // the bulge entry that the rotation annihilates
                    __syncwarp();
                    if (j < n) row[j] = out;
                }
            }
            __syncthreads();
            // columns k, k+1 of A (rows 0..min(k+2, h), from the last upwards) and of Q
            // (all rows):  [a, b] <- [a, b] G^H
            {
                const int i1 = min(k + 2, h);
                const C u = half ? cx : conj_(cx), w = half ? -cy : conj_(cy);
                for (int base = warp << 4; base < i1 + 1 + n; base += 16 * EW) {
                    const int t = base + (lane & 15), tc = min(t, i1 + n);
                    C* row = (tc <= i1 ? A + (i1 - tc) * lda : Q + (tc - i1 - 1) * lda) + k;
                    const C out = M::lin2(u, row[half], w, row[1 - half]);
                    __syncwarp();
                    if (t == tc) row[half] = out;
                    // rows k+1 and k+2 are warp 0's first: the next rotation
                    if (base == 0 && k + 1 < h) {
                        __syncwarp();
                        C nx, ny;
                        M::givens(A[(k + 1) * lda + k], A[(k + 2) * lda + k], nx, ny);
                        if (lane == 0) { s_cx[(k + 1) & 1] = nx; s_cy[(k + 1) & 1] = ny; }
                    }
                }
            }
            __syncthreads();
        }
    }
    const int fail = s_fail;
    __syncthreads();
    for (int e = tid; e < n * lda; e += ET) {   // back to FP64, in place
        if (e % lda < n) {
            const C a = A[e], q = Q[e];
            A64[e] = M::to(a);
            Q64[e] = M::to(q);
        }
    }
    __syncthreads();
    return fail;
}

// Order of the eigenvalues on the diagonal of T: smallest |lambda|, then Im, then
// position. Squared moduli order the same way as moduli (ties included). key: n slots.
__device__ void order_eigs(const double2* T, int n, int lda, int* ord, double2* key) {
    for (int i = threadIdx.x; i < n; i += ET) {
        key[i] = make_double2(cabs2(T[i * lda + i]), T[i * lda + i].y);
        ord[i] = i;   // every slot a valid index, should a NaN leave one without a rank
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += ET) {
        const double2 a = key[i];
        int rank = 0;
        for (int j = 0; j < n; ++j) {
            const double2 b = key[j];
            const bool before = b.x < a.x || (b.x == a.x && (b.y < a.y || (b.y == a.y && j < i)));
            rank += before ? 1 : 0;
        }
        ord[rank] = i;
    }
    __syncthreads();
}

constexpr int ES = (MAX_SMALL + 31) / 32;   // elements of a vector per lane

__device__ __forceinline__ double2 shfl_c(double2 a, int src) {
    return make_double2(__shfl_sync(FULL, a.x, src), __shfl_sync(FULL, a.y, src));
}

// Eigenvectors for the eigenvalues T[ord[i], ord[i]], i < nsel, one warp per
// eigenvalue. Y, Z (global), column i of an n x nsel row-major array (ld =
// ldyz). wbuf: n slots per warp. rev: T is of the matrix with rows and columns in
// reverse order (load_reversed); the vectors are written in the original order.
// Substitution in outer-product form: as soon as w_l is known, every lane adds
// its rows' terms with w_l, so a step is two dependent complex multiply-adds
// whatever the length (the row-sum form is a serial chain of that length).
__device__ void eigvecs(const double2* T, const double2* Q, int n, int lda, const int* ord, int nsel,
                        double2* Y, double2* Z, int ldyz, double2* wbuf, double anorm, bool rev) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double smin = fmax(EPS * anorm, 1e-300);
    double2* wb = wbuf + warp * n;
    for (int i = warp; i < nsel; i += EW) {
        const int k = ord[i];
        const double2 lam = T[k * lda + k];
        double2 dinv[ES], vec[2][ES];
#pragma unroll
        for (int t = 0; t < ES; ++t) {
            const int j = lane + 32 * t;
            dinv[t] = czero();
            if (j < n && j != k) {
                double2 d = T[j * lda + j] - lam;
                if (cabs1(d) < smin) d = make_double2(smin, 0.0);
                const double m = fmax(fabs(d.x), fabs(d.y));
                if (m > 1e-14 && m < 1e14) dinv[t] = rcp_fp64(cabs2(d)) * conj_(d);
                else dinv[t] = cdiv(cone(), d);
            }
        }
#pragma unroll
        for (int side = 0; side < 2; ++side) {   // 0: right (rows above k), 1: left (columns right of k)
            double2 s[ES];
#pragma unroll
            for (int t = 0; t < ES; ++t) {
                const int j = lane + 32 * t;
                s[t] = czero();
                if (side == 0 ? j < k : (j > k && j < n)) s[t] = side == 0 ? T[j * lda + k] : T[k * lda + j];
                if (j < n) wb[j] = j == k ? cone() : czero();
            }
            __syncwarp();
            const int steps = side == 0 ? k : n - 1 - k;
            for (int q = 1; q <= steps; ++q) {
                const int l = side == 0 ? k - q : k + q;
                const int own = l >> 5;
                double2 sv = s[0], dv = dinv[0];
#pragma unroll
                for (int t = 1; t < ES; ++t)
                    if (own == t) { sv = s[t]; dv = dinv[t]; }
                double2 w = shfl_c(-(sv * dv), l & 31);
                // |w| above about 1e150 (exponent test): rescale the whole vector
                if (max(__double2hiint(w.x) & 0x7fffffff, __double2hiint(w.y) & 0x7fffffff) > 0x5f100000) {
                    __syncwarp();
                    w = 1e-150 * w;
#pragma unroll
                    for (int t = 0; t < ES; ++t) {
                        const int j = lane + 32 * t;
                        s[t] = 1e-150 * s[t];
                        if (j < n) wb[j] = 1e-150 * wb[j];
                    }
                    __syncwarp();
                }
                if (lane == 0) wb[l] = w;
#pragma unroll
                for (int t = 0; t < ES; ++t) {
                    const int j = lane + 32 * t;
                    if (side == 0 ? 32 * t < l : 32 * t + 31 > l)   // warp-uniform: this slice still has rows to go
                        if (side == 0 ? j < l : (j > l && j < n))
                            s[t] = NumD::fms(s[t], -(side == 0 ? T[j * lda + l] : T[l * lda + j]), w);
                }
            }
            __syncwarp();
            // y = Q y', z = Q conj(w)
            double2 acc[ES];
#pragma unroll
            for (int t = 0; t < ES; ++t) acc[t] = czero();
            const int l0 = side == 0 ? 0 : k, l1 = side == 0 ? k : n - 1;
            for (int l = l0; l <= l1; ++l) {
                const double2 w = side == 0 ? wb[l] : conj_(wb[l]);
#pragma unroll
                for (int t = 0; t < ES; ++t) {
                    const int r = lane + 32 * t;
                    if (32 * t < n && r < n) acc[t] = NumD::fms(acc[t], -Q[r * lda + l], w);
                }
            }
#pragma unroll
            for (int t = 0; t < ES; ++t) vec[side][t] = acc[t];
            __syncwarp();
        }
        // Normalise: ||y|| = 1, largest entry real positive, z^H y = 1.
        double nrm2 = 0.0, best = -1.0;
        int arg = 0;
#pragma unroll
        for (int t = 0; t < ES; ++t) {
            const int r = lane + 32 * t;
            if (r < n) {
                const double a2 = cabs2(vec[0][t]);
                nrm2 += a2;
                if (a2 > best || (rev && a2 == best)) { best = a2; arg = r; }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            nrm2 += __shfl_xor_sync(FULL, nrm2, o);
            const double ob = __shfl_xor_sync(FULL, best, o);
            const int oa = __shfl_xor_sync(FULL, arg, o);
            if (ob > best || (ob == best && (rev ? oa > arg : oa < arg))) { best = ob; arg = oa; }
        }
        double2 pk = vec[0][0];
#pragma unroll
        for (int t = 1; t < ES; ++t)
            if ((arg >> 5) == t) pk = vec[0][t];
        pk = shfl_c(pk, arg & 31);
        // factor = conj(pk)/|pk| / nrm
        const double inrm = nrm2 > 0.0 ? rsqrt_fp64(nrm2) : 1.0;
        const double2 f = best > 0.0 && nrm2 > 0.0 ? (rsqrt_fp64(best) * inrm) * conj_(pk) : make_double2(inrm, 0.0);
        double2 d = czero();
#pragma unroll
        for (int t = 0; t < ES; ++t)
            if (lane + 32 * t < n) {
                vec[0][t] = f * vec[0][t];
                d = d + cdot(vec[1][t], vec[0][t]);
            }
        d = warp_sum(d);
        const double2 g = cabs2(d) > 0.0 ? cdiv(cone(), conj_(d)) : cone();
#pragma unroll
        for (int t = 0; t < ES; ++t) {
            const int r = lane + 32 * t;
            if (r < n) {
                const int ro = rev ? n - 1 - r : r;
                Y[ro * ldyz + i] = vec[0][t];
                Z[ro * ldyz + i] = g * vec[1][t];
            }
        }
        __syncwarp();
    }
    __syncthreads();
}

// Dynamic shared memory of an eigen CTA of capacity nmax. Rows are lda = n | 1
// slots apart (odd: the lanes of a warp read a column without bank conflicts).
__host__ __device__ constexpr int eig_lda(int n) { return n | 1; }
struct EigSmem {
    double2 *A, *Q, *v, *wb;
    double* sh;
    int* ord;
    __device__ EigSmem(char* base, int nmax) {
        A = reinterpret_cast<double2*>(base);
        Q = A + nmax * eig_lda(nmax);
        v = Q + nmax * eig_lda(nmax);
        wb = v + nmax;
        sh = reinterpret_cast<double*>(wb + EW * nmax);
        ord = reinterpret_cast<int*>(sh + 8);
    }
    static size_t bytes(int nmax) {
        return (size_t)(2 * nmax * eig_lda(nmax) + nmax + EW * nmax) * sizeof(double2) + 8 * sizeof(double) +
               nmax * sizeof(int) + 16;
    }
};

// A window's projected matrix H (leading n x n, row stride ldh) with rows and columns
// in reverse order: the tridiagonal part first, then the coupling arrow's hub, then
// the kept Ritz values. In this order the tridiagonal columns are Hessenberg already
// and only the last block (the arrow) needs reflections; in the original order each
// reflection's fill-in moves one row down and all n columns need one of the arrow's
// length (1.4e6 against 0.25e6 cycles in FP64 at n = 60).
__device__ void load_reversed(const double2* H, int ldh, int n, double2* A) {
    for (int e = threadIdx.x; e < n * n; e += ET) A[(n - 1 - e / n) * eig_lda(n) + n - 1 - e % n] = H[(e / n) * ldh + e % n];
    __syncthreads();
}

// Full eigen-solve of the n x n matrix in S.A (row stride eig_lda(n); rev: in reverse
// order). Outputs sorted eigenvalues to lam (n), and vectors for the first nsel.
template <class M>
__device__ int eig_block(EigSmem& S, int n, int nsel, double2* lam, double2* Y, double2* Z, int ldyz, bool rev = false) {
    const int lda = eig_lda(n);
    const int fail = schur<M>(S.A, S.Q, n, lda, S.v, S.sh);
    const double anorm = S.sh[4];
    order_eigs(S.A, n, lda, S.ord, S.v);
    for (int i = threadIdx.x; i < n; i += ET) lam[i] = S.A[S.ord[i] * lda + S.ord[i]];
    __syncthreads();
    if (nsel > 0) eigvecs(S.A, S.Q, n, lda, S.ord, nsel, Y, Z, ldyz, S.wb, anorm, rev);
    return fail;
}

__global__ void __launch_bounds__(ET) small_eig_kernel(int n, const double2* Ain, int lda_in, int nsel,
                                                       double2* lam, double2* Y, double2* Z, int ldyz, int* info) {
    extern __shared__ __align__(16) char smem[];
    EigSmem S(smem, n);
    for (int e = threadIdx.x; e < n * n; e += ET) S.A[(e / n) * eig_lda(n) + e % n] = Ain[(e / n) * lda_in + (e % n)];
    __syncthreads();
    const int fail = eig_block<NumD>(S, n, nsel, lam, Y, Z, ldyz);
    if (threadIdx.x == 0 && info) *info = fail;
}

// LU with complete pivoting of the n x n matrix a (row stride ld), one warp.
// Stops before a pivot p that keep(|p|^2, i) rejects (i = its index); returns the
// pivots kept; rowp / colp: the row and column order. The pivot search reads an
// element per lane; ties go to the first in row-major order.
template <class Keep>
__device__ int warp_lu_complete(double2* a, int n, int ld, int* rowp, int* colp, Keep keep) {
    const int lane = threadIdx.x & 31;
    for (int i = lane; i < n; i += 32) { rowp[i] = i; colp[i] = i; }
    __syncwarp();
    int i = 0;
    for (; i < n; ++i) {
        const int w = n - i;
        double best = -1.0;
        int arg = 0;
        for (int e = lane; e < w * w; e += 32) {
            const double v = cabs2(a[(i + e / w) * ld + i + e % w]);
            if (v > best) { best = v; arg = e; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double ob = __shfl_xor_sync(FULL, best, o);
            const int oa = __shfl_xor_sync(FULL, arg, o);
            if (ob > best || (ob == best && oa < arg)) { best = ob; arg = oa; }
        }
        if (!keep(best, i)) break;
        const int p = i + arg / w, q = i + arg % w;
        if (p != i) {
            for (int c = lane; c < n; c += 32) { const double2 t = a[i * ld + c]; a[i * ld + c] = a[p * ld + c]; a[p * ld + c] = t; }
            if (lane == 0) { const int t = rowp[i]; rowp[i] = rowp[p]; rowp[p] = t; }
        }
        __syncwarp();
        if (q != i) {
            for (int r = lane; r < n; r += 32) { const double2 t = a[r * ld + i]; a[r * ld + i] = a[r * ld + q]; a[r * ld + q] = t; }
            if (lane == 0) { const int t = colp[i]; colp[i] = colp[q]; colp[q] = t; }
        }
        __syncwarp();
        const double2 piv = a[i * ld + i];
        for (int r = i + 1 + lane; r < n; r += 32) a[r * ld + i] = cdiv(a[r * ld + i], piv);
        __syncwarp();
        const int u = w - 1;
        for (int e = lane; e < u * u; e += 32) {
            const int r = i + 1 + e / u, c = i + 1 + e % u;
            a[r * ld + c] = NumD::fms(a[r * ld + c], a[r * ld + i], a[i * ld + c]);
        }
        __syncwarp();
    }
    return i;
}

// ------------------------------------------------------- BiCG-eigen (coeffs)
// Work arrays (global, per problem) for the restart coefficient computation.
struct RestartWork {
    double2 *y1, *z1, *y2, *z2, *HY, *u, *q, *yt, *zt, *lamtmp, *lamtmp2;
    static size_t elems(int m, int nev) {
        const int r = 2 * nev;
        return (size_t)m * nev * 4 + (size_t)m * r * 3 + (size_t)r * r * 2 + 2 * m + 64;
    }
    __device__ RestartWork(double2* base, int m, int nev) {
        const int r = 2 * nev;
        y1 = base; z1 = y1 + m * nev; y2 = z1 + m * nev; z2 = y2 + m * nev;
        HY = z2 + m * nev; u = HY + m * r; q = u + r * r;
        yt = q + r * r; zt = yt + m * r; lamtmp = zt + m * r; lamtmp2 = lamtmp + m;
    }
};

// Algorithm BiCG-eigen in coefficient space, first part: which = 0 computes
// eig(H^(m)) -> y1, z1 (nev smallest); which = 1 computes eig(H^(m-1)) -> y2, z2,
// padded with a zero row. The two parts use disjoint work arrays: the two CTAs
// of a cluster run them at the same time.
__device__ int restart_eigs_part(const double2* H, int ldh, int m, int nev, int which, EigSmem& S,
                                 RestartWork& Wk) {
    const int tid = threadIdx.x;
    const int n = which ? m - 1 : m;
    load_reversed(H, ldh, n, S.A);
    const int fail = eig_block<NumF>(S, n, nev, which ? Wk.lamtmp2 : Wk.lamtmp, which ? Wk.y2 : Wk.y1,
                                     which ? Wk.z2 : Wk.z1, nev, true);
    if (which)
        for (int i = tid; i < nev; i += ET) { Wk.y2[(m - 1) * nev + i] = czero(); Wk.z2[(m - 1) * nev + i] = czero(); }
    __syncthreads();
    return fail;
}

// Second part: bi-orthogonalize, T = zt^H H yt, eig(T), Yc = yt u, Zc = zt q.
// Writes Yc, Zc (m x r, ld = ldc), lam (r); returns r. FP64 throughout.
__device__ int restart_finish_part(const double2* H, int ldh, int m, int nev, double2* Yc, double2* Zc, int ldc,
                                   double2* lam, EigSmem& S, RestartWork& Wk, int* fail_out) {
    const int tid = threadIdx.x;
    // 3. y2 -= y1 (z1^H y2), z2 -= z1 (y1^H z2)   (coefficients in S.A as scratch)
    double2* G1 = S.A;                 // nev x nev : z1^H y2
    double2* G2 = S.A + nev * nev;     // nev x nev : y1^H z2
    double2* Mx = G2 + nev * nev;      // nev x nev : z2^H y2 (3 nev^2 < m^2 slots in all)
    int* rowp = reinterpret_cast<int*>(S.v);
    int* colp = rowp + MAX_M / 2;
    for (int e = tid; e < 2 * nev * nev; e += ET) {
        const bool second = e >= nev * nev;
        const int ee = second ? e - nev * nev : e;
        const int i = ee / nev, j = ee % nev;
        const double2* L = second ? Wk.y1 : Wk.z1;
        const double2* R = second ? Wk.z2 : Wk.y2;
        double2 acc = czero();
        for (int r = 0; r < m; ++r) acc = acc + cdot(L[r * nev + i], R[r * nev + j]);
        (second ? G2 : G1)[i * nev + j] = acc;
    }
    __syncthreads();
    for (int e = tid; e < 2 * m * nev; e += ET) {
        const bool second = e >= m * nev;
        const int ee = second ? e - m * nev : e;
        const int r = ee / nev, j = ee % nev;
        const double2* B = second ? Wk.z1 : Wk.y1;
        const double2* G = second ? G2 : G1;
        double2 acc = czero();
        for (int i = 0; i < nev; ++i) acc = acc + B[r * nev + i] * G[i * nev + j];
        double2* X = second ? Wk.z2 : Wk.y2;
        X[r * nev + j] = X[r * nev + j] - acc;
    }
    __syncthreads();
    // 4. M = z2^H y2, LU with complete pivoting, rank by pivot >= 1e-10
    for (int e = tid; e < nev * nev; e += ET) {
        const int i = e / nev, j = e % nev;
        double2 acc = czero();
        for (int r = 0; r < m; ++r) acc = acc + cdot(Wk.z2[r * nev + i], Wk.y2[r * nev + j]);
        Mx[i * nev + j] = acc;
    }
    __syncthreads();
    __shared__ int s_rank;
    if (tid < 32) {
        const int rank = warp_lu_complete(Mx, nev, nev, rowp, colp, [](double p2, int) { return p2 >= 1e-20; });
        if (tid == 0) s_rank = rank;
    }
    __syncthreads();
    const int rank = s_rank;
    const int r = nev + rank;
    // 5. yt = [y1, y2(:,colp) U^{-1}], zt = [z1, z2(:,rowp) L^{-H}]  (m x r)
    for (int e = tid; e < m * nev; e += ET) {
        const int row = e / nev, i = e % nev;
        Wk.yt[row * r + i] = Wk.y1[row * nev + i];
        Wk.zt[row * r + i] = Wk.z1[row * nev + i];
    }
    for (int j = tid; j < rank; j += ET) G1[j] = cdiv(cone(), Mx[j * nev + j]);   // 1 / U_jj
    __syncthreads();
    for (int row = tid; row < 2 * m; row += ET) {
        const bool zs = row >= m;
        const int rr = zs ? row - m : row;
        double2* out = (zs ? Wk.zt : Wk.yt) + rr * r + nev;
        const double2* in = (zs ? Wk.z2 : Wk.y2) + rr * nev;
        for (int j = 0; j < rank; ++j) {
            double2 acc = in[zs ? rowp[j] : colp[j]];
            for (int i = 0; i < j; ++i) {
                if (!zs) acc = acc - out[i] * Mx[i * nev + j];            // U_{ij}
                else acc = acc - out[i] * conj_(Mx[j * nev + i]);         // conj(L_{ji})
            }
            out[j] = zs ? acc : acc * G1[j];
        }
    }
    __syncthreads();
    // 6. T = zt^H H yt (r x r). H has four or five nonzeros per row but for the arrow's: skip the zeros.
    for (int e = tid; e < m * r; e += ET) {
        const int row = e / r, j = e % r;
        double2 acc = czero();
        for (int l = 0; l < m; ++l) {
            const double2 h = H[row * ldh + l];
            if (h.x != 0.0 || h.y != 0.0) acc = acc + h * Wk.yt[l * r + j];
        }
        Wk.HY[row * r + j] = acc;
    }
    __syncthreads();
    for (int e = tid; e < r * r; e += ET) {
        const int i = e / r, j = e % r;
        double2 acc = czero();
        for (int l = 0; l < m; ++l) acc = acc + cdot(Wk.zt[l * r + i], Wk.HY[l * r + j]);
        S.A[i * eig_lda(r) + j] = acc;
    }
    __syncthreads();
    // 7. eig(T): all r pairs -> u, q, lam
    const int fail = eig_block<NumD>(S, r, r, lam, Wk.u, Wk.q, r);
    // 8. Yc = yt u, Zc = zt q
    for (int e = tid; e < 2 * m * r; e += ET) {
        const bool zs = e >= m * r;
        const int ee = zs ? e - m * r : e;
        const int row = ee / r, j = ee % r;
        const double2* X = zs ? Wk.zt : Wk.yt;
        const double2* C = zs ? Wk.q : Wk.u;
        double2 acc = czero();
        for (int l = 0; l < r; ++l) acc = acc + X[row * r + l] * C[l * r + j];
        (zs ? Zc : Yc)[row * ldc + j] = acc;
    }
    __syncthreads();
    *fail_out = fail;
    return r;
}

// Both CTAs of a two-CTA cluster arrive and wait (release / acquire: global writes
// before it are visible after it in the other CTA).
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// One restart's coefficients by the two CTAs of a cluster: each eigen-solve on its
// own SM, then CTA 0 finishes. fails: two words. Returns r in CTA 0 (fail in *fail),
// -1 in CTA 1.
__device__ int restart_cluster(const double2* H, int ldh, int m, int nev, double2* Yc, double2* Zc, int ldc,
                               double2* lam, EigSmem& S, RestartWork& Wk, int* fails, int* fail) {
    const int which = blockIdx.x & 1;
    const int f = restart_eigs_part(H, ldh, m, nev, which, S, Wk);
    if (threadIdx.x == 0) fails[which] = f;
    __syncthreads();
    cluster_sync();
    if (which) return -1;
    int f2 = 0;
    const int r = restart_finish_part(H, ldh, m, nev, Yc, Zc, ldc, lam, S, Wk, &f2);
    *fail = f2 | __ldcg(fails) | __ldcg(fails + 1);
    return r;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(ET)
    restart_single_kernel(int m, int nev, const double2* H, int* r_out, double2* Yc, double2* Zc, double2* lam,
                          double2* work, int* fails, int* info) {
    extern __shared__ __align__(16) char smem[];
    EigSmem S(smem, m);
    RestartWork Wk(work, m, nev);
    int fail = 0;
    const int r = restart_cluster(H, m, m, nev, Yc, Zc, 2 * nev, lam, S, Wk, fails, &fail);
    if (r >= 0 && threadIdx.x == 0) { *r_out = r; *info = fail; }
}

// Restart of every slot whose window is full (vs == m), one cluster per slot (grid
// 2 nslots): the two eigen-solves, the coefficients and H = diag(lam). The other
// slots' clusters return at once (uniform over the cluster: CTA 0 writes the
// slot's state only after the cluster barrier).
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(ET)
    restart_slots_kernel(SlotState* states, const SlotPtrs* ptrs, double2* work_base, size_t work_stride, int* fails) {
    const int slot = blockIdx.x >> 1;
    SlotState& st = states[slot];
    const SlotPtrs& P = ptrs[slot];
    __shared__ int go;
    if (threadIdx.x == 0) {
        go = (st.status == ST_RUNNING && st.m > 0 && st.vs == st.m);
        if (!go && (blockIdx.x & 1) == 0) st.restart_r = 0;
    }
    __syncthreads();
    if (!go) return;
    extern __shared__ __align__(16) char smem[];
    const int m = st.m, nev = st.nev;
    EigSmem S(smem, m);
    RestartWork Wk(work_base + work_stride * slot, m, nev);
    int fail = 0;
    const int r = restart_cluster(P.H, m, m, nev, P.coefY, P.coefZ, 2 * nev + 1, P.lam, S, Wk, fails + 2 * slot, &fail);
    if (r < 0) return;
    // H = diag(lam)
    for (int e = threadIdx.x; e < m * m; e += ET) {
        const int i = e / m, j = e % m;
        P.H[e] = (i == j && i < r) ? P.lam[i] : czero();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (fail) st.status = ST_BREAKDOWN;
        st.restart_r = r;
        st.vs = r;
        st.restarts += 1;
    }
}

// Final Ritz pairs of a window: eig(H^(vs)), nev smallest, scales folded.
// Block j: slot slot0 + j, outputs at Yc + j ostride, Zc + j ostride, lam + j lstride,
// nout[j] (the windows' final Ritz pairs of several slots at once: each depends
// only on its own window).
__global__ void __launch_bounds__(ET) final_ritz_kernel(SlotState* states, const SlotPtrs* ptrs, int slot0,
                                                        double2* Yc, double2* Zc, double2* lam, int* nout,
                                                        size_t ostride, size_t lstride) {
    const int slot = slot0 + blockIdx.x;
    Yc += blockIdx.x * ostride;
    Zc += blockIdx.x * ostride;
    lam += blockIdx.x * lstride;
    nout += blockIdx.x;
    const SlotState& st = states[slot];
    const SlotPtrs& P = ptrs[slot];
    const int n = st.vs, m = st.m;
    const int nsel = min(st.nev, n);
    if (n == 0) { if (threadIdx.x == 0) *nout = 0; return; }
    extern __shared__ __align__(16) char smem[];
    EigSmem S(smem, n);
    load_reversed(P.H, m, n, S.A);
    eig_block<NumD>(S, n, nsel, lam, Yc, Zc, nsel, true);
    for (int e = threadIdx.x; e < n * nsel; e += ET) {
        const int row = e / nsel;
        Yc[e] = P.vscale[row] * Yc[e];
        Zc[e] = P.wscale[row] * Zc[e];
    }
    if (threadIdx.x == 0) *nout = nsel;
}

// 1/d of a pivot: conj(d) / |d|^2 where the square stays inside FP32's normal
// range, Smith's division otherwise.
__device__ __forceinline__ double2 pivot_rcp(double2 d) {
    const double m = fmax(fabs(d.x), fabs(d.y));
    if (m > 1e-14 && m < 1e14) return rcp_fp64(cabs2(d)) * conj_(d);
    return cdiv(cone(), d);
}

// LU with partial pivoting, one CTA per matrix (blockIdx.x selects one of two of
// the same size), in shared memory. Warp 0 searches the pivot column, a row per
// lane, and forms 1/pivot; the rank-1 updates are bound by FP64 issue.
struct LuJob {
    double2* A;
    int* piv;
    int* info;
};
__global__ void __launch_bounds__(ET) lu_factor_kernel(int n, LuJob j0, LuJob j1, int lda) {
    const LuJob job = blockIdx.x ? j1 : j0;
    extern __shared__ __align__(16) char smem[];
    double2* A = reinterpret_cast<double2*>(smem);
    const int ld = eig_lda(n), tid = threadIdx.x, lane = tid & 31;
    __shared__ int s_p, s_bad;
    __shared__ double2 s_inv;
    for (int e = tid; e < n * n; e += ET) A[(e / n) * ld + e % n] = job.A[(size_t)(e / n) * lda + e % n];
    if (tid == 0) s_bad = 0;
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        if (tid < 32) {
            double best = -1.0;
            int p = k;
            for (int i = k + lane; i < n; i += 32) {
                const double v = cabs2(A[i * ld + k]);
                if (v > best) { best = v; p = i; }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const double ob = __shfl_xor_sync(FULL, best, o);
                const int op = __shfl_xor_sync(FULL, p, o);
                if (ob > best || (ob == best && op < p)) { best = ob; p = op; }
            }
            const double2 inv = best > 0.0 ? pivot_rcp(A[p * ld + k]) : czero();
            if (lane == 0) {
                s_p = p;
                job.piv[k] = p;
                s_inv = inv;
                if (!(best > 0.0)) s_bad = 1;
            }
        }
        __syncthreads();
        const int p = s_p;
        const double2 inv = s_inv;
        if (p != k)
            for (int j = tid; j < n; j += ET) { const double2 t = A[k * ld + j]; A[k * ld + j] = A[p * ld + j]; A[p * ld + j] = t; }
        __syncthreads();
        if (inv.x != 0.0 || inv.y != 0.0)
            for (int i = k + 1 + tid; i < n; i += ET) A[i * ld + k] = A[i * ld + k] * inv;
        __syncthreads();
        const int w = n - k - 1;
        for (int e = tid; e < w * w; e += ET) {
            const int i = k + 1 + e / w, j = k + 1 + e % w;
            A[i * ld + j] = NumD::fms(A[i * ld + j], A[i * ld + k], A[k * ld + j]);
        }
        __syncthreads();
    }
    for (int e = tid; e < n * n; e += ET) job.A[(size_t)(e / n) * lda + e % n] = A[(e / n) * ld + e % n];
    if (tid == 0 && job.info) *job.info = s_bad;
}

// Solve with the LU factors: one warp per right-hand-side column, LS columns per
// CTA, the factors in shared memory. Outer-product substitution: a step is one
// broadcast and one complex multiply-add per lane instead of a serial row sum.
constexpr int LS = 4;
__global__ void __launch_bounds__(32 * LS) lu_solve_kernel(int n, const double2* LU, int lda, const int* piv, int trans,
                                                          int nrhs, double2* B, int ldb) {
    extern __shared__ __align__(16) char smem[];
    double2* F = reinterpret_cast<double2*>(smem);
    const int ld = eig_lda(n), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double2* x = F + n * ld + warp * n;
    int* pv = reinterpret_cast<int*>(F + n * ld + LS * n);
    for (int e = tid; e < n * n; e += 32 * LS) F[(e / n) * ld + e % n] = LU[(size_t)(e / n) * lda + e % n];
    for (int e = tid; e < n; e += 32 * LS) pv[e] = piv[e];
    __syncthreads();
    const int c = blockIdx.x * LS + warp;
    if (c >= nrhs) return;
    for (int i = lane; i < n; i += 32) x[i] = B[(size_t)i * ldb + c];
    __syncwarp();
    if (!trans && lane == 0)   // P b
        for (int k = 0; k < n; ++k) {
            const int p = pv[k];
            if (p != k) { const double2 t = x[k]; x[k] = x[p]; x[p] = t; }
        }
    __syncwarp();
    double2 s[ES], dinv[ES];
#pragma unroll
    for (int t = 0; t < ES; ++t) {
        const int j = lane + 32 * t;
        s[t] = dinv[t] = czero();
        if (j < n) {
            s[t] = x[j];
            const double2 d = pivot_rcp(F[j * ld + j]);
            dinv[t] = trans ? conj_(d) : d;
        }
    }
    // not transposed: L y = b (unit), then U x = y; transposed (A^H = U^H L^H P):
    // U^H y = b, then L^H w = y (unit), x = P^T w
#pragma unroll
    for (int pass = 0; pass < 2; ++pass) {
        const bool divide = trans ? pass == 0 : pass == 1;
        for (int q = 0; q < n; ++q) {
            const int l = pass == 0 ? q : n - 1 - q;
            const int own = l >> 5;
            double2 v = s[0], dv = dinv[0];
#pragma unroll
            for (int t = 1; t < ES; ++t)
                if (own == t) { v = s[t]; dv = dinv[t]; }
            if (divide) v = v * dv;
            const double2 w = shfl_c(v, l & 31);
#pragma unroll
            for (int t = 0; t < ES; ++t) {
                const int j = lane + 32 * t;
                if (j == l) s[t] = w;
                if (32 * t < n && (pass == 0 ? (j > l && j < n) : j < l))
                    s[t] = NumD::fms(s[t], trans ? conj_(F[l * ld + j]) : F[j * ld + l], w);
            }
        }
    }
#pragma unroll
    for (int t = 0; t < ES; ++t)
        if (lane + 32 * t < n) x[lane + 32 * t] = s[t];
    __syncwarp();
    if (trans && lane == 0)   // P^T w
        for (int k = n - 1; k >= 0; --k) {
            const int p = pv[k];
            if (p != k) { const double2 t = x[k]; x[k] = x[p]; x[p] = t; }
        }
    __syncwarp();
    for (int i = lane; i < n; i += 32) B[(size_t)i * ldb + c] = x[i];
}
size_t lu_factor_smem(int n) { return (size_t)n * eig_lda(n) * sizeof(double2); }
size_t lu_solve_smem(int n) { return (size_t)(n * eig_lda(n) + LS * n) * sizeof(double2) + n * sizeof(int); }

// One factor of P A = L U applied to B (n x nrhs, or nrows x n for LU_RIGHT_U),
// one thread per column (per row for LU_RIGHT_U):
//   LU_LEFT_PL : B <- L^{-1} P B        LU_LEFT_U : B <- U^{-1} B
//   LU_RIGHT_U : B <- B U^{-1}          LU_LEFT_LH: B <- P^T L^{-H} B
__global__ void lu_part_kernel(int n, const double2* LU, int lda, const int* piv, int part, int ncols, double2* B,
                               int ldb) {
    for (int c = threadIdx.x; c < ncols; c += blockDim.x) {
        if (part == LU_LEFT_PL) {
            for (int k = 0; k < n; ++k) {
                const int p = piv[k];
                if (p != k) { double2 t = B[k * ldb + c]; B[k * ldb + c] = B[p * ldb + c]; B[p * ldb + c] = t; }
            }
            for (int i = 0; i < n; ++i) {
                double2 acc = B[i * ldb + c];
                for (int j = 0; j < i; ++j) acc = acc - LU[i * lda + j] * B[j * ldb + c];
                B[i * ldb + c] = acc;
            }
        } else if (part == LU_LEFT_U) {
            for (int i = n - 1; i >= 0; --i) {
                double2 acc = B[i * ldb + c];
                for (int j = i + 1; j < n; ++j) acc = acc - LU[i * lda + j] * B[j * ldb + c];
                B[i * ldb + c] = cdiv(acc, LU[i * lda + i]);
            }
        } else if (part == LU_RIGHT_U) {   // row c: x U = b, x_j = (b_j - sum_{i<j} x_i U_ij) / U_jj
            double2* row = B + (size_t)c * ldb;
            for (int j = 0; j < n; ++j) {
                double2 acc = row[j];
                for (int i = 0; i < j; ++i) acc = acc - row[i] * LU[i * lda + j];
                row[j] = cdiv(acc, LU[j * lda + j]);
            }
        } else {   // LU_LEFT_LH: L^H w = b (unit upper), then x = P^T w
            for (int i = n - 1; i >= 0; --i) {
                double2 acc = B[i * ldb + c];
                for (int j = i + 1; j < n; ++j) acc = acc - conj_(LU[j * lda + i]) * B[j * ldb + c];
                B[i * ldb + c] = acc;
            }
            for (int k = n - 1; k >= 0; --k) {
                const int p = piv[k];
                if (p != k) { double2 t = B[k * ldb + c]; B[k * ldb + c] = B[p * ldb + c]; B[p * ldb + c] = t; }
            }
        }
    }
}

// Rank-revealing selection on a small square block B (n <= 32, row-major, ld):
// LU with complete pivoting on a copy, stopped at the first pivot below
// tau * |first pivot|. out[0] = r (pivots kept), out[1 + i] = row index of pivot
// i, out[1 + n + i] = its column index (i < r). One warp.
__global__ void __launch_bounds__(32) pivot_select_kernel(int n, const double2* B, int ld, double tau, int* out) {
    __shared__ double2 a[32 * 33];
    __shared__ int rowp[32], colp[32];
    for (int e = threadIdx.x; e < n * n; e += 32) a[(e / n) * 33 + e % n] = B[(size_t)(e / n) * ld + e % n];
    __syncwarp();
    double first = 0.0;
    const int r = warp_lu_complete(a, n, 33, rowp, colp, [&](double p2, int i) {
        if (i == 0) first = p2;
        return p2 > tau * tau * first && p2 != 0.0;
    });
    if (threadIdx.x == 0) out[0] = r;
    for (int i = threadIdx.x; i < n; i += 32) { out[1 + i] = rowp[i]; out[1 + n + i] = colp[i]; }
}

}  // namespace

// ------------------------------------------------------------------ launchers
static cudaError_t set_smem(const void* fn, size_t bytes) {
    if (bytes > 48 * 1024) return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    return cudaSuccess;
}

cudaError_t prepare_eig_kernels() {
    cudaError_t e;
    if ((e = set_smem((const void*)small_eig_kernel, EigSmem::bytes(MAX_SMALL))) != cudaSuccess) return e;
    if ((e = set_smem((const void*)restart_single_kernel, EigSmem::bytes(MAX_M))) != cudaSuccess) return e;
    if ((e = set_smem((const void*)restart_slots_kernel, EigSmem::bytes(MAX_M))) != cudaSuccess) return e;
    if ((e = set_smem((const void*)lu_factor_kernel, lu_factor_smem(MAX_SMALL))) != cudaSuccess) return e;
    if ((e = set_smem((const void*)lu_solve_kernel, lu_solve_smem(MAX_SMALL))) != cudaSuccess) return e;
    return set_smem((const void*)final_ritz_kernel, EigSmem::bytes(MAX_M));
}

size_t eig_work_elems() {
    return RestartWork::elems(MAX_M, MAX_M / 2);
}

cudaError_t launch_small_eig(int n, const double2* A, int lda, int nsel, double2* lam, double2* Y, double2* Z,
                             int ldyz, int* info, cudaStream_t st) {
    if (n < 1 || n > MAX_SMALL) return cudaErrorInvalidValue;
    // The kernel's shared-memory limit is only ever set to the largest size
    // (bytes(MAX_SMALL)); a smaller per-call value would lower it for every
    // other caller of this kernel, including the allocation-free entry point.
    cudaError_t e = set_smem((const void*)small_eig_kernel, EigSmem::bytes(MAX_SMALL));
    if (e != cudaSuccess) return e;
    const size_t sm = EigSmem::bytes(n);
    small_eig_kernel<<<1, ET, sm, st>>>(n, A, lda, nsel, lam, Y, Z, ldyz, info);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_restart_coeffs_single(int m, int nev, const double2* H, int* r, double2* Yc, double2* Zc,
                                         double2* lam, int* info, double2* w, cudaStream_t st) {
    if (m < 3 || m > MAX_M || 2 * nev >= m || nev < 1) return cudaErrorInvalidValue;
    const size_t sm = EigSmem::bytes(m);
    cudaError_t e = set_smem((const void*)restart_single_kernel, EigSmem::bytes(MAX_M));   // never lowered
    if (e != cudaSuccess) return e;
    int* fails = reinterpret_cast<int*>(w + eig_work_elems() - 4);   // inside the area's slack
    restart_single_kernel<<<2, ET, sm, st>>>(m, nev, H, r, Yc, Zc, lam, w, fails, info);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_restart_coeffs(SlotState* states, const SlotPtrs* ptrs, int nslots, double2* w,
                                  cudaStream_t st) {
    // Per-slot work stride: capacity for the largest window; the dynamic shared
    // memory opt-in is done once by prepare_eig_kernels (this launcher runs under
    // graph capture).
    const size_t stride = eig_work_elems();
    int* fails = reinterpret_cast<int*>(w + stride * MAX_SLOTS);   // 2 ints per slot after the slot work areas
    size_t sm = EigSmem::bytes(MAX_M);
    restart_slots_kernel<<<2 * nslots, ET, sm, st>>>(states, ptrs, w, stride, fails);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_final_ritz_slots(SlotState* states, const SlotPtrs* ptrs, int slot0, int nslots, double2* Yc,
                                    double2* Zc, double2* lam, int* nout, size_t ostride, size_t lstride,
                                    cudaStream_t st) {
    if (nslots < 1 || nslots > MAX_SLOTS) return cudaErrorInvalidValue;
    size_t sm = EigSmem::bytes(MAX_M);
    final_ritz_kernel<<<nslots, ET, sm, st>>>(states, ptrs, slot0, Yc, Zc, lam, nout, ostride, lstride);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_lu_factor(int n, double2* A, int lda, int* piv, int* info, cudaStream_t st, double2* A2,
                             int* piv2, int* info2) {
    if (n < 1 || n > MAX_SMALL) return cudaErrorInvalidValue;
    lu_factor_kernel<<<A2 ? 2 : 1, ET, lu_factor_smem(n), st>>>(n, LuJob{A, piv, info}, LuJob{A2, piv2, info2}, lda);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_lu_solve(int n, const double2* LU, int lda, const int* piv, int trans, int nrhs, double2* B,
                            int ldb, cudaStream_t st) {
    if (n < 1 || n > MAX_SMALL || nrhs < 1) return cudaErrorInvalidValue;
    lu_solve_kernel<<<(nrhs + LS - 1) / LS, 32 * LS, lu_solve_smem(n), st>>>(n, LU, lda, piv, trans, nrhs, B, ldb);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_lu_part(int n, const double2* LU, int lda, const int* piv, int part, int ncols, double2* B,
                           int ldb, cudaStream_t st) {
    lu_part_kernel<<<1, 128, 0, st>>>(n, LU, lda, piv, part, ncols, B, ldb);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_pivot_select(int n, const double2* B, int ld, double tau, int* out, cudaStream_t st) {
    if (n < 1 || n > 32) return cudaErrorInvalidValue;
    pivot_select_kernel<<<1, 32, 0, st>>>(n, B, ld, tau, out);
    count_launches(1);
    return cudaGetLastError();
}

// ============================================================================
// Allocation-free variant of the small eigen-solver (no counterpart in the paper).
//
// lqcd_small_eig stages its operands through cudaMalloc'd buffers. Some callers
// cannot allocate device memory at the point where they need an eigen-solve:
// host applications that hand all device memory to their own pool or fixed
// budget up front, and latency-critical loops where the implicit device
// synchronisation of cudaMalloc/cudaFree would stall work on other streams.
// lqcd_small_eig_noalloc takes device pointers for the input and every output;
// its working set is the kernel's shared memory, and its status word lives in
// the file-scope device variable below. The word is shared by all calls on a
// device and cleared by each: calls whose kernels overlap on the GPU (different
// streams, or host threads) race on it.
// The per-device set-up (the word's address, the shared-memory limit) is kept
// for the life of the process: a cudaDeviceReset between calls is not supported.
// Every other launcher of the same kernel keeps its shared-memory limit at the
// maximum, so no other call can lower it below what this entry point needs.
namespace {

constexpr int NOALLOC_MAX_N = MAX_SMALL;

static __device__ int g_noalloc_info;

struct NoAllocSetup {
    bool ready = false;
    int* info = nullptr;   // device address of g_noalloc_info on this device
};
constexpr int NOALLOC_MAX_DEVICES = 64;
NoAllocSetup g_noalloc_dev[NOALLOC_MAX_DEVICES];
std::mutex g_noalloc_mutex;

// Once per device, with that device current: the word's device address and the
// kernel's shared-memory opt-in.
cudaError_t noalloc_setup(int dev, int** info) {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    NoAllocSetup& d = g_noalloc_dev[dev];
    if (!d.ready) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_info);
        if (e != cudaSuccess) return e;
        e = set_smem((const void*)small_eig_kernel, EigSmem::bytes(NOALLOC_MAX_N));
        if (e != cudaSuccess) return e;
        d.info = reinterpret_cast<int*>(p);
        d.ready = true;
    }
    *info = d.info;
    return cudaSuccess;
}

}  // namespace
}  // namespace lqcd

extern "C" lqcd_status lqcd_small_eig_noalloc(int n, const double* C, double* evals, double* Y, double* Z,
                                              void* stream) {
    using namespace lqcd;
    if (n < 1 || n > NOALLOC_MAX_N || !C || !evals || (Y == nullptr) != (Z == nullptr)) return LQCD_ERR_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES) return LQCD_ERR_CUDA;
    int* info = nullptr;
    if (noalloc_setup(dev, &info) != cudaSuccess) return LQCD_ERR_CUDA;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const int nsel = Y ? n : 0;
    if (cudaMemsetAsync(info, 0, sizeof(int), st) != cudaSuccess) return LQCD_ERR_CUDA;
    (void)cudaGetLastError();   // an earlier, unrelated launch error is not this call's
    small_eig_kernel<<<1, ET, EigSmem::bytes(n), st>>>(n, reinterpret_cast<const double2*>(C), n, nsel,
                                                       reinterpret_cast<double2*>(evals), reinterpret_cast<double2*>(Y),
                                                       reinterpret_cast<double2*>(Z), n, info);
    count_launches(1);
    if (cudaPeekAtLastError() != cudaSuccess) { (void)cudaGetLastError(); return LQCD_ERR_CUDA; }
    int hinfo = 0;
    if (cudaMemcpyAsync(&hinfo, info, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return LQCD_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return LQCD_ERR_CUDA;
    return hinfo ? LQCD_ERR_NOCONV : LQCD_OK;
}
