// Vector units, gamma5 helpers and the per-iteration scalar bookkeeping shared by
// the BiCG / BiCGStab iteration kernels (kernels.cu, reliable.cu).
#pragma once
#include "reduce.cuh"

namespace lqcd {

// Vector units: two complex numbers (one float4 in FP32, two double2 in FP64).
template <typename S> struct Unit;
template <> struct Unit<float> {
    float2 a, b;
    __device__ __forceinline__ static Unit load(const void* p, size_t u) {
        float4 t = reinterpret_cast<const float4*>(p)[u];
        return Unit{make_float2(t.x, t.y), make_float2(t.z, t.w)};
    }
    __device__ __forceinline__ void store(void* p, size_t u) const {
        reinterpret_cast<float4*>(p)[u] = make_float4(a.x, a.y, b.x, b.y);
    }
};
template <> struct Unit<double> {
    double2 a, b;
    __device__ __forceinline__ static Unit load(const void* p, size_t u) {
        const double2* d = reinterpret_cast<const double2*>(p);
        return Unit{d[2 * u], d[2 * u + 1]};
    }
    __device__ __forceinline__ void store(void* p, size_t u) const {
        double2* d = reinterpret_cast<double2*>(p);
        d[2 * u] = a; d[2 * u + 1] = b;
    }
};

// Compensated FP32 accumulation of a complex sum (Knuth's two-sum per term), for
// the gamma5 variant's inner products rho = r^H gamma5 r and sigma = p^H gamma5 A p:
// their terms have both signs and cancel down to about ||r||^2 / sqrt(N), so a
// plain FP32 sum would lose three to four digits of them. The per-thread value
// goes to FP64 block and cross-block sums.
struct CompC {
    float sx = 0.f, cx = 0.f, sy = 0.f, cy = 0.f;
    __device__ __forceinline__ static void add1(float& s, float& c, float v) {
        const float t = s + v, bp = t - s;
        c += (s - (t - bp)) + (v - bp);
        s = t;
    }
    __device__ __forceinline__ void add(float2 v) { add1(sx, cx, v.x); add1(sy, cy, v.y); }
    __device__ __forceinline__ double2 value() const { return make_double2((double)sx + cx, (double)sy + cy); }
};

// Block and cross-block sum of (z, (a, b)) per slot: over the warp in the storage
// precision, or (gamma5 variant with FP32 storage, compensated z) in FP64 throughout.
template <typename S>
__device__ __forceinline__ bool reduce2(const SlotPtrs& P, int kind, bool comp, const CompC& cz, const Acc<S>& acc,
                                        double2 (&tot)[2], unsigned nblocks, unsigned bid) {
    if (comp) {
        double2 v[2] = {cz.value(), make_double2((double)acc.a, (double)acc.b)};
        return reduce_slot<2>(P, kind, v, tot, nblocks, bid);
    }
    cplx<S> v[2];
    acc.to(v);
    return reduce_slot<2>(P, kind, v, tot, nblocks, bid);
}

// gamma5 = diag(1, 1, -1, -1) on a vector unit: units u < N/4 hold spins 0 and 1
// (chunks q = 0..2 of the field layout), the rest spins 2 and 3.
template <typename S> __device__ __forceinline__ Unit<S> g5u(Unit<S> v, size_t u, size_t N) {
    if (u >= N / 4) { v.a = -v.a; v.b = -v.b; }
    return v;
}

// Scalar bookkeeping at the end of an iteration (one thread; after the residual
// update, or after the reliable update where one was asked for):
// beta_{j-1} = rho_j / rho_{j-1}; window append v = r/||r||, w = (||r||/conj(rho)) rhat;
// tridiagonal entries of H (Algorithm eigBiCG, step 3); iteration counters.
// Not inlined: its registers would cut the occupancy of the vector kernels whose last
// block calls it.
static __device__ __noinline__ void bicg_scalars(SlotState& st, const SlotPtrs& P) {
    const double2 beta = cdiv_fp64(st.rho_new, st.rho);
    if (st.m > 0) {
        const int k = st.vs;   // 0-based index of the appended vector
        const int m = st.m;
        P.vscale[k] = rcp_fp64(st.rnorm);
        P.wscale[k] = cdiv_fp64(make_double2(st.rnorm, 0.0), conj_(st.rho));
        const double2 inv_a = cdiv_fp64(make_double2(1.0, 0.0), st.alpha);
        double2 diag = inv_a;
        if (st.iter > 0) diag = diag + cdiv_fp64(st.beta_prev, st.alpha_prev);
        P.H[k * m + k] = diag;
        if (k + 1 < m) {
            P.H[k * m + k + 1] = -(st.rnorm * rcp_fp64(st.rnorm_new)) * cdiv_fp64(beta, st.alpha);
            P.H[(k + 1) * m + k] = -(st.rnorm_new * P.vscale[k]) * inv_a;
        }
        st.vs = k + 1;
    }
    st.beta = st.fresh_dir ? make_double2(0.0, 0.0) : beta;
    st.fresh_dir = 0;
    st.alpha_prev = st.alpha;
    st.beta_prev = beta;
    st.rho = st.rho_new;
    st.rnorm = st.rnorm_new;
    st.iter += 1;
    if (st.status == ST_RUNNING) {
        if (st.iter >= st.maxiter) st.status = ST_NOCONV;
        else if (!abs_at_least(st.rho, BREAK_TOL, st.rhat_norm, st.rnorm)) st.status = ST_BREAKDOWN;
    }
    if (st.status != ST_RUNNING) st.live = 0;
    // the direction update adds the owed alpha p; a slot that stops here keeps it
    // owed for the final fold
    if (st.status == ST_RUNNING) { st.x_dir = st.x_owed; st.x_owed = 0; }
    else st.x_dir = 0;
}

// beta = (rho' / rho) (alpha / omega); counters; maxiter and breakdown (rho or omega).
static __device__ __noinline__ void stab_scalars(SlotState& st) {
    st.iter += 1;
    const bool om0 = cabs2(st.omega) == 0.0;
    if (!om0) st.beta = cdiv_fp64(st.rho_new, st.rho) * cdiv_fp64(st.alpha, st.omega);
    st.rho = st.rho_new;
    st.rnorm = st.rnorm_new;
    if (st.status == ST_RUNNING) {
        if (st.iter >= st.maxiter) st.status = ST_NOCONV;
        else if (om0 || !abs_at_least(st.rho, BREAK_TOL, st.rhat_norm, st.rnorm)) st.status = ST_BREAKDOWN;
    }
    if (st.status != ST_RUNNING) st.live = 0;
}

}  // namespace lqcd
