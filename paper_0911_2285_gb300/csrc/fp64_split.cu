// FP64 operator on small grids: the eight neighbour terms of a site on eight threads.
//
// What bounds it: each quarter of an SM issues one FP64 warp instruction per 64 clocks,
// and a site takes about 950 of them. With a site per thread a 4^4 operator pair has 16
// warps, so 16 of the 608 quarters work for 36 us. Here a block of four warps (one per
// quarter) takes SPLIT_SITES sites: warp mu, lanes 0-15 the forward and lanes 16-31 the
// backward neighbour of direction mu; the terms meet in shared memory and are added in
// the order of the site-per-thread kernels (the same bits), one component of one site
// per thread and step. The two kinds of lane share one code path: the backward link is
// the conjugate transpose, the projector's sign flips the lower spinor half. Per warp
// about 150 instructions instead of 950 for twice the sites. Measured, pair on
// 4^4: 36.5 -> 13 us (5 of them the reduction of sigma); A on 8^4: 31 -> 7.4 us.
#include "dslash.cuh"
#include "fp64.cuh"
#include "kernels.cuh"
#include "reduce.cuh"
#include "vec.cuh"

namespace lqcd {
namespace {

constexpr int SPLIT_SITES = 16, SPLIT_THREADS = 128, SPLIT_ITEMS = 12 * SPLIT_SITES;

__device__ __forceinline__ double2 flip(double2 a, int sign_bit) {
    return make_double2(__hiloint2double(__double2hiint(a.x) ^ sign_bit, __double2loint(a.x)),
                        __hiloint2double(__double2hiint(a.y) ^ sign_bit, __double2loint(a.y)));
}

// o = (1 + sg M_mu) hop term of site s from its forward (bwd = 0) or backward neighbour.
template <int MU>
__device__ __forceinline__ void split_term(const Geom& g, const LinksD& U, const void* in, int s, bool bwd, int sign_bit,
                                           double2 (&o)[12]) {
    const int n = bwd ? g.bwd(s, MU) : g.fwd(s, MU);
    double2 psi[12], h[2][3], uh[2][3], u[3][3], w[3][3];
    U.load(MU, bwd ? n : s, u);
    Field<double>::load(in, g.V, n, psi);
#pragma unroll
    for (int c = 6; c < 12; ++c) psi[c] = flip(psi[c], sign_bit);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) w[r][c] = bwd ? conj_(u[c][r]) : u[r][c];
    project<MU, +1>(psi, h);
    su3_mul(w, h, uh);
    reconstruct<MU, +1, true>(uh, o);
#pragma unroll
    for (int c = 6; c < 12; ++c) o[c] = flip(o[c], sign_bit);
}

// The block's terms of sites s0 .. s0 + SPLIT_SITES - 1 in sm[direction][component][site].
__device__ __forceinline__ void split_terms(const Geom& g, const LinksD& U, const void* in, int s0, bool dag,
                                            double2 (*sm)[12][SPLIT_SITES]) {
    const int mu = threadIdx.x >> 5, site = threadIdx.x & 15, s = s0 + site;
    const bool bwd = threadIdx.x & 16;
    if (s < g.V) {
        const int sign_bit = bwd != dag ? 0 : (int)0x80000000;   // 1 - M forward, 1 + M backward; A^+ the other way
        double2 o[12];
        if (mu == 0) split_term<0>(g, U, in, s, bwd, sign_bit, o);
        else if (mu == 1) split_term<1>(g, U, in, s, bwd, sign_bit, o);
        else if (mu == 2) split_term<2>(g, U, in, s, bwd, sign_bit, o);
        else split_term<3>(g, U, in, s, bwd, sign_bit, o);
#pragma unroll
        for (int c = 0; c < 12; ++c) sm[2 * mu + (bwd ? 1 : 0)][c][site] = o[c];
    }
    __syncthreads();
}
__device__ __forceinline__ double2 split_sum(const double2 (*sm)[12][SPLIT_SITES], int c, int site) {
    double2 a = sm[0][c][site];
#pragma unroll
    for (int d = 1; d < 8; ++d) a = a + sm[d][c][site];
    return a;
}
// Component c of site s in the field layout.
__device__ __forceinline__ size_t split_elem(int V, int s, int c) { return ((size_t)(c >> 1) * V + s) * 2 + (c & 1); }

template <bool RES>
__global__ void __launch_bounds__(SPLIT_THREADS) apply_split_kernel(Geom g, const double2* links, double kappa,
                                                                    const double2* src, double2* dst, const double2* aux,
                                                                    int dagger, int nf) {
    __shared__ double2 sm[8][12][SPLIT_SITES];
    const size_t off = (size_t)(blockIdx.x % nf) * 12 * g.V;
    const int s0 = blockIdx.x / nf * SPLIT_SITES;
    split_terms(g, LinksD{links, g.V}, src + off, s0, dagger != 0, sm);
    for (int i = threadIdx.x; i < SPLIT_ITEMS; i += SPLIT_THREADS) {
        const int site = i & 15, c = i >> 4, s = s0 + site;
        if (s >= g.V) continue;
        const size_t e = off + split_elem(g.V, s, c);
        double2 a = src[e] - kappa * split_sum(sm, c, site);
        if (RES) a = aux[e] - a;
        dst[e] = a;
    }
}

// A p (even jobs, with sigma = (phat, A p) and the norms of its breakdown test) and
// A^+ phat (odd jobs) of each slot: the contract of the site-per-thread matvec kernel.
__global__ void __launch_bounds__(SPLIT_THREADS) matvec_split_kernel(Geom g, const double2* links, double kappa,
                                                                     SlotState* states, const SlotPtrs* ptrs, int njobs) {
    __shared__ double2 sm[8][12][SPLIT_SITES];
    __shared__ int go;
    const int job = blockIdx.x % njobs, sblock = blockIdx.x / njobs, which = job & 1;
    SlotState& st = states[job >> 1];
    const SlotPtrs& P = ptrs[job >> 1];
    // One thread reads the status for the block: the last even block may store a breakdown
    // while an odd block, which it does not wait for, still starts; threads that read it
    // themselves could part before the barrier in split_terms.
    if (threadIdx.x == 0) go = st.status == ST_RUNNING && !st.stab;
    __syncthreads();
    if (!go) return;
    const int par = st.iter & 1, s0 = sblock * SPLIT_SITES;
    const double2* src = reinterpret_cast<const double2*>(which ? P.phat : P.p);
    const double2* ph = reinterpret_cast<const double2*>(P.phat);
    double2* dst = reinterpret_cast<double2*>(which ? P.Ahp[par] : P.Ap[par]);
    split_terms(g, LinksD{links, g.V}, src, s0, which != 0, sm);
    Acc<double> sacc;   // sigma, |phat|^2, |Ap|^2
    CompC none;
    for (int i = threadIdx.x; i < SPLIT_ITEMS; i += SPLIT_THREADS) {
        const int site = i & 15, c = i >> 4, s = s0 + site;
        if (s >= g.V) continue;
        const size_t e = split_elem(g.V, s, c);
        const double2 a = src[e] - kappa * split_sum(sm, c, site);
        dst[e] = a;
        if (!which) {
            const double2 h = ph[e];
            sacc.z = cdot_acc(sacc.z, h, a);
            sacc.a = abs2_acc(sacc.a, h);
            sacc.b = abs2_acc(sacc.b, a);
        }
    }
    if (which) return;
    double2 tot[2];
    if (reduce2<double>(P, CNT_MATVEC, false, none, sacc, tot, gridDim.x / njobs, sblock) && threadIdx.x == 0)
        finish_sigma(st, tot[0], tot[1].x, tot[1].y, 2);
}

}  // namespace

// Up to two site-per-thread warps per SM: more than half of the chip's quarters idle
// (4^4 pair 36.5 -> 13 us). Above four the site-per-thread form keeps every FP64 pipe
// busy with less work in all (four warps of 150 instructions per 16 sites against one of 950 per 32);
// between the two both take as long.
bool fp64_split_ok(size_t V, int jobs) { return (V + 31) / 32 * jobs <= 2 * 152; }

cudaError_t launch_apply_split(const Geom& g, const void* links64, double kappa, const void* in, void* out,
                               const double2* aux, int dagger, int nf, cudaStream_t st) {
    const int grid = (g.V + SPLIT_SITES - 1) / SPLIT_SITES * nf;
    const double2* U = reinterpret_cast<const double2*>(links64);
    const double2* src = reinterpret_cast<const double2*>(in);
    double2* dst = reinterpret_cast<double2*>(out);
    if (aux) apply_split_kernel<true><<<grid, SPLIT_THREADS, 0, st>>>(g, U, kappa, src, dst, aux, dagger, nf);
    else apply_split_kernel<false><<<grid, SPLIT_THREADS, 0, st>>>(g, U, kappa, src, dst, aux, dagger, nf);
    return cudaGetLastError();
}

cudaError_t launch_matvec_split(const Geom& g, const void* links64, double kappa, SlotState* states, const SlotPtrs* ptrs,
                                int nslots, cudaStream_t st) {
    const int grid = (g.V + SPLIT_SITES - 1) / SPLIT_SITES * 2 * nslots;
    matvec_split_kernel<<<grid, SPLIT_THREADS, 0, st>>>(g, reinterpret_cast<const double2*>(links64), kappa, states, ptrs,
                                                        2 * nslots);
    return cudaGetLastError();
}

}  // namespace lqcd
