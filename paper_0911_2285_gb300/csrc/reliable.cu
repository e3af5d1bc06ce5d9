// Reliable update of the mixed- and double-precision iterations (Sleijpen and van
// der Vorst): for the slots whose residual update asked for it,
//   x_hi += x_lo (+ the owed alpha p), x_lo = 0;
//   r = b - A x_hi in FP64-class arithmetic;
//   converged if ||r|| <= tol ||b||, else the recursive residual becomes r (the
//   gamma5 variant's shadow follows) and rho is recomputed;
//   the scalars that end the iteration.
//
// One kernel, whose blocks share the work of however many slots need it and return at once
// when none does, which is all but about six times in a solve (one thread per site in four
// kernels took 50 us of a 2.7 ms iteration at 24^3 x 64 in empty launches and 8 of 39 us on
// small lattices). It has two (even-odd: three) phases, each reading neighbours that the
// one before wrote:
//  * up to RU_COOP units of work: one cooperative launch with a grid barrier between the
//    phases, about 1.5 us per iteration less than a launch per phase (FP64 solve on 4^4
//    2.33 ms, 2.42 the other way; 10x6x14x9 mixed 5.25 and 5.31);
//  * above: a launch per phase. A cooperative launch starts only when all its blocks fit on
//    the GPU at once, so that a large one waited in every iteration for room beside the
//    kernels of another context: 16^3 x 32 solves beside 24^3 x 64 ones 343 ms, now 264
//    (four kernels: 284); alone 15.7 and 15.9, even-odd batches 51.3 and 51.8. At the line
//    (8^4, 8 slots, 256 units) 125 ms beside, 143 with four kernels.
//
// Double-float residual: about 10^4 FP32 instructions per site. Written out for
// eight hops that is 175 KB of code, more than the instruction caches hold: ncu
// showed 6.5 of 13.8 stall cycles per issue as "no instruction" and 21 % FMA
// pipe use. Here one loop body serves all eight hops, with the direction's
// sources and swaps as selects and its signs as FMA factors; and the FP64 pipe,
// which fold, residual and rounding to FP32 filled with conversions (44 % busy),
// keeps only the additions (fp64.cuh). Fold, residual and replacement of one
// field at 24^3 x 64: 1.7 -> 0.75 ms; what bounds it now is issue (a third of
// the time) and the latency of the neighbour loads at 12 warps per SM.
#include "async.cuh"
#include "dfloat.cuh"
#include "dslash.cuh"
#include "evenodd.cuh"
#include "kernels.cuh"
#include "reduce.cuh"
#include "vec.cuh"

namespace lqcd {
namespace {

constexpr int RU_THREADS = 128;
constexpr int RU_COOP = 2 * 152;   // 128-site units (slots x units) of a cooperative launch: two blocks per SM
constexpr int RU_RUNS = 4096;   // partial sums per slot at most (24^3 x 64: 3456 of two units)
static_assert(2 * RU_RUNS <= PARTIAL_STRIDE, "partials of a slot");
static_assert(MAX_SLOTS <= 32, "a slot per lane");

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Barrier over the grid's nblocks co-resident blocks (cooperative launch): bar[0]
// counts arrivals, *gen the completed barriers. Every global write before it is
// visible after it. The wait is bounded; false (uniform over the block) if it gave up.
__device__ bool grid_barrier(unsigned* bar, unsigned* gen, unsigned nblocks) {
    __shared__ int s_ok;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned g = ld_acquire(gen);
        bool ok = true;
        if (atomicAdd(bar, 1u) == nblocks - 1) {
            *bar = 0;
            __threadfence();
            atomicAdd(gen, 1u);
        } else {
            const long long t0 = clock64(), lim = wait_cycles();
            while (ld_acquire(gen) == g)
                if (clock64() - t0 > lim) { ok = false; break; }
        }
        s_ok = ok;
    }
    __syncthreads();
    __threadfence();
    return s_ok != 0;
}

// FP64 field read with ordinary loads: x_hi and the even-odd stage buffer change
// during the kernel, so the read-only path of Field<double>::load is not for them.
struct LiveField {
    const double2* p;
    int V;
    __device__ __forceinline__ void load(int s, double2 (&v)[12]) const {
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            v[2 * q] = p[((size_t)q * V + s) * 2];
            v[2 * q + 1] = p[((size_t)q * V + s) * 2 + 1];
        }
    }
};
struct LiveHalf {
    const double2* p;
    int Vh;
    __device__ __forceinline__ void load(int s, double2 (&v)[12]) const { LiveField{p, Vh}.load(s >> 1, v); }
};

__device__ __forceinline__ dfc dfc_of(float4 t) { return {{t.x, t.z}, {t.y, t.w}}; }
__device__ __forceinline__ dfl pick(bool c, dfl a, dfl b) { return {c ? a.h : b.h, c ? a.l : b.l}; }

// acc = D_hop x at site s in double-float arithmetic, unnormalised sums (s + c).
// Chiral basis: a hop projects h_a = p_a + sg (M p_lo)_a with (M p_lo) a spin
// permutation times +-1 or +-i, multiplies by the link, and adds (o, sg M^+ o).
__device__ __forceinline__ void hop_site_df(const Geom& g, const float4* __restrict__ U, const float4* x, int s,
                                            Dot2 (&ax)[12], Dot2 (&ay)[12]) {
    const int V = g.V;
    int c0, c1, c2, c3;
    {
        int r = s;
        c0 = r % g.L[0]; r /= g.L[0];
        c1 = r % g.L[1]; r /= g.L[1];
        c2 = r % g.L[2];
        c3 = r / g.L[2];
    }
#pragma unroll
    for (int c = 0; c < 12; ++c) ax[c] = ay[c] = Dot2{0.f, 0.f};
#pragma unroll 1
    for (int hop = 0; hop < 8; ++hop) {
        const int mu = hop >> 1;
        const bool bwd = hop & 1;
        const int cm = mu == 0 ? c0 : mu == 1 ? c1 : mu == 2 ? c2 : c3;
        const int st = g.stride[mu], L1 = g.L[mu] - 1;
        const int nb = bwd ? (cm == 0 ? s + L1 * st : s - st) : (cm == L1 ? s - L1 * st : s + st);
        const float sg = bwd ? 1.f : -1.f;
        const bool swap = (mu & 1) == 0;     // M's entries are +-i: real and imaginary parts change places
        const bool cross = mu < 2;           // h_0 takes spin 3 and h_1 spin 2
        // signs of (Re, Im) of M p_lo in h_0 and h_1, projector sign included
        const float f0x = mu == 1 ? -sg : sg, f0y = mu == 3 ? sg : -sg;
        const float f1x = mu == 2 ? -sg : sg, f1y = mu == 0 ? -sg : sg;
        dfc h[2][3];
        {
            const float4* xs = x + (size_t)nb * 2;
            const int lo0 = cross ? 9 : 6, lo1 = cross ? 6 : 9;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                auto at = [&](int e) { return dfc_of(xs[(size_t)(e >> 1) * V * 2 + (e & 1)]); };
                const dfc p0 = at(c), p1 = at(3 + c), m0 = at(lo0 + c), m1 = at(lo1 + c);
                h[0][c] = {df_axpy(p0.x, f0x, pick(swap, m0.y, m0.x)), df_axpy(p0.y, f0y, pick(swap, m0.x, m0.y))};
                h[1][c] = {df_axpy(p1.x, f1x, pick(swap, m1.y, m1.x)), df_axpy(p1.y, f1y, pick(swap, m1.x, m1.y))};
            }
        }
        // row r of U (forward, at s), or column r conjugated (backward, at the neighbour)
        const float4* u = U + (size_t)mu * 9 * V + (bwd ? nb : s);
        const size_t rs = (size_t)(bwd ? 1 : 3) * V, cs = (size_t)(bwd ? 3 : 1) * V;
        // signs of (Re, Im) of M^+ o in spins 2 and 3: conjugate phases, swapped sources
        const float l0x = swap ? -sg : sg, l0y = sg;
        const float l1x = mu == 0 || mu == 1 ? -sg : sg, l1y = mu == 1 || mu == 2 ? -sg : sg;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            Dot2 re[2], im[2];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                dfc v = dfc_of(__ldg(u + r * rs + c * cs));
                if (bwd) v.y = -v.y;
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    if (c == 0) { re[a].first(v.x, h[a][c].x); im[a].first(v.x, h[a][c].y); }
                    else { re[a].add(v.x, h[a][c].x); im[a].add(v.x, h[a][c].y); }
                    re[a].add(-v.y, h[a][c].y);
                    im[a].add(v.y, h[a][c].x);
                }
            }
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                ax[3 * a + r].plus(re[a].s, re[a].c);
                ay[3 * a + r].plus(im[a].s, im[a].c);
            }
            const Dot2 q0r = cross ? re[1] : re[0], q0i = cross ? im[1] : im[0];
            const Dot2 q1r = cross ? re[0] : re[1], q1i = cross ? im[0] : im[1];
            const Dot2 w0r = swap ? q0i : q0r, w0i = swap ? q0r : q0i, w1r = swap ? q1i : q1r, w1i = swap ? q1r : q1i;
            ax[6 + r].plus(l0x, w0r.s, w0r.c);
            ay[6 + r].plus(l0y, w0i.s, w0i.c);
            ax[9 + r].plus(l1x, w1r.s, w1r.c);
            ay[9 + r].plus(l1y, w1i.s, w1i.c);
        }
    }
}

enum RuMode { RU_F64 = 0, RU_DF = 1, RU_EO = 2 };
enum RuPhase { RU_ALL = -1, RU_FOLD = 0, RU_STAGE = 1, RU_RESID = 2 };   // RU_ALL: cooperative launch

template <typename S, int MODE>
__global__ void __launch_bounds__(RU_THREADS, MODE == RU_DF ? 3 : 2)
    ru_kernel(Geom g, const double2* links64, const float4* links_df, double kappa, SlotState* states,
              const SlotPtrs* ptrs, int nslots, size_t N, int phase, int* err) {
    __shared__ int list[MAX_SLOTS];
    __shared__ int s_n;
    if (threadIdx.x < 32) {   // a slot per lane, its words read at once: most launches end here
        const int j = threadIdx.x;
        const SlotState& st = states[j < nslots ? j : 0];
        // After a wait that gave up, the counters may be stale until the host has seen err:
        // no further update. (Set by a block of this launch while others start, it only
        // makes them give up too.)
        const bool on = (j < nslots) & (st.status == ST_RUNNING) & (st.live != 0) & (st.need_ru != 0) & (*(volatile int*)err == 0);
        const unsigned m = __ballot_sync(0xffffffffu, on);
        if (on) list[__popc(m & ((1u << j) - 1u))] = j;
        if (j == 0) s_n = __popc(m);
    }
    __syncthreads();
    const int nact = s_n;
    if (nact == 0) return;   // uniform over the grid: these words change only after every block has read them
    const int gt = blockIdx.x * RU_THREADS + threadIdx.x, gn = gridDim.x * RU_THREADS;
    unsigned* bar = ptrs[0].counters + CNT_BAR;
    unsigned* gen = ptrs[0].counters + CNT_GEN;
    // x_hi += x_lo, x_lo = 0
    const size_t units = N / 2;
    for (int i = 0; i < nact && phase <= RU_FOLD; ++i) {
        const SlotState& st = states[list[i]];
        const SlotPtrs& P = ptrs[list[i]];
        const cplx<S> al = cvt<S>(st.alpha);
        // gamma5 variant, FP32 vectors: the best x so far is kept in r_true (free between the
        // start and the end of a solve), for a solve that has to go back to it
        const bool guard = sizeof(S) == 4 && st.g5 != 0, back = guard && st.fresh_dir == FRESH_BEST;
        const bool keep = guard && st.x_best != 0 && !back, fetch = back && !st.x_best;
        const bool owed = st.x_owed != 0 && !back;
        const Unit<S> zero{mk<S>(0, 0), mk<S>(0, 0)};
        for (size_t u = gt; u < units; u += gn) {
            Unit<double> xh = Unit<double>::load(fetch ? P.r_true : P.x_hi, u);
            Unit<S> xl = back ? zero : Unit<S>::load(P.x_lo, u);
            if (keep) xh.store(P.r_true, u);
            if (owed) {   // alpha p of this iteration's residual update
                const Unit<S> p = Unit<S>::load(P.p, u);
                xl.a = cfma(xl.a, al, p.a); xl.b = cfma(xl.b, al, p.b);
            }
            xh.a = xh.a + wid(xl.a); xh.b = xh.b + wid(xl.b);
            xh.store(P.x_hi, u);
            zero.store(P.x_lo, u);
            if (MODE == RU_DF) {   // the double-float copy that the residual reads
                const dfl ar = df_split(xh.a.x), ai = df_split(xh.a.y), br = df_split(xh.b.x), bi = df_split(xh.b.y);
                P.x_df[2 * u] = make_float4(ar.h, ai.h, ar.l, ai.l);
                P.x_df[2 * u + 1] = make_float4(br.h, bi.h, br.l, bi.l);
            }
        }
    }
    if (phase == RU_FOLD) return;
    bool ok = phase != RU_ALL || grid_barrier(bar, gen, gridDim.x);
    const int Vs = MODE == RU_EO ? g.V / 2 : g.V;   // sites of the solver's space
    if (MODE == RU_EO && ok && phase != RU_RESID) {   // stage 1: D_eo x_hi on the even sites
        const LinksD U{links64, g.V};
        for (int i = 0; i < nact; ++i) {
            const SlotPtrs& P = ptrs[list[i]];
            const LiveHalf in{P.x_hi, Vs};
            for (int h = gt; h < Vs; h += gn) {
                double2 acc[12];
                hop_site<false, double>(g, U, in, eo_site(g, h, 0), acc);
                Field<double>::store(P.eo64, Vs, h, acc);
            }
        }
        if (phase == RU_STAGE) return;
        ok = grid_barrier(bar, gen, gridDim.x);
    }
    if (!ok) {   // uniform over the block: report and leave, the host discards the solve
        if (threadIdx.x == 0) atomicExch(err, 1);
        return;
    }
    // Residual, its norm, the new r and rho. A slot's sites are RU_THREADS-site units, its
    // units runs of `per` with one partial sum each: both follow from the lattice alone, so
    // the sums of a source do not depend on the grid or on the other slots. The blocks
    // share the slots' runs equally.
    const int nunits = (Vs + RU_THREADS - 1) / RU_THREADS;
    const int per = (nunits + RU_RUNS - 1) / RU_RUNS, nruns = (nunits + per - 1) / per;
    const long long T = (long long)nact * nruns;
    const long long t0 = blockIdx.x * T / gridDim.x, t1 = (blockIdx.x + 1) * T / gridDim.x;
    __shared__ double smd[RU_THREADS / 32 * 4];
    const double kk = MODE == RU_EO ? kappa * kappa : kappa;
    for (int i = 0; i < nact; ++i) {
        const SlotState& st = states[list[i]];
        const SlotPtrs& P = ptrs[list[i]];
        const int q0 = (int)max(t0 - (long long)i * nruns, 0ll), q1 = (int)min(t1 - (long long)i * nruns, (long long)nruns);
        void* rcur = slot_field<S>(P.V, next_slot(st), N);
        void* hcur = slot_field<S>(P.W, next_slot(st), N);
        const bool g5 = st.g5 != 0, win = st.m > 0, comp = g5 && sizeof(S) == 4;
        for (int q = q0; q < q1; ++q) {
            double nrm = 0.0;
            cplx<S> rho = mk<S>(S(0), S(0));
            CompC cz;
            for (int u = q * per; u < min(q * per + per, nunits); ++u) {
                const int s = u * RU_THREADS + (int)threadIdx.x;
                if (s >= Vs) continue;
                double2 r[12];
                if constexpr (MODE == RU_DF) {
                    Dot2 ax[12], ay[12];
                    hop_site_df(g, links_df, P.x_df, s, ax, ay);
                    const LiveField xin{P.x_hi, Vs}, bin{P.b, Vs};
                    double2 self[12];
                    xin.load(s, self);
                    bin.load(s, r);
#pragma unroll
                    for (int c = 0; c < 12; ++c) {   // b - x + kappa D x, the FP64 part of it 4 instructions per real
                        r[c].x = fma(kk, widen(ax[c].s), fma(kk, widen(ax[c].c), r[c].x - self[c].x));
                        r[c].y = fma(kk, widen(ay[c].s), fma(kk, widen(ay[c].c), r[c].y - self[c].y));
                    }
                } else {
                    const LinksD U{links64, g.V};
                    double2 acc[12], self[12];
                    if constexpr (MODE == RU_EO) hop_site<false, double>(g, U, LiveHalf{P.eo64, Vs}, eo_site(g, s, 1), acc);
                    else hop_site<false, double>(g, U, LiveField{P.x_hi, Vs}, s, acc);
                    LiveField{P.x_hi, Vs}.load(s, self);
                    LiveField{P.b, Vs}.load(s, r);
#pragma unroll
                    for (int c = 0; c < 12; ++c)
                        r[c] = r[c] - make_double2(fma(-kk, acc[c].x, self[c].x), fma(-kk, acc[c].y, self[c].y));
                }
                cplx<S> rs[12], hs[12];
#pragma unroll
                for (int c = 0; c < 12; ++c) {
                    nrm = fma(r[c].x, r[c].x, fma(r[c].y, r[c].y, nrm));
                    rs[c] = nar<S>(r[c]);
                }
                Field<S>::store(rcur, Vs, s, rs);
                if (g5) {   // the shadow residual follows: rhat = gamma5 r
#pragma unroll
                    for (int c = 0; c < 12; ++c) hs[c] = c < 6 ? rs[c] : -rs[c];
                    if (win) Field<S>::store(hcur, Vs, s, hs);
                } else {
                    Field<S>::load(hcur, Vs, s, hs);
                }
                if (comp) {
                    if constexpr (sizeof(S) == 4) {
#pragma unroll
                        for (int c = 0; c < 12; ++c) cz.add(cdot(hs[c], rs[c]));
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < 12; ++c) rho = cdot_acc(rho, hs[c], rs[c]);
                }
            }
            double2 v[2] = {comp ? cz.value() : to_d(rho), make_double2(nrm, 0.0)};
            block_sum_wide<2>(v, v, smd);
            if (threadIdx.x == 0) {
                double2* pp = part(P, CNT_RU) + 2 * (size_t)q;
                pp[0] = v[0];
                pp[1] = v[1];
            }
        }
    }
    // the last block adds the partials in a fixed order and ends the iteration
    if (!last_block(ptrs[0].counters + CNT_RU, gridDim.x)) return;
    for (int i = 0; i < nact; ++i) {
        SlotState& st = states[list[i]];
        const SlotPtrs& P = ptrs[list[i]];
        const double2* pp = part(P, CNT_RU);
        double2 v[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
        for (int b = threadIdx.x; b < nruns; b += RU_THREADS) {
            v[0] = v[0] + __ldcg(pp + 2 * (size_t)b);
            v[1] = v[1] + __ldcg(pp + 2 * (size_t)b + 1);
        }
        block_sum_wide<2>(v, v, smd);
        if (threadIdx.x == 0) {
            st.true_rnorm = sqrt_fp64(v[1].x);
            st.matvecs += 1;
            if (st.true_rnorm <= st.tol * st.bnorm) {
                st.status = ST_CONVERGED;
            } else {
                st.rho_new = v[0];
                st.rnorm_new = st.true_rnorm;
                st.rmax = st.true_rnorm;
                st.r_ru = st.true_rnorm;
            }
            st.need_ru = 0;
            st.ru_count += 1;
            if (sizeof(S) == 4 && st.g5) {
                if (st.fresh_dir == FRESH_NONE) st.stall_lim = max(st.stall_lim, 4 * (st.iter + 1 - st.ru_iter));
                else st.stall_lim = min(2 * st.stall_lim, 1 << 28);
                st.x_best = st.fresh_dir == FRESH_BEST || st.true_rnorm < st.r_best;
                if (st.x_best) {
                    st.r_best = st.true_rnorm;
                    st.best_used = st.fresh_dir == FRESH_BEST;
                }
                st.r_min = st.true_rnorm;
                st.min_iter = st.iter + 1;
            }
            st.ru_iter = st.iter + 1;
            st.x_owed = 0;   // the fold added alpha p
            if (st.stab) stab_scalars(st);
            else bicg_scalars(st, P);
        }
        __syncthreads();
    }
}

// FP64 links [mu][9][V] double2 -> double-float float4 (h.re, h.im, l.re, l.im).
__global__ void links_df_kernel(const double2* l64, float4* ldf, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const double2 v = l64[i];
        const dfl r = df_split(v.x), m = df_split(v.y);
        ldf[i] = make_float4(r.h, m.h, r.l, m.l);
    }
}

using RuKernel = void (*)(Geom, const double2*, const float4*, double, SlotState*, const SlotPtrs*, int, size_t, int, int*);
RuKernel ru_select(int prec, int df, int eo) {
    if (prec == 0) return eo ? ru_kernel<double, RU_EO> : ru_kernel<double, RU_F64>;
    if (eo) return ru_kernel<float, RU_EO>;
    return df ? ru_kernel<float, RU_DF> : ru_kernel<float, RU_F64>;
}

}  // namespace

cudaError_t set_wait_cycles_ru(long long cycles) { return set_wait_cycles_here(cycles); }

cudaError_t launch_links_df(const double2* l64, float4* ldf, size_t n, cudaStream_t st) {
    links_df_kernel<<<1216, 256, 0, st>>>(l64, ldf, n);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t ru_max_blocks(int prec, int df, int eo, int* blocks) {
    int dev = 0, nsm = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, ru_select(prec, df, eo), RU_THREADS, 0);
    if (e != cudaSuccess) return e;
    *blocks = nsm * per < PARTIAL_STRIDE / 2 ? nsm * per : PARTIAL_STRIDE / 2;
    return *blocks > 0 ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t launch_bicg_ru(const Geom& g, const void* links64, double kappa, int prec, SlotState* states,
                           const SlotPtrs* ptrs, int nslots, size_t N, cudaStream_t s, const float4* links_df, int eo,
                           int max_blocks, int* err) {
    const int Vs = eo ? g.V / 2 : g.V;
    const long long units = (long long)((Vs + RU_THREADS - 1) / RU_THREADS) * nslots;
    const RuKernel kernel = ru_select(prec, links_df && !eo, eo);
    const double2* l64 = reinterpret_cast<const double2*>(links64);
    if (units > RU_COOP) {
        const unsigned grid = (unsigned)(units < max_blocks ? units : max_blocks);
        for (int phase : {RU_FOLD, RU_STAGE, RU_RESID}) {
            if (phase == RU_STAGE && !eo) continue;
            kernel<<<grid, RU_THREADS, 0, s>>>(g, l64, links_df, kappa, states, ptrs, nslots, N, phase, err);
            count_launches(1);
        }
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(units < max_blocks ? units : max_blocks));
    cfg.blockDim = dim3(RU_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, g, l64, links_df, kappa, states, ptrs, nslots, N, (int)RU_ALL, err);
    count_launches(1);
    return e;
}

}  // namespace lqcd
