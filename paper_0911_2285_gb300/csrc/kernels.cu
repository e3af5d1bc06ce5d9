// Lattice-sized kernels: the Wilson operator applications, the BiCG iteration
// (Algorithm eigBiCG, steps 1-3 of the paper, Sec. 2), the window product of
// the BiCG-eigen restart with its coupling row/column, and the tall-skinny
// products of the oblique deflation (Algorithm Incremental eigBiCG).
//
// All reductions are two-level and deterministic: each block writes its
// partial sums to a fixed slot, and the last block to finish adds them in
// block order (same result alone or inside a batch).
#include "dslash.cuh"
#include "kernels.cuh"
#include "reduce.cuh"
#include "vec.cuh"

namespace lqcd {
namespace {

constexpr int DS_THREADS = 128;   // operator kernels
constexpr int BL_THREADS = 256;   // vector kernels
constexpr int G5_STALL = 500;     // least number of iterations that make a stall of the gamma5 variant

inline int div_up(size_t a, size_t b) { return (int)((a + b - 1) / b); }

// Threads per block of the FP64 site and vector kernels (jobs: of a full batch, so that
// a source's sums are the same alone and in a batch of its context): the FP64 pipe of an SM serves
// 2 lanes per clock, so what matters is how many SMs take part. Below two blocks of
// the full size per SM, one-warp blocks spread the same warps over the chip: operator
// pair on 4^4 (16 warps) 42 us on 4 SMs, 36 on 16. The smallest operator grids go to
// fp64_split.cu.
constexpr int SMALL_GRID = 2 * 152;
int site_threads(size_t sites, int jobs, int full) { return (sites + full - 1) / full * jobs < SMALL_GRID ? 32 : full; }

int blas_blocks(size_t units) {
    int nb = div_up(units, BL_THREADS);
    if (nb > 1216) nb = 1216;   // 8 blocks of 256 per SM on 152 SMs
    if (nb < 1) nb = 1;
    return nb;
}
// Blocks per slot of the vector kernels that end in a reduction. A block's end (block
// sum, partial, a fence that waits for its stores) takes about 2 us of its place on the
// SM, so a thread takes at least four units where that leaves two blocks per SM; whole
// blocks per SM. A function of the field alone: a source's sums must not depend on the
// batch. Half lattice of 16^3 x 32, 8 slots: residual
// update 71.6 -> 53.9 us (floor 44); from 24^3 x 64 on the same grid as blas_blocks.
int red_blocks(size_t units) {
    int nb = (int)(units / (4 * BL_THREADS) / 152) * 152;
    if (nb < 2 * 152) nb = 2 * 152;
    const int most = blas_blocks(units);
    return nb < most ? nb : most;
}
int ds_blocks(int V) {
    int nb = div_up((size_t)V, DS_THREADS);
    if (nb > PARTIAL_STRIDE / 2) nb = PARTIAL_STRIDE / 2;
    return nb;
}

// ------------------------------------------------------------------- apply
// r = b - A x with FP64 x and b and the hop in FP32 arithmetic on FP32 links: the
// starting and deflation residuals of the mixed-precision solver, which are consumed
// in FP32 (the reliable updates and the final residual use FP64-class arithmetic).
// x32: x rounded to FP32; SO: storage of r. nf consecutive fields.
// What bounds it: rounding each of the eight neighbours from FP64 costs 16 conversions
// per number on the FP64 pipe (26 operations with the rest: 480 us for 8 fields of
// 16^3 x 32); from x32 four FP64 operations are left (86 us on that pipe), and bytes:
// x, b and x32 read once, r written, 48 to 56 per number. Measured 480 -> 184 us
// and 52 for x32.
template <typename SO>
__global__ void __launch_bounds__(DS_THREADS) residual32_kernel(Geom g, const float4* links, double kappa,
                                                                const double2* x, const float2* x32, const double2* b,
                                                                cplx<SO>* r, int nf) {
    const int jid = blockIdx.x % nf, sblock = blockIdx.x / nf, nsb = gridDim.x / nf;   // fields fastest: shared links
    const size_t off = (size_t)jid * 12 * g.V;
    LinksF U{links, g.V};
    FieldIn<float> in{x32 + off, g.V};
    const double k = kappa;
    for (int s = sblock * blockDim.x + threadIdx.x; s < g.V; s += nsb * blockDim.x) {
        float2 acc[12];
        hop_site<false, float>(g, U, in, s, acc);
        double2 xs[12], bs[12];
        Field<double>::load(x + off, g.V, s, xs);
        Field<double>::load(b + off, g.V, s, bs);
        cplx<SO> out[12];
#pragma unroll
        for (int c = 0; c < 12; ++c) out[c] = nar<SO>(bs[c] - (xs[c] - k * widen(acc[c])));
        Field<SO>::store(r + off, g.V, s, out);
    }
}

// nf consecutive fields, fields fastest in the grid: they share each block's links.
template <typename S, bool RES>
__global__ void __launch_bounds__(DS_THREADS) apply_kernel(Geom g, const void* links, double kappa,
                                                           const void* src, void* dst, const double2* aux, int dagger,
                                                           int nf) {
    using C = cplx<S>;
    const int jid = blockIdx.x % nf, sblock = blockIdx.x / nf, nsb = gridDim.x / nf;
    const size_t off = (size_t)jid * 12 * g.V;
    typename LinkSel<S>::type U{reinterpret_cast<decltype(U.u)>(links), g.V};
    FieldIn<S> in{reinterpret_cast<const C*>(src) + off, g.V};
    const S k = (S)kappa;
    for (int s = sblock * blockDim.x + threadIdx.x; s < g.V; s += nsb * blockDim.x) {
        C acc[12], self[12];
        if (dagger) hop_site<true, S>(g, U, in, s, acc);
        else hop_site<false, S>(g, U, in, s, acc);
        in.load(s, self);
#pragma unroll
        for (int c = 0; c < 12; ++c) acc[c] = self[c] - k * acc[c];
        if (RES) {
            double2 b[12];
            Field<double>::load(aux + off, g.V, s, b);
#pragma unroll
            for (int c = 0; c < 12; ++c) acc[c] = cvt<S>(b[c] - to_d(acc[c]));
        }
        Field<S>::store(reinterpret_cast<C*>(dst) + off, g.V, s, acc);
    }
}

// -------------------------------------------------------------- pack/unpack
// Host layout AoS [site][12] complex128 <-> device chunk layout.
// A block turns PK_SITES sites of one field through shared memory, so that both sides
// are read and written in whole lines (a site is 13 units apart there: no conflicts).
// Bound by bytes: 24 or 32 per number; the conversions run on the integer pipe (two per
// number on the FP64 pipe take as long as the bytes). Element by element, with 64-bit
// divisions and 16-byte pieces, 4 fields of 24^3 x 64 took 181 us in and 171 out, now
// 141 and 154 (1.0 GB each way).
constexpr int PK_SITES = BL_THREADS / 2;
template <typename S>
__global__ void __launch_bounds__(BL_THREADS) pack_kernel(const double2* aos, cplx<S>* dev, int V) {
    __shared__ double2 sm[PK_SITES * 13];
    const int s0 = blockIdx.x * PK_SITES, ns = V - s0 < PK_SITES ? V - s0 : PK_SITES, t = threadIdx.x;
    const size_t f = (size_t)blockIdx.y * V * 12;
    const double2* src = aos + f + (size_t)s0 * 12;
    double2 v[6];
#pragma unroll
    for (int r = 0; r < 6; ++r)
        if (r * BL_THREADS + t < ns * 12) v[r] = src[r * BL_THREADS + t];
#pragma unroll
    for (int r = 0; r < 6; ++r) {
        const int i = r * BL_THREADS + t;
        if (i < ns * 12) sm[i / 12 * 13 + i % 12] = v[r];
    }
    __syncthreads();
    if (t >= 2 * ns) return;
#pragma unroll
    for (int h = 0; h < 6; ++h)
        dev[f + ((size_t)h * V + s0) * 2 + t] = nar<S>(sm[(t >> 1) * 13 + 2 * h + (t & 1)]);
}
template <typename S>
__global__ void __launch_bounds__(BL_THREADS) unpack_kernel(const cplx<S>* dev, double2* aos, int V) {
    __shared__ double2 sm[PK_SITES * 13];
    const int s0 = blockIdx.x * PK_SITES, ns = V - s0 < PK_SITES ? V - s0 : PK_SITES, t = threadIdx.x;
    const size_t f = (size_t)blockIdx.y * V * 12;
    if (t < 2 * ns) {
        cplx<S> v[6];
#pragma unroll
        for (int h = 0; h < 6; ++h) v[h] = dev[f + ((size_t)h * V + s0) * 2 + t];
#pragma unroll
        for (int h = 0; h < 6; ++h) sm[(t >> 1) * 13 + 2 * h + (t & 1)] = wid(v[h]);
    }
    __syncthreads();
    double2* dst = aos + f + (size_t)s0 * 12;
#pragma unroll
    for (int r = 0; r < 6; ++r) {
        const int i = r * BL_THREADS + t;
        if (i < ns * 12) dst[i] = sm[i / 12 * 13 + i % 12];
    }
}
template <typename SI, typename SO>
__global__ void convert_kernel(const void* src, void* dst, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        st_elem<SO>(dst, i, nar<SO>(wid(ld_elem<SI>(src, i))));
}

// ------------------------------------------------------------- multidot
// C[i][j] = sum_e conj(X_i(e)) Y_j(e) for i in [i0, i0+TI), j < b <= BMAX.
constexpr int MD_TI = 4, MD_BMAX = 8;
// Grid: (element chunk x column group) flattened with the column group fastest,
// so the groups that read the same Y chunk run together (Y leaves DRAM once).
template <typename SX, typename SY, typename T>
__global__ void __launch_bounds__(BL_THREADS) multidot_kernel(int a, const void* X, int b, const void* Y, size_t N,
                                                              double2* scratch, int nby) {
    using C = cplx<T>;
    const int by = blockIdx.x % nby, bx = blockIdx.x / nby, nbx = gridDim.x / nby;
    const int i0 = by * MD_TI;
    C acc[MD_TI][MD_BMAX];
#pragma unroll
    for (int i = 0; i < MD_TI; ++i)
#pragma unroll
        for (int j = 0; j < MD_BMAX; ++j) acc[i][j] = mk<T>(T(0), T(0));
    for (size_t e = bx * (size_t)blockDim.x + threadIdx.x; e < N; e += (size_t)nbx * blockDim.x) {
        C y[MD_BMAX];
#pragma unroll
        for (int j = 0; j < MD_BMAX; ++j)
            if (j < b) {
                auto v = ld_elem<SY>(reinterpret_cast<const char*>(Y) + (size_t)j * N * sizeof(cplx<SY>), e);
                y[j] = mk<T>((T)v.x, (T)v.y);
            }
#pragma unroll
        for (int i = 0; i < MD_TI; ++i)
            if (i0 + i < a) {
                auto v = ld_elem<SX>(reinterpret_cast<const char*>(X) + (size_t)(i0 + i) * N * sizeof(cplx<SX>), e);
                C x = mk<T>((T)v.x, (T)v.y);
#pragma unroll
                for (int j = 0; j < MD_BMAX; ++j)
                    if (j < b) acc[i][j] = acc[i][j] + cdot(x, y[j]);
            }
    }
    C v[MD_TI * MD_BMAX];
#pragma unroll
    for (int i = 0; i < MD_TI; ++i)
#pragma unroll
        for (int j = 0; j < MD_BMAX; ++j) v[i * MD_BMAX + j] = acc[i][j];
    __shared__ C sm[(BL_THREADS / 32) * MD_TI * MD_BMAX];
    block_sum<MD_TI * MD_BMAX>(v, sm);   // in the accumulation precision T
    if (threadIdx.x == 0) {
        double2* out = scratch + ((size_t)by * nbx + bx) * (MD_TI * MD_BMAX);
#pragma unroll
        for (int q = 0; q < MD_TI * MD_BMAX; ++q) out[q] = to_d(v[q]);
    }
}
__global__ void multidot_reduce_kernel(int a, int b, int nbx, const double2* scratch, double2* Cm, int ldc,
                                       int conj_store) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;   // (i, j) pair
    if (q >= a * b) return;
    const int i = q / b, j = q % b;
    const int by = i / MD_TI, ii = i % MD_TI;
    double2 acc = make_double2(0.0, 0.0);
    for (int bx = 0; bx < nbx; ++bx) acc = acc + scratch[((size_t)by * nbx + bx) * (MD_TI * MD_BMAX) + ii * MD_BMAX + j];
    if (conj_store) Cm[(size_t)j * ldc + i] = conj_(acc);
    else Cm[(size_t)i * ldc + j] = acc;
}

// ------------------------------------------------------------- vupdate
// mode 0: Y_j += sum_i X_i D[i][j];  mode 1: Y_j = sum_i X_i D[i][j]  (j < b <= MD_BMAX).
template <typename SX, typename SY, typename T>
__global__ void __launch_bounds__(BL_THREADS) vupdate_kernel(int a, const void* X, const double2* D, int ldd, int b,
                                                             void* Y, int overwrite, size_t N) {
    using C = cplx<T>;
    __shared__ C Ds[MAX_SMALL * MD_BMAX];
    for (int q = threadIdx.x; q < a * b; q += blockDim.x) {
        const int i = q / b, j = q % b;
        double2 d = D[(size_t)i * ldd + j];
        Ds[i * MD_BMAX + j] = mk<T>((T)d.x, (T)d.y);
    }
    __syncthreads();
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < N; e += (size_t)gridDim.x * blockDim.x) {
        C acc[MD_BMAX];
#pragma unroll
        for (int j = 0; j < MD_BMAX; ++j) acc[j] = mk<T>(T(0), T(0));
        for (int i = 0; i < a; ++i) {
            auto v = ld_elem<SX>(reinterpret_cast<const char*>(X) + (size_t)i * N * sizeof(cplx<SX>), e);
            C x = mk<T>((T)v.x, (T)v.y);
#pragma unroll
            for (int j = 0; j < MD_BMAX; ++j)
                if (j < b) acc[j] = acc[j] + x * Ds[i * MD_BMAX + j];
        }
#pragma unroll
        for (int j = 0; j < MD_BMAX; ++j)
            if (j < b) {
                char* yj = reinterpret_cast<char*>(Y) + (size_t)j * N * sizeof(cplx<SY>);
                double2 upd = to_d(acc[j]);
                if (!overwrite) upd = upd + to_d(ld_elem<SY>(yj, e));   // add in the target precision
                st_elem<SY>(yj, e, cvt<SY>(upd));
            }
    }
}

// The same with FP32 X and FP32 sums, added to an FP64 Y in FP64. A thread takes two
// consecutive elements, so a coefficient read from shared memory (two Y fields per
// 16-byte load) serves 16 multiply-adds, and four X loads are in flight. Bound: X once
// and Y twice over memory (40 x 8 on 16^3 x 32: 0.5 + 0.4 GB, 133 us) against 54 us of
// multiply-adds; with one element per thread and conversions on the FP64 pipe 325 us,
// measured 223. N even.
template <typename SY>
__global__ void __launch_bounds__(BL_THREADS) vupdate32_kernel(int a, const float4* X, const double2* D, int ldd, int b,
                                                               void* Y, int overwrite, size_t N) {
    __shared__ float4 Ds[MAX_SMALL * MD_BMAX / 2];
    for (int q = threadIdx.x; q < a * (MD_BMAX / 2); q += blockDim.x) {
        const int i = q / (MD_BMAX / 2), j = 2 * (q % (MD_BMAX / 2));
        const double2 z = make_double2(0.0, 0.0);
        const double2 d0 = j < b ? D[(size_t)i * ldd + j] : z, d1 = j + 1 < b ? D[(size_t)i * ldd + j + 1] : z;
        Ds[q] = make_float4((float)d0.x, (float)d0.y, (float)d1.x, (float)d1.y);
    }
    __syncthreads();
    const size_t units = N / 2;
    for (size_t u = blockIdx.x * (size_t)blockDim.x + threadIdx.x; u < units; u += (size_t)gridDim.x * blockDim.x) {
        float2 acc[MD_BMAX][2];
#pragma unroll
        for (int j = 0; j < MD_BMAX; ++j) acc[j][0] = acc[j][1] = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int i = 0; i < a; ++i) {
            const float4 x = X[(size_t)i * units + u];
            const float2 x0 = make_float2(x.x, x.y), x1 = make_float2(x.z, x.w);
#pragma unroll
            for (int p = 0; p < MD_BMAX / 2; ++p)
                if (2 * p < b) {
                    const float4 d = Ds[i * (MD_BMAX / 2) + p];
                    const float2 d0 = make_float2(d.x, d.y), d1 = make_float2(d.z, d.w);
                    acc[2 * p][0] = acc[2 * p][0] + x0 * d0;
                    acc[2 * p][1] = acc[2 * p][1] + x1 * d0;
                    acc[2 * p + 1][0] = acc[2 * p + 1][0] + x0 * d1;
                    acc[2 * p + 1][1] = acc[2 * p + 1][1] + x1 * d1;
                }
        }
#pragma unroll
        for (int j = 0; j < MD_BMAX; ++j)
            if (j < b) {
                cplx<SY>* y = reinterpret_cast<cplx<SY>*>(Y) + (size_t)j * N + 2 * u;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    double2 v = widen(acc[j][h]);
                    if (!overwrite) v = v + wid(y[h]);
                    y[h] = nar<SY>(v);
                }
            }
    }
}

// Per-field squared 2-norms of b fields: block partials (FP64) for a second pass.
template <typename S>
__global__ void __launch_bounds__(BL_THREADS) norms_kernel(const void* Y, size_t N, double2* scratch) {
    const int j = blockIdx.y;
    const cplx<S>* y = reinterpret_cast<const cplx<S>*>(Y) + (size_t)j * N;
    S acc = S(0);
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < N; e += (size_t)gridDim.x * blockDim.x)
        acc += abs2(y[e]);
    cplx<S> v[1] = {mk<S>(acc, S(0))};
    __shared__ cplx<S> sm[BL_THREADS / 32];
    block_sum<1>(v, sm);
    if (threadIdx.x == 0) scratch[(size_t)j * gridDim.x + blockIdx.x] = to_d(v[0]);
}
__global__ void norms_reduce_kernel(int b, int nb, const double2* scratch, double* out) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= b) return;
    double acc = 0.0;
    for (int i = 0; i < nb; ++i) acc += scratch[(size_t)j * nb + i].x;
    out[j] = sqrt(acc);
}

// Y_j *= s_j (per-field scale), j < b.
template <typename S>
__global__ void scale_fields_kernel(int b, void* Y, const double2* sc, size_t N) {
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < N * b; q += (size_t)gridDim.x * blockDim.x) {
        const int j = (int)(q / N);
        const double2 s = sc[j];
        st_elem<S>(Y, q, cvt<S>(s * to_d(ld_elem<S>(Y, q))));
    }
}

// ------------------------------------------------------------ BiCG kernels
// Start: r0 = b - A x_hi (already in r_true, FP64), rhat0 = r0 (gamma5 r0 in the
// gamma5 variant), p = r, phat = rhat, x_lo = 0; rho_0 = (rhat_0, r_0), ||r_0||,
// ||b||  (Algorithm eigBiCG, steps 1-2).
template <typename S>
__global__ void __launch_bounds__(BL_THREADS) start_kernel(SlotState* states, const SlotPtrs* ptrs, size_t N) {
    SlotState& st = states[blockIdx.y];
    const SlotPtrs& P = ptrs[blockIdx.y];
    if (st.status != ST_RUNNING) return;
    if (st.m > 0 && blockIdx.x == 0)   // a fresh window: H is tridiagonal until the first restart
        for (int e = threadIdx.x; e < st.m * st.m; e += blockDim.x) P.H[e] = make_double2(0.0, 0.0);
    using C = cplx<S>;
    Acc<S> acc;   // rho, |r|^2, |b|^2
    CompC cz;     // rho of the gamma5 variant (FP32 storage)
    const bool comp = st.g5 && sizeof(S) == 4;
    const size_t units = N / 2;
    Unit<S> zero{mk<S>(0, 0), mk<S>(0, 0)};
    for (size_t u = blockIdx.x * (size_t)blockDim.x + threadIdx.x; u < units; u += (size_t)gridDim.x * blockDim.x) {
        Unit<double> rt = Unit<double>::load(P.r_true, u);
        Unit<double> bb = Unit<double>::load(P.b, u);
        Unit<S> r{nar<S>(rt.a), nar<S>(rt.b)};
        r.store(P.V, u);
        r.store(P.p, u);
        Unit<S> h = r;
        if (st.g5) {   // rhat0 = gamma5 r0: only the window keeps it
            h = g5u(r, u, N);
            if (st.m > 0) h.store(P.W, u);
        } else {
            r.store(P.W, u);
            r.store(P.phat, u);
        }
        zero.store(P.x_lo, u);
        if (comp) {
            if constexpr (sizeof(S) == 4) { cz.add(cdot(h.a, r.a)); cz.add(cdot(h.b, r.b)); }
        } else {
            acc.z = cdot_acc(cdot_acc(acc.z, h.a, r.a), h.b, r.b);
        }
        acc.a = abs2_two(acc.a, r.a, r.b);
        acc.b += (S)(cabs2(bb.a) + cabs2(bb.b));
    }
    double2 tot[2];
    if (reduce2<S>(P, CNT_START, comp, cz, acc, tot, gridDim.x, blockIdx.x) && threadIdx.x == 0) {
        st.rho = tot[0];
        st.rnorm = sqrt_fp64(tot[1].x);
        st.bnorm = P.bnorm_ref ? *P.bnorm_ref : sqrt_fp64(tot[1].y);   // even-odd: ||b|| of the full system
        st.rhat_norm = st.rnorm;
        st.rmax = st.rnorm;
        st.r_ru = st.rnorm;
        st.r_min = st.r_best = st.rnorm;
        st.ru_iter = 0; st.min_iter = 0; st.fresh_dir = FRESH_NONE;
        st.x_best = 1; st.best_used = 0; st.stall_lim = G5_STALL;
        st.true_rnorm = st.rnorm;
        st.iter = 0; st.vs = 0; st.need_ru = 0; st.ru_count = 0; st.restarts = 0; st.restart_r = 0;
        st.matvecs = 1; st.live = 1;
        st.alpha_prev = make_double2(0, 0); st.beta_prev = make_double2(0, 0);
        if (st.rnorm <= st.tol * st.bnorm) { st.status = ST_CONVERGED; st.live = 0; }
        // rho_0 = (rhat_0, r_0) must not vanish (e.g. the gamma5 shadow start on a
        // source whose upper and lower spin halves have equal norms)
        else if (!abs_at_least(st.rho, BREAK_TOL, st.rhat_norm, st.rnorm)) { st.status = ST_BREAKDOWN; st.live = 0; }
    }
    (void)sizeof(C);
}

// Operator pair of one iteration: A p -> Ap[par], A^+ phat -> Ahp[par];
// sigma = (phat, A p) and alpha = rho / sigma in the last block.
// Grid: (site blocks x jobs) flattened with the job index fastest, so the jobs
// that share a block of sites (and its links) run together and the links come
// from DRAM once per launch. Variants (picked by the autotuner):
//   PAIR = false: one thread per (site, operator) job, 2 jobs per slot;
//   PAIR = true : one thread per (site, slot) computes both operators and
//                 shares each link load between them.
//   BZ > 0: a block covers an 8 x 8 x BZ brick of sites (THREADS = 64 BZ) instead
//           of THREADS consecutive sites, so more y and z neighbours are L1 hits.
//   TM (t march, with BZ > 0): the units of a brick at consecutive t are
//           consecutive, so a block walks one brick through several t-planes
//           and the t neighbours of a step are the centres of the steps before
//           and after it (L1 hits instead of L2 reads).
template <int THREADS, int BZ, bool TM = false> struct SiteMap {
    int nunits;
    __device__ __forceinline__ SiteMap(const Geom& g) {
        nunits = BZ > 0 ? (g.L[0] / 8) * (g.L[1] / 8) * (g.L[2] / (BZ > 0 ? BZ : 1)) * g.L[3]
                        : (g.V + THREADS - 1) / THREADS;
    }
    __device__ __forceinline__ int site(const Geom& g, int u) const {   // -1: none
        if (BZ == 0) {
            const int s = u * THREADS + (int)threadIdx.x;
            return s < g.V ? s : -1;
        }
        const int nbx = g.L[0] / 8, nby = g.L[1] / 8, nbz = g.L[2] / (BZ > 0 ? BZ : 1);
        int b = u, t = 0;
        if (TM) { t = u % g.L[3]; b = u / g.L[3]; }
        const int bx = b % nbx, r1 = b / nbx, by = r1 % nby, r2 = r1 / nby, bz = r2 % nbz;
        if (!TM) t = r2 / nbz;
        const int x = bx * 8 + (threadIdx.x & 7), y = by * 8 + ((threadIdx.x >> 3) & 7);
        const int z = bz * BZ + (threadIdx.x >> 6);
        return x + g.L[0] * (y + g.L[1] * (z + g.L[2] * t));
    }
};

//   G5   = true : the gamma5 variant (Sec. 4): one job per slot, A p only, with
//                 phat = gamma5 p formed in registers for sigma; windowed slots
//                 also store A^+ phat = gamma5 A p for the restart's coupling.
template <typename S, int THREADS, int MINB, bool PAIR, int BZ = 0, bool G5 = false, bool TM = false>
__global__ void __launch_bounds__(THREADS, MINB) matvec_kernel(Geom g, const void* links, double kappa,
                                                               SlotState* states, const SlotPtrs* ptrs,
                                                               int njobs) {
    const int job = blockIdx.x % njobs, sblock = blockIdx.x / njobs, nsb = gridDim.x / njobs;
    const SiteMap<THREADS, BZ, TM> map(g);
    // each block takes a contiguous run of site units (neighbouring sites stay on one SM)
    const int per = (map.nunits + nsb - 1) / nsb;
    const int u0 = sblock * per, u1 = min(map.nunits, u0 + per);
    const int slot = (PAIR || G5) ? job : job >> 1, which = (PAIR || G5) ? 0 : job & 1;
    SlotState& st = states[slot];
    const SlotPtrs& P = ptrs[slot];
    if (st.status != ST_RUNNING || st.stab) return;   // BiCGStab slots run their own kernels
    using C = cplx<S>;
    const int par = st.iter & 1;
    typename LinkSel<S>::type U{reinterpret_cast<decltype(U.u)>(links), g.V};
    const S k = (S)kappa;
    Acc<S> sacc;   // sigma, |phat|^2, |Ap|^2
    CompC scomp;   // sigma of the gamma5 variant (FP32)
    if (PAIR) {
        FieldIn<S> inp{P.p, g.V}, inh{P.phat, g.V};
        for (int u = u0; u < u1; ++u) {
            const int s = map.site(g, u);
            if (s < 0) continue;
            C a[12], b[12], self[12];
            hop_site_pair<S>(g, U, inp, inh, s, a, b);
            inp.load(s, self);
#pragma unroll
            for (int c = 0; c < 12; ++c) a[c] = self[c] - k * a[c];
            Field<S>::store(P.Ap[par], g.V, s, a);
            inh.load(s, self);
#pragma unroll
            for (int c = 0; c < 12; ++c) {
                b[c] = self[c] - k * b[c];
                sacc.z = cdot_acc(sacc.z, self[c], a[c]);
                sacc.a = abs2_acc(sacc.a, self[c]);
                sacc.b = abs2_acc(sacc.b, a[c]);
            }
            Field<S>::store(P.Ahp[par], g.V, s, b);
        }
    } else {
        FieldIn<S> in{which ? P.phat : P.p, g.V};
        void* out = which ? P.Ahp[par] : P.Ap[par];
        const bool win = G5 && st.m > 0;
        for (int u = u0; u < u1; ++u) {
            const int s = map.site(g, u);
            if (s < 0) continue;
            C acc[12], self[12];
            if (which) hop_site<true, S>(g, U, in, s, acc);
            else hop_site<false, S>(g, U, in, s, acc);
            in.load(s, self);
            const C (&self_p)[12] = self;
#pragma unroll
            for (int c = 0; c < 12; ++c) acc[c] = self[c] - k * acc[c];
            Field<S>::store(out, g.V, s, acc);
            if (G5) {   // phat = gamma5 p: spins 0, 1 (c < 6) keep their sign
#pragma unroll
                for (int c = 0; c < 12; ++c) {
                    const C ph = c < 6 ? self_p[c] : -self_p[c];
                    if constexpr (sizeof(S) == 4) scomp.add(cdot(ph, acc[c]));
                    else sacc.z = cdot_acc(sacc.z, ph, acc[c]);
                    sacc.a = abs2_acc(sacc.a, ph);
                    sacc.b = abs2_acc(sacc.b, acc[c]);
                }
                if (win) {
#pragma unroll
                    for (int c = 6; c < 12; ++c) acc[c] = -acc[c];
                    Field<S>::store(P.Ahp[par], g.V, s, acc);
                }
            } else if (!which) {
                C ph[12];
                Field<S>::load(P.phat, g.V, s, ph);
#pragma unroll
                for (int c = 0; c < 12; ++c) {
                    sacc.z = cdot_acc(sacc.z, ph[c], acc[c]);
                    sacc.a = abs2_acc(sacc.a, ph[c]);
                    sacc.b = abs2_acc(sacc.b, acc[c]);
                }
            }
        }
        if (which) return;
    }
    double2 tot[2];
    if (reduce2<S>(P, CNT_MATVEC, G5 && sizeof(S) == 4, scomp, sacc, tot, nsb, sblock) && threadIdx.x == 0) {
        finish_sigma(st, tot[0], tot[1].x, tot[1].y, G5 ? 1 : 2);   // the gamma5 variant applies A only
    }
}

// Operator pair with one warp per (32-site group, job): a block holds the
// jobs (slot, operator) of up to JPB/2 slots for the same sites, so the link
// loads of one site group are shared through L1 by every job of the block.
// Blocks loop over site groups (grid-stride, a fixed grid independent of the
// number of slots, so each slot's sigma partition does not depend on the
// batch). sigma: per-lane FP32 sums, warp sums, one FP64 partial per (block,
// slot) in that slot's partial buffer; the last block of the launch (one
// counter in slot 0) adds each slot's partials in block order.
constexpr int GRP_BLOCKS = 4 * 152;   // blocks per job half (fixed)
template <int JPB, int MINB>
__global__ void __launch_bounds__(32 * JPB, MINB)
    matvec_group_kernel(Geom g, const void* links, float kappa, SlotState* states, const SlotPtrs* ptrs,
                        int nslots) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int njobs = 2 * nslots;
    const int job = blockIdx.y * JPB + warp;
    const int slot = job >> 1, which = job & 1;
    const int ngroups = (g.V + 31) >> 5;
    LinksF U{reinterpret_cast<const float4*>(links), g.V};
    Acc<float> sacc;
    if (job < njobs && states[slot].status == ST_RUNNING && !states[slot].stab) {
        const SlotState& st = states[slot];
        const SlotPtrs& P = ptrs[slot];
        const int par = st.iter & 1;
        FieldIn<float> in{which ? P.phat : P.p, g.V};
        void* out = which ? P.Ahp[par] : P.Ap[par];
        for (int grp = blockIdx.x; grp < ngroups; grp += gridDim.x) {
            const int s = (grp << 5) + lane;
            if (s >= g.V) break;
            float2 acc[12], self[12];
            if (which) hop_site<true, float>(g, U, in, s, acc);
            else hop_site<false, float>(g, U, in, s, acc);
            in.load(s, self);
#pragma unroll
            for (int c = 0; c < 12; ++c) acc[c] = self[c] - kappa * acc[c];
            Field<float>::store(out, g.V, s, acc);
            if (!which) {
                float2 ph[12];
                Field<float>::load(P.phat, g.V, s, ph);
#pragma unroll
                for (int c = 0; c < 12; ++c) {
                    sacc.z = cdot_acc(sacc.z, ph[c], acc[c]);
                    sacc.a = abs2_acc(sacc.a, ph[c]);
                    sacc.b = abs2_acc(sacc.b, acc[c]);
                }
            }
        }
        if (!which) {
            float2 z = warp_sum(sacc.z);
            float2 ab = warp_sum(make_float2(sacc.a, sacc.b));
            if (lane == 0) {
                double2* pp = P.partials + (size_t)CNT_MATVEC * PARTIAL_STRIDE + (size_t)blockIdx.x * 2;
                pp[0] = to_d(z);
                pp[1] = to_d(ab);
                __threadfence();
            }
        }
    }
    // one arrival per block; the last block finishes every slot
    if (!last_block(ptrs[0].counters + CNT_GROUP, gridDim.x * gridDim.y)) return;
    for (int sl = warp; sl < nslots; sl += JPB) {
        SlotState& st = states[sl];
        if (st.status != ST_RUNNING || st.stab) continue;
        const double2* pp = ptrs[sl].partials + (size_t)CNT_MATVEC * PARTIAL_STRIDE;
        double2 z = make_double2(0.0, 0.0), ab = make_double2(0.0, 0.0);
        for (int b = lane; b < (int)gridDim.x; b += 32) {
            z = z + __ldcg(pp + 2 * b);
            ab = ab + __ldcg(pp + 2 * b + 1);
        }
        z = warp_sum(z);
        ab = warp_sum(ab);
        if (lane == 0) {
            finish_sigma(st, z, ab.x, ab.y, 2);
        }
    }
}

// r_j = r_{j-1} - alpha A p; rhat_j = rhat_{j-1} - conj(alpha) A^+ phat;
// rho_j, ||r_j||, ||rhat_j||; flags for the FP64 residual check. The solution
// update x_lo += alpha p is owed (x_owed): the direction update, which reads p
// anyway, or the reliable-update fold, or the final fold adds it.
template <typename S>
__global__ void __launch_bounds__(BL_THREADS) update_kernel(SlotState* states, const SlotPtrs* ptrs, size_t N) {
    SlotState& st = states[blockIdx.y];
    const SlotPtrs& P = ptrs[blockIdx.y];
    if (st.status != ST_RUNNING || st.stab) return;   // BiCGStab slots run their own kernels
    using C = cplx<S>;
    const int par = st.iter & 1;
    const C al = cvt<S>(st.alpha), alc = conj_(al);
    const void* rin = slot_field<S>(P.V, cur_slot(st), N);
    void* rout = slot_field<S>(P.V, next_slot(st), N);
    const void* hin = slot_field<S>(P.W, cur_slot(st), N);
    void* hout = slot_field<S>(P.W, next_slot(st), N);
    const void* ap = P.Ap[par];
    const void* ahp = P.Ahp[par];
    Acc<S> acc;   // rho_j, |r_j|^2, |rhat_j|^2
    CompC cz;     // rho_j of the gamma5 variant (FP32 storage)
    const bool comp = st.g5 && sizeof(S) == 4;
    const size_t units = N / 2;
    if (st.g5) {   // rhat_j = gamma5 r_j: one vector update, the window keeps gamma5 r_j
        const bool win = st.m > 0;
        for (size_t u = blockIdx.x * (size_t)blockDim.x + threadIdx.x; u < units; u += (size_t)gridDim.x * blockDim.x) {
            Unit<S> r = Unit<S>::load(rin, u), a = Unit<S>::load(ap, u);
            r.a = cfms(r.a, al, a.a); r.b = cfms(r.b, al, a.b);
            r.store(rout, u);
            const Unit<S> h = g5u(r, u, N);
            if (win) h.store(hout, u);
            if constexpr (sizeof(S) == 4) { cz.add(cdot(h.a, r.a)); cz.add(cdot(h.b, r.b)); }
            else acc.z = cdot_acc(cdot_acc(acc.z, h.a, r.a), h.b, r.b);
            acc.a += abs2(r.a) + abs2(r.b);
        }
        acc.b = acc.a;
    } else {
        for (size_t u = blockIdx.x * (size_t)blockDim.x + threadIdx.x; u < units; u += (size_t)gridDim.x * blockDim.x) {
            Unit<S> r = Unit<S>::load(rin, u), a = Unit<S>::load(ap, u);
            Unit<S> h = Unit<S>::load(hin, u), ah = Unit<S>::load(ahp, u);
            r.a = cfms(r.a, al, a.a); r.b = cfms(r.b, al, a.b);
            h.a = cfms(h.a, alc, ah.a); h.b = cfms(h.b, alc, ah.b);
            r.store(rout, u);
            h.store(hout, u);
            acc.z = cdot_acc(cdot_acc(acc.z, h.a, r.a), h.b, r.b);
            acc.a = abs2_two(acc.a, r.a, r.b);
            acc.b = abs2_two(acc.b, h.a, h.b);
        }
    }
    double2 tot[2];
    if (reduce2<S>(P, CNT_UPDATE, comp, cz, acc, tot, gridDim.x, blockIdx.x) && threadIdx.x == 0) {
        st.rho_new = tot[0];
        st.rnorm_new = sqrt_fp64(tot[1].x);
        st.rhat_norm = sqrt_fp64(tot[1].y);
        st.x_owed = 1;
        if (!isfinite(st.rnorm_new) || !isfinite(st.rho_new.x) || !isfinite(st.rho_new.y)) {
            st.status = ST_BREAKDOWN;
            st.live = 0;
        } else {
            // Reliable update (FP32 Krylov vectors): when the residual has dropped by
            // delta since the last update, or far below the largest residual seen
            // since then (the recursion's rounding error scales with that maximum);
            // and always to confirm convergence. A slot with rec_stop set (the
            // eigBiCG leg of a mixed-precision solve) never replaces r, which
            // would break the Lanczos relation of its window, and stops at the
            // first recursive convergence candidate instead.
            if (st.rnorm_new <= st.tol * st.bnorm) {
                if (st.rec_stop) st.status = ST_CONVERGED;
                else st.need_ru = 1;
            }
            if (st.rnorm_new > st.rmax) st.rmax = st.rnorm_new;
            if (st.delta > 0.0 && (st.rnorm_new < st.delta * st.r_ru || st.rnorm_new < 1e-3 * st.rmax)) st.need_ru = 1;
            // gamma5 variant with FP32 vectors: its shadow recursion can lose its
            // biorthogonality for good, which rounding decides (about one deflated solve
            // in twelve on a near-free 4^4 field, whatever the kernels). A residual whose
            // minimum has not halved in stall_lim iterations is taken for lost: the solve
            // starts over with a fresh direction, from the current x if its residual is
            // below that of every update so far, else from the best x of them (a second
            // time from the same x would repeat the first: then from the current x if its
            // residual is not far above). stall_lim is at least four times the iterations of
            // any update so far, so that slow convergence is not a stall, and doubles with
            // each restart. Solves that fail: near-free 4^4, 35 of 336 without restarts, 7
            // with them; 6^4 at kappa 0.130 and 0.134, 8 of 16 and none; 4^3 x 6 past critical
            // (0.16) end at 3e-5 to 0.2 ||b||, without restarts at 0.01 to 2e5. (Restarts
            // after 200 iterations without an update, from whatever x there was, ended there
            // at up to 1e15 and did not wait for slow solves.)
            if (st.g5 && st.delta > 0.0) {
                if (st.rnorm_new < 0.5 * st.r_min) { st.r_min = st.rnorm_new; st.min_iter = st.iter; }
                if (!st.need_ru && st.iter - st.min_iter >= st.stall_lim) {
                    st.need_ru = 1;
                    st.fresh_dir = st.rnorm_new < (st.best_used ? 1e3 : 1.0) * st.r_best ? FRESH_HERE : FRESH_BEST;
                }
            }
            if (!st.need_ru) bicg_scalars(st, P);   // else the reliable update ends the iteration
        }
    }
}

// FP64 true residual r = b - A x_hi at the end of a solve, for every slot that was
// started (x_lo has been folded into x_hi just before).
template <int THREADS, int MINB>
__global__ void __launch_bounds__(THREADS, MINB) true_resid_kernel(Geom g, const void* links64, double kappa,
                                                                   SlotState* states, const SlotPtrs* ptrs) {
    SlotState& st = states[blockIdx.y];
    const SlotPtrs& P = ptrs[blockIdx.y];
    if (st.status == ST_IDLE) return;
    LinksD U{reinterpret_cast<const double2*>(links64), g.V};
    FieldIn<double> in{P.x_hi, g.V};
    double2 v[1] = {make_double2(0, 0)};
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < g.V; s += gridDim.x * blockDim.x) {
        double2 acc[12], self[12], b[12];
        hop_site<false, double>(g, U, in, s, acc);
        in.load(s, self);
        Field<double>::load(P.b, g.V, s, b);
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            acc[c] = b[c] - make_double2(fma(-kappa, acc[c].x, self[c].x), fma(-kappa, acc[c].y, self[c].y));
            v[0].x = abs2_acc(v[0].x, acc[c]);
        }
        Field<double>::store(P.r_true, g.V, s, acc);
    }
    double2 tot[1];
    if (reduce_slot<1>(P, CNT_RU, v, tot, gridDim.x, blockIdx.x) && threadIdx.x == 0) {
        st.true_rnorm = sqrt_fp64(tot[0].x);
        st.matvecs += 1;
    }
}

// p_j = r_j + beta p_{j-1}, phat_j = rhat_j + conj(beta) phat_{j-1}.
template <typename S>
__global__ void __launch_bounds__(BL_THREADS) direction_kernel(SlotState* states, const SlotPtrs* ptrs, size_t N) {
    const SlotState& st = states[blockIdx.y];
    const SlotPtrs& P = ptrs[blockIdx.y];
    if (st.status != ST_RUNNING || st.stab) return;   // BiCGStab slots run their own kernels
    using C = cplx<S>;
    const C be = cvt<S>(st.beta), bec = conj_(be);
    const C al = cvt<S>(st.alpha);
    const bool addx = st.x_dir != 0;
    const bool g5 = st.g5 != 0;   // gamma5 variant: phat = gamma5 p is never stored
    const void* r = slot_field<S>(P.V, cur_slot(st), N);
    const void* h = slot_field<S>(P.W, cur_slot(st), N);
    const size_t units = N / 2;
    for (size_t u = blockIdx.x * (size_t)blockDim.x + threadIdx.x; u < units; u += (size_t)gridDim.x * blockDim.x) {
        Unit<S> p = Unit<S>::load(P.p, u), ph, hh, rr = Unit<S>::load(r, u);
        if (!g5) { ph = Unit<S>::load(P.phat, u); hh = Unit<S>::load(h, u); }
        if (addx) {   // x_lo += alpha p_{j-1} (owed by the residual update)
            Unit<S> x = Unit<S>::load(P.x_lo, u);
            x.a = cfma(x.a, al, p.a); x.b = cfma(x.b, al, p.b);
            x.store(P.x_lo, u);
        }
        p.a = cfma(rr.a, be, p.a); p.b = cfma(rr.b, be, p.b);
        p.store(P.p, u);
        if (!g5) {
            ph.a = cfma(hh.a, bec, ph.a); ph.b = cfma(hh.b, bec, ph.b);
            ph.store(P.phat, u);
        }
    }
}

// ------------------------------------------------------------- BiCGStab
// The phase-2 solver of Alg. Incremental eigBiCG as the paper runs it (Sec. 2),
// BiCGStab (van der Vorst) with the shadow start rhat = r_0 (W slot 0):
//   p = r + beta (p - omega v);  v = A p;  alpha = rho / (rhat, v);  s = r - alpha v;
//   t = A s;  omega = (t, s) / (t, t);  x += alpha p + omega s;  r = s - omega t;
//   rho' = (rhat, r);  beta = (rho' / rho) (alpha / omega).
// Buffers of a slot: r in V slot 0, rhat in W slot 0, p, v = Ap[0], s in the phat
// buffer, t = Ahp[0]. Two products with A per step, none with A^+.

// p = r + beta (p - omega v); the first step (iter 0) takes p = r.
template <typename S>
__global__ void __launch_bounds__(BL_THREADS) stab_dir_kernel(SlotState* states, const SlotPtrs* ptrs, size_t N) {
    const SlotState& st = states[blockIdx.y];
    const SlotPtrs& P = ptrs[blockIdx.y];
    if (st.status != ST_RUNNING || !st.stab) return;
    using C = cplx<S>;
    const C be = cvt<S>(st.beta), om = cvt<S>(st.omega);
    const bool first = st.iter == 0;
    const size_t units = N / 2;
    for (size_t u = blockIdx.x * (size_t)blockDim.x + threadIdx.x; u < units; u += (size_t)gridDim.x * blockDim.x) {
        Unit<S> r = Unit<S>::load(P.V, u);
        if (!first) {
            const Unit<S> p = Unit<S>::load(P.p, u), v = Unit<S>::load(P.Ap[0], u);
            r.a = cfma(r.a, be, cfms(p.a, om, v.a));
            r.b = cfma(r.b, be, cfms(p.b, om, v.b));
        }
        r.store(P.p, u);
    }
}

// PHASE 1: v = A p, sigma = (rhat, v), alpha = rho / sigma.
// PHASE 2: t = A s, (t, s), (t, t), omega = (t, s) / (t, t).
// One job per slot (grid: site blocks x slots, slots fastest).
template <typename S, int THREADS, int MINB, int PHASE>
__global__ void __launch_bounds__(THREADS, MINB) stab_matvec_kernel(Geom g, const void* links, double kappa,
                                                                    SlotState* states, const SlotPtrs* ptrs,
                                                                    int nslots) {
    const int slot = blockIdx.x % nslots, sblock = blockIdx.x / nslots, nsb = gridDim.x / nslots;
    SlotState& st = states[slot];
    const SlotPtrs& P = ptrs[slot];
    if (st.status != ST_RUNNING || !st.stab) return;
    using C = cplx<S>;
    typename LinkSel<S>::type U{reinterpret_cast<decltype(U.u)>(links), g.V};
    FieldIn<S> in{PHASE == 1 ? P.p : P.phat, g.V};
    void* out = PHASE == 1 ? P.Ap[0] : P.Ahp[0];
    const S k = (S)kappa;
    Acc<S> acc;   // PHASE 1: (rhat, v), |rhat|^2, |v|^2;  PHASE 2: (t, s), (t, t), |s|^2
    for (int s = sblock * blockDim.x + threadIdx.x; s < g.V; s += nsb * blockDim.x) {
        C o[12], self[12];
        hop_site<false, S>(g, U, in, s, o);
        in.load(s, self);
#pragma unroll
        for (int c = 0; c < 12; ++c) o[c] = self[c] - k * o[c];
        Field<S>::store(out, g.V, s, o);
        if (PHASE == 1) {
            C h[12];
            Field<S>::load(P.W, g.V, s, h);
#pragma unroll
            for (int c = 0; c < 12; ++c) {
                acc.z = cdot_acc(acc.z, h[c], o[c]);
                acc.a = abs2_acc(acc.a, h[c]);
                acc.b = abs2_acc(acc.b, o[c]);
            }
        } else {
#pragma unroll
            for (int c = 0; c < 12; ++c) {
                acc.z = cdot_acc(acc.z, o[c], self[c]);
                acc.a = abs2_acc(acc.a, o[c]);
                acc.b = abs2_acc(acc.b, self[c]);
            }
        }
    }
    cplx<S> v[2];
    acc.to(v);
    double2 tot[2];
    if (reduce_slot<2>(P, CNT_MATVEC, v, tot, nsb, sblock) && threadIdx.x == 0) {
        if (PHASE == 1) {
            finish_sigma(st, tot[0], tot[1].x, tot[1].y, 1);
        } else {
            st.matvecs += 1;
            st.ts = tot[0];
            st.tt = tot[1].x;
            st.omega = st.tt > 0.0 ? rcp_fp64(st.tt) * st.ts : make_double2(0.0, 0.0);
        }
    }
}

// s = r - alpha v  (into the phat buffer)
template <typename S>
__global__ void __launch_bounds__(BL_THREADS) stab_s_kernel(SlotState* states, const SlotPtrs* ptrs, size_t N) {
    const SlotState& st = states[blockIdx.y];
    const SlotPtrs& P = ptrs[blockIdx.y];
    if (st.status != ST_RUNNING || !st.stab) return;
    const cplx<S> al = cvt<S>(st.alpha);
    const size_t units = N / 2;
    for (size_t u = blockIdx.x * (size_t)blockDim.x + threadIdx.x; u < units; u += (size_t)gridDim.x * blockDim.x) {
        Unit<S> r = Unit<S>::load(P.V, u);
        const Unit<S> v = Unit<S>::load(P.Ap[0], u);
        r.a = cfms(r.a, al, v.a);
        r.b = cfms(r.b, al, v.b);
        r.store(P.phat, u);
    }
}

// x_lo += alpha p + omega s;  r = s - omega t;  rho' = (rhat, r), ||r||; the
// reliable-update flags as in the BiCG residual update.
template <typename S>
__global__ void __launch_bounds__(BL_THREADS) stab_update_kernel(SlotState* states, const SlotPtrs* ptrs, size_t N) {
    SlotState& st = states[blockIdx.y];
    const SlotPtrs& P = ptrs[blockIdx.y];
    if (st.status != ST_RUNNING || !st.stab) return;
    using C = cplx<S>;
    const C al = cvt<S>(st.alpha), om = cvt<S>(st.omega);
    Acc<S> acc;   // rho', |r|^2
    const size_t units = N / 2;
    for (size_t u = blockIdx.x * (size_t)blockDim.x + threadIdx.x; u < units; u += (size_t)gridDim.x * blockDim.x) {
        Unit<S> x = Unit<S>::load(P.x_lo, u);
        const Unit<S> p = Unit<S>::load(P.p, u), sv = Unit<S>::load(P.phat, u), t = Unit<S>::load(P.Ahp[0], u);
        const Unit<S> h = Unit<S>::load(P.W, u);
        x.a = cfma(cfma(x.a, al, p.a), om, sv.a);
        x.b = cfma(cfma(x.b, al, p.b), om, sv.b);
        x.store(P.x_lo, u);
        Unit<S> r{cfms(sv.a, om, t.a), cfms(sv.b, om, t.b)};
        r.store(P.V, u);
        acc.z = cdot_acc(cdot_acc(acc.z, h.a, r.a), h.b, r.b);
        acc.a = abs2_two(acc.a, r.a, r.b);
    }
    cplx<S> v[2];
    acc.to(v);
    double2 tot[2];
    if (reduce_slot<2>(P, CNT_UPDATE, v, tot, gridDim.x, blockIdx.x) && threadIdx.x == 0) {
        st.rho_new = tot[0];
        st.rnorm_new = sqrt_fp64(tot[1].x);
        st.x_owed = 0;   // x is complete after this step
        if (!isfinite(st.rnorm_new) || !isfinite(st.rho_new.x) || !isfinite(st.rho_new.y)) {
            st.status = ST_BREAKDOWN;
        } else {
            if (st.rnorm_new <= st.tol * st.bnorm) st.need_ru = 1;
            if (st.rnorm_new > st.rmax) st.rmax = st.rnorm_new;
            if (st.delta > 0.0 && (st.rnorm_new < st.delta * st.r_ru || st.rnorm_new < 1e-3 * st.rmax)) st.need_ru = 1;
            if (!st.need_ru) stab_scalars(st);
        }
    }
}

// Fold x_lo into x_hi at the end of a solve (x = 0 for a zero source).
template <typename S>
__global__ void fold_kernel(SlotState* states, const SlotPtrs* ptrs, size_t N) {
    const SlotState& st = states[blockIdx.y];
    const SlotPtrs& P = ptrs[blockIdx.y];
    if (st.status == ST_IDLE) return;
    const bool zero_src = st.bnorm == 0.0;
    // a gamma5 solve that failed returns its best x (see ru_kernel)
    const bool back = sizeof(S) == 4 && st.g5 && st.delta > 0.0 && st.status != ST_CONVERGED && !(st.rnorm_new <= st.r_best);
    const bool owed = st.x_owed != 0 && !back;   // the last residual update's alpha p (no direction update ran)
    const cplx<S> al = cvt<S>(st.alpha);
    const size_t units = N / 2;
    Unit<S> zero{mk<S>(0, 0), mk<S>(0, 0)};
    for (size_t u = blockIdx.x * (size_t)blockDim.x + threadIdx.x; u < units; u += (size_t)gridDim.x * blockDim.x) {
        Unit<double> xh = Unit<double>::load(back && !st.x_best ? P.r_true : P.x_hi, u);
        Unit<S> xl = back ? zero : Unit<S>::load(P.x_lo, u);
        if (owed) {
            const Unit<S> p = Unit<S>::load(P.p, u);
            xl.a = cfma(xl.a, al, p.a); xl.b = cfma(xl.b, al, p.b);
        }
        if (zero_src) { xh.a = make_double2(0, 0); xh.b = make_double2(0, 0); }
        else { xh.a = xh.a + wid(xl.a); xh.b = xh.b + wid(xl.b); }
        xh.store(P.x_hi, u);
        zero.store(P.x_lo, u);
    }
}

// -------------------------------------------------------- restart product
// In-place window product of the BiCG-eigen restart (one job per slot and side):
//   new slot k = sum_{i<m} scale_i coef[i][k] old slot i   (k < r)
//   new slot r = old slot m                                  (r_{j-1}, appended next)
// with the coupling dots of the new vectors:
//   V side: H[r][k] = (||r_{j-1}|| / rho_{j-1}) (A^+ phat - conj(beta_{j-2}) s)^H v_k
//   W side: H[k][r] = (1 / ||r_{j-1}||) w_k^H (A p - beta_{j-2} q)
// where q, s are the products of the previous iteration (Algorithm eigBiCG).
//
// Register tiling: a block covers tiles of WG_E * WG_T elements; each of the
// RMAX / WG_K column groups computes WG_K output columns for WG_E elements per
// thread, so one shared-memory coefficient read serves WG_E elements. All
// groups read a tile's inputs before any group overwrites them (one block
// barrier per tile: the product is in place).
constexpr int WG_E = 4, WG_K = 8, WG_T = 64;

template <typename S, int RMAX>
__global__ void __launch_bounds__(WG_T * ((RMAX + WG_K - 1) / WG_K))
    window_gemm_kernel(SlotState* states, const SlotPtrs* ptrs, size_t N) {
    constexpr int G = (RMAX + WG_K - 1) / WG_K;
    const int slot = blockIdx.y >> 1, side = blockIdx.y & 1;
    SlotState& st = states[slot];
    const SlotPtrs& P = ptrs[slot];
    if (st.status != ST_RUNNING || st.restart_r == 0) return;
    using C = cplx<S>;
    const int m = st.m, r = st.restart_r, ldc = 2 * st.nev + 1;
    const int par = st.iter & 1;
    __shared__ C Cs[MAX_M * RMAX];
    const double2* coef = side ? P.coefZ : P.coefY;
    for (int q = threadIdx.x; q < m * RMAX; q += blockDim.x) {
        const int i = q / RMAX, k = q % RMAX;
        double2 v = make_double2(0.0, 0.0);
        if (k < r) {
            double2 sc = side ? P.wscale[i] : make_double2(P.vscale[i], 0.0);
            v = sc * coef[i * ldc + k];
        }
        Cs[q] = cvt<S>(v);
    }
    __syncthreads();
    const int g = threadIdx.x / WG_T, t = threadIdx.x % WG_T, k0 = g * WG_K;
    // coupling vector: V side c = A^+phat - conj(beta) s ; W side a = A p - beta q
    const C bp = cvt<S>(side ? st.beta_prev : conj_(st.beta_prev));
    const void* cur = side ? P.Ap[par] : P.Ahp[par];
    const void* prv = side ? P.Ap[par ^ 1] : P.Ahp[par ^ 1];
    void* base = side ? P.W : P.V;
    C dot[WG_K];
#pragma unroll
    for (int kk = 0; kk < WG_K; ++kk) dot[kk] = mk<S>(S(0), S(0));
    const size_t tile = (size_t)WG_E * WG_T;
    for (size_t e0 = (size_t)blockIdx.x * tile; e0 < N; e0 += (size_t)gridDim.x * tile) {
        const size_t eb = e0 + (size_t)t * WG_E;
        const int ne = eb >= N ? 0 : (int)min((size_t)WG_E, N - eb);
        C out[WG_E][WG_K];
#pragma unroll
        for (int e = 0; e < WG_E; ++e)
#pragma unroll
            for (int kk = 0; kk < WG_K; ++kk) out[e][kk] = mk<S>(S(0), S(0));
        // inputs of slot i+1 are loaded while slot i is multiplied (software pipelining)
        C x[WG_E], xn[WG_E];
        {
            const C* src = reinterpret_cast<const C*>(base) + eb;
#pragma unroll
            for (int e = 0; e < WG_E; ++e) x[e] = e < ne ? src[e] : mk<S>(S(0), S(0));
        }
        for (int i = 0; i < m; ++i) {
            if (i + 1 < m) {
                const C* src = reinterpret_cast<const C*>(slot_field<S>(base, i + 1, N)) + eb;
#pragma unroll
                for (int e = 0; e < WG_E; ++e) xn[e] = e < ne ? src[e] : mk<S>(S(0), S(0));
            }
#pragma unroll
            for (int kk = 0; kk < WG_K; ++kk) {
                const C c = Cs[i * RMAX + k0 + kk];
#pragma unroll
                for (int e = 0; e < WG_E; ++e) out[e][kk] = out[e][kk] + x[e] * c;
            }
#pragma unroll
            for (int e = 0; e < WG_E; ++e) x[e] = xn[e];
        }
        C last[WG_E], cv[WG_E];
        {
            const C* lsrc = reinterpret_cast<const C*>(slot_field<S>(base, m, N)) + eb;
            const C* cs = reinterpret_cast<const C*>(cur) + eb;
            const C* ps = reinterpret_cast<const C*>(prv) + eb;
#pragma unroll
            for (int e = 0; e < WG_E; ++e) {
                last[e] = (g == 0 && e < ne) ? lsrc[e] : mk<S>(S(0), S(0));
                cv[e] = e < ne ? cs[e] - bp * ps[e] : mk<S>(S(0), S(0));
            }
        }
        __syncthreads();   // every group has read this tile's inputs
#pragma unroll
        for (int kk = 0; kk < WG_K; ++kk) {
            const int k = k0 + kk;
            if (k < r) {
                C* dst = reinterpret_cast<C*>(slot_field<S>(base, k, N)) + eb;
#pragma unroll
                for (int e = 0; e < WG_E; ++e)
                    if (e < ne) {
                        dst[e] = out[e][kk];
                        dot[kk] = dot[kk] + (side ? cdot(out[e][kk], cv[e]) : cdot(cv[e], out[e][kk]));
                    }
            }
        }
        if (g == 0) {
            C* dst = reinterpret_cast<C*>(slot_field<S>(base, r, N)) + eb;
#pragma unroll
            for (int e = 0; e < WG_E; ++e)
                if (e < ne) dst[e] = last[e];
        }
    }
    // block sums of the coupling dots: warp shuffles, then one value per thread
    __shared__ double2 wdot[(WG_T * G / 32) * WG_K];
    __shared__ bool am_last;
#pragma unroll
    for (int kk = 0; kk < WG_K; ++kk) {
        double2 d = warp_sum(to_d(dot[kk]));
        if ((threadIdx.x & 31) == 0) wdot[(threadIdx.x >> 5) * WG_K + kk] = d;
    }
    __syncthreads();
    constexpr int WPG = WG_T / 32;   // warps per column group
    double2* pp = P.partials + (size_t)(side ? CNT_GEMM_W : CNT_GEMM_V) * PARTIAL_STRIDE;
    const int q = threadIdx.x;       // output column q = group * WG_K + kk
    if (q < G * WG_K) {
        double2 acc = make_double2(0.0, 0.0);
        for (int w = 0; w < WPG; ++w) acc = acc + wdot[((q / WG_K) * WPG + w) * WG_K + q % WG_K];
        pp[(size_t)blockIdx.x * (G * WG_K) + q] = acc;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned prev = atomicAdd(P.counters + (side ? CNT_GEMM_W : CNT_GEMM_V), 1u);
        am_last = (prev == gridDim.x - 1);
        if (am_last) P.counters[side ? CNT_GEMM_W : CNT_GEMM_V] = 0;
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    if (q < r) {
        // the last block adds the partials in block order (deterministic)
        double2 tot = make_double2(0.0, 0.0);
        for (unsigned b = 0; b < gridDim.x; ++b) tot = tot + __ldcg(pp + (size_t)b * (G * WG_K) + q);
        // the new basis vectors are stored normalised: their window scale is 1
        if (side) {
            P.H[q * m + r] = (1.0 / st.rnorm) * tot;
            P.wscale[q] = make_double2(1.0, 0.0);
        } else {
            P.H[r * m + q] = cdiv(make_double2(st.rnorm, 0.0), st.rho) * tot;
            P.vscale[q] = 1.0;
        }
    }
}

}  // namespace

// ------------------------------------------------------------------ launchers
static Geom geom_of(const Geom& g) { return g; }

static long long g_launches = 0;
void count_launches(long long n) { g_launches += n; }
long long launches_so_far() { return g_launches; }
void set_launches(long long n) { g_launches = n; }

cudaError_t launch_apply(const Geom& g, const void* links, double kappa, int precision, const void* in, void* out,
                         const double2* aux, int dagger, int nf, cudaStream_t st) {
    int grid = ds_blocks(g.V) * nf;
    if (precision == 0 && fp64_split_ok(g.V, nf)) {
        count_launches(1);
        return launch_apply_split(g, links, kappa, in, out, aux, dagger, nf, st);
    }
    if (precision == 0) {
        const int t = site_threads(g.V, nf, DS_THREADS);
        if (t == 32) grid = div_up(g.V, 32) * nf;
        if (aux) apply_kernel<double, true><<<grid, t, 0, st>>>(geom_of(g), links, kappa, in, out, aux, dagger, nf);
        else apply_kernel<double, false><<<grid, t, 0, st>>>(geom_of(g), links, kappa, in, out, aux, dagger, nf);
    } else {
        if (aux) return cudaErrorInvalidValue;
        apply_kernel<float, false><<<grid, DS_THREADS, 0, st>>>(geom_of(g), links, kappa, in, out, aux, dagger, nf);
    }
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_residual32(const Geom& g, const void* links32, double kappa, const double2* x, void* x32,
                              const double2* b, void* r, int rprec, int nf, cudaStream_t st) {
    cudaError_t e = launch_convert(x, 0, x32, 1, (size_t)nf * 12 * g.V, st);
    if (e != cudaSuccess) return e;
    const int grid = ds_blocks(g.V) * nf;
    const float4* U = reinterpret_cast<const float4*>(links32);
    const float2* xs = reinterpret_cast<const float2*>(x32);
    if (rprec) residual32_kernel<float><<<grid, DS_THREADS, 0, st>>>(g, U, kappa, x, xs, b, reinterpret_cast<float2*>(r), nf);
    else residual32_kernel<double><<<grid, DS_THREADS, 0, st>>>(g, U, kappa, x, xs, b, reinterpret_cast<double2*>(r), nf);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_pack(const double* aos, void* dev, int V, int k, int precision, cudaStream_t st) {
    const dim3 grid(div_up(V, PK_SITES), k);
    const double2* src = reinterpret_cast<const double2*>(aos);
    if (precision == 0) pack_kernel<double><<<grid, BL_THREADS, 0, st>>>(src, reinterpret_cast<double2*>(dev), V);
    else pack_kernel<float><<<grid, BL_THREADS, 0, st>>>(src, reinterpret_cast<float2*>(dev), V);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t launch_unpack(const void* dev, double* aos, int V, int k, int precision, cudaStream_t st) {
    const dim3 grid(div_up(V, PK_SITES), k);
    double2* dst = reinterpret_cast<double2*>(aos);
    if (precision == 0) unpack_kernel<double><<<grid, BL_THREADS, 0, st>>>(reinterpret_cast<const double2*>(dev), dst, V);
    else unpack_kernel<float><<<grid, BL_THREADS, 0, st>>>(reinterpret_cast<const float2*>(dev), dst, V);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t launch_convert(const void* src, int sp, void* dst, int dp, size_t n, cudaStream_t st) {
    int nb = blas_blocks(n);
    if (sp == 0 && dp == 1) convert_kernel<double, float><<<nb, BL_THREADS, 0, st>>>(src, dst, n);
    else if (sp == 1 && dp == 0) convert_kernel<float, double><<<nb, BL_THREADS, 0, st>>>(src, dst, n);
    else if (sp == 0 && dp == 0) convert_kernel<double, double><<<nb, BL_THREADS, 0, st>>>(src, dst, n);
    else convert_kernel<float, float><<<nb, BL_THREADS, 0, st>>>(src, dst, n);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_multidot(int a, const void* X, int xp, int b, const void* Y, int yp, size_t N, double2* Cm,
                            int ldc, int conj_store, double2* scratch, size_t scratch_elems, cudaStream_t st,
                            int* err, int staged) {
    if (a <= 0 || b <= 0) return cudaSuccess;
    // The tensor-core form takes a tile of 128 X against 24 Y fields whatever part of it is
    // filled (4.3 ms at N = 10.6 M), the FP32 form 1.35 ms per 80 X and 8 Y fields: 128 x 24
    // cost as much as 252 x 8. With a <= MAX_SMALL = 80 fields the line is never crossed; the
    // blocks beyond it come from lqcd_field_dots.
    if (staged && xp == 1 && yp == 1 && div_up(b, 8) * a > 252 * div_up(a, 128) * div_up(b, 24) &&
        dots_tc_supported(a, X, Y, N) && dots_tc_scratch_doubles(a) <= 2 * scratch_elems)
        return launch_dots_tc(a, X, N * 8, b, Y, N * 8, N, Cm, ldc, conj_store, reinterpret_cast<double*>(scratch),
                              2 * scratch_elems, err, st);
    if (staged && err && xp == 1 && yp == 1 && dots_supported(a, X, Y, N) && dots_scratch(a, b, N) <= scratch_elems)
        return launch_dots(a, X, b, Y, N, Cm, ldc, conj_store, scratch, scratch_elems, err, st);
    for (int j0 = 0; j0 < b; j0 += MD_BMAX) {
        const int bb = b - j0 < MD_BMAX ? b - j0 : MD_BMAX;
        const int nby = div_up(a, MD_TI);
        int nbx = blas_blocks(N) / 2;
        if (nbx < 1) nbx = 1;
        while ((size_t)nbx * nby * MD_TI * MD_BMAX > scratch_elems && nbx > 1) nbx /= 2;
        if ((size_t)nbx * nby * MD_TI * MD_BMAX > scratch_elems) return cudaErrorInvalidValue;
        const char* Yj = reinterpret_cast<const char*>(Y) + (size_t)j0 * N * (yp == 0 ? 16 : 8);
        const int grid = nbx * nby;
        if (xp == 1 && yp == 1) multidot_kernel<float, float, float><<<grid, BL_THREADS, 0, st>>>(a, X, bb, Yj, N, scratch, nby);
        else if (xp == 1 && yp == 0) multidot_kernel<float, double, double><<<grid, BL_THREADS, 0, st>>>(a, X, bb, Yj, N, scratch, nby);
        else if (xp == 0 && yp == 1) multidot_kernel<double, float, double><<<grid, BL_THREADS, 0, st>>>(a, X, bb, Yj, N, scratch, nby);
        else multidot_kernel<double, double, double><<<grid, BL_THREADS, 0, st>>>(a, X, bb, Yj, N, scratch, nby);
        count_launches(2);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        double2* Cj = conj_store ? Cm + j0 * ldc : Cm + j0;
        multidot_reduce_kernel<<<div_up((size_t)a * bb, 128), 128, 0, st>>>(a, bb, nbx, scratch, Cj, ldc, conj_store);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_vupdate(int a, const void* X, int xp, const double2* D, int ldd, int b, void* Y, int yp,
                           int overwrite, size_t N, cudaStream_t st, int fp64_arith) {
    if (a > MAX_SMALL || N % 2) return cudaErrorInvalidValue;   // fields hold 12 numbers per site
    for (int j0 = 0; j0 < b; j0 += MD_BMAX) {
        const int bb = b - j0 < MD_BMAX ? b - j0 : MD_BMAX;
        char* Yj = reinterpret_cast<char*>(Y) + (size_t)j0 * N * (yp == 0 ? 16 : 8);
        const double2* Dj = D + j0;
        int nb = blas_blocks(N);
        const float4* X4 = reinterpret_cast<const float4*>(X);
        if (xp == 1 && yp == 1) vupdate32_kernel<float><<<blas_blocks(N / 2), BL_THREADS, 0, st>>>(a, X4, Dj, ldd, bb, Yj, overwrite, N);
        else if (xp == 1 && yp == 0 && fp64_arith) vupdate_kernel<float, double, double><<<nb, BL_THREADS, 0, st>>>(a, X, Dj, ldd, bb, Yj, overwrite, N);
        else if (xp == 1 && yp == 0) vupdate32_kernel<double><<<blas_blocks(N / 2), BL_THREADS, 0, st>>>(a, X4, Dj, ldd, bb, Yj, overwrite, N);
        else if (xp == 0 && yp == 1) vupdate_kernel<double, float, double><<<nb, BL_THREADS, 0, st>>>(a, X, Dj, ldd, bb, Yj, overwrite, N);
        else vupdate_kernel<double, double, double><<<nb, BL_THREADS, 0, st>>>(a, X, Dj, ldd, bb, Yj, overwrite, N);
        count_launches(1);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_norms(int b, const void* Y, int yp, size_t N, double* out, double2* scratch,
                         size_t scratch_elems, cudaStream_t st) {
    if (b <= 0) return cudaSuccess;
    int nb = blas_blocks(N) / 2;
    if (nb < 1) nb = 1;
    while ((size_t)nb * b > scratch_elems && nb > 1) nb /= 2;
    dim3 grid(nb, b);
    if (yp == 0) norms_kernel<double><<<grid, BL_THREADS, 0, st>>>(Y, N, scratch);
    else norms_kernel<float><<<grid, BL_THREADS, 0, st>>>(Y, N, scratch);
    norms_reduce_kernel<<<(b + 63) / 64, 64, 0, st>>>(b, nb, scratch, out);
    count_launches(2);
    return cudaGetLastError();
}

cudaError_t launch_scale_fields(int b, void* Y, int yp, const double2* sc, size_t N, cudaStream_t st) {
    int nb = blas_blocks(N * b);
    if (yp == 0) scale_fields_kernel<double><<<nb, BL_THREADS, 0, st>>>(b, Y, sc, N);
    else scale_fields_kernel<float><<<nb, BL_THREADS, 0, st>>>(b, Y, sc, N);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_bicg_start(const Geom& g, const void* links64, double kappa, int prec, SlotState* states,
                              const SlotPtrs* ptrs, int nslots, size_t N, cudaStream_t s) {
    (void)g; (void)links64; (void)kappa;
    dim3 grid(blas_blocks(N / 2), nslots);
    if (prec == 0) start_kernel<double><<<grid, BL_THREADS, 0, s>>>(states, ptrs, N);
    else start_kernel<float><<<grid, BL_THREADS, 0, s>>>(states, ptrs, N);
    count_launches(1);
    return cudaGetLastError();
}

// SPT: sites per thread (grid-stride), which amortises each block's set-up and
// reduction tail over more sites.
template <typename S, int THREADS, int MINB, bool PAIR, int BZ = 0, int SPT = 1, bool G5 = false, bool TM = false>
static void matvec_launch(const Geom& g, const void* links, double kappa, SlotState* states, const SlotPtrs* ptrs,
                          int nslots, cudaStream_t s) {
    const int njobs = (PAIR || G5) ? nslots : 2 * nslots;
    int nb = div_up((size_t)g.V, (size_t)THREADS * SPT);
    if (nb > PARTIAL_STRIDE / 2) nb = PARTIAL_STRIDE / 2;
    matvec_kernel<S, THREADS, MINB, PAIR, BZ, G5, TM><<<nb * njobs, THREADS, 0, s>>>(g, links, kappa, states, ptrs,
                                                                                    njobs);
}
// The brick shapes need Lx, Ly multiples of 8 and Lz a multiple of BZ.
static bool brick_ok(const Geom& g, int bz) { return g.L[0] % 8 == 0 && g.L[1] % 8 == 0 && g.L[2] % bz == 0; }

template <int JPB, int MINB>
static void matvec_group_launch(const Geom& g, const void* links, double kappa, SlotState* states,
                                const SlotPtrs* ptrs, int nslots, cudaStream_t s) {
    const int njobs = 2 * nslots;
    dim3 grid(GRP_BLOCKS, (njobs + JPB - 1) / JPB);
    matvec_group_kernel<JPB, MINB><<<grid, 32 * JPB, 0, s>>>(g, links, (float)kappa, states, ptrs, nslots);
}

int matvec_variants() { return 30; }
bool matvec_variant_ok(const Geom& g, int v) {
    if (v == STAGED_VARIANT) return staged_variant_ok(g);
    if (v >= 25 && v < 30) return brick_variant_ok(g, v);
    if (v == 13 || v == 14) return brick_ok(g, 4);
    if (v == 15 || v == 23) return brick_ok(g, 2);
    if (v >= 19 && v < 25) return brick_ok(g, 4);
    return v >= 0 && v < 25;
}

cudaError_t launch_bicg_matvec(const Geom& g, const void* links, double kappa, int prec, SlotState* states,
                               const SlotPtrs* ptrs, int nslots, cudaStream_t s, int variant,
                                  int kmax) {
    if (prec != 0 && variant == STAGED_VARIANT) return cudaErrorInvalidValue;   // needs the context's tensor maps
    if (prec != 0 && variant >= 25 && variant < 30)   // 4-D bricks, every slot per block (dslash_brick.cu)
        return launch_matvec_brick(g, links, kappa, states, ptrs, nslots, s, variant);
    if (prec == 0) {
        if (fp64_split_ok(g.V, 2 * kmax)) {
            const cudaError_t e = launch_matvec_split(g, links, kappa, states, ptrs, nslots, s);
            if (e != cudaSuccess) return e;
        } else if (site_threads(g.V, 2 * kmax, 128) == 32) matvec_launch<double, 32, 8, false>(g, links, kappa, states, ptrs, nslots, s);
        else matvec_launch<double, 128, 1, false>(g, links, kappa, states, ptrs, nslots, s);
    } else {
        switch (variant) {
            case 1: matvec_launch<float, 128, 6, false>(g, links, kappa, states, ptrs, nslots, s); break;
            case 2: matvec_launch<float, 256, 3, false>(g, links, kappa, states, ptrs, nslots, s); break;
            case 3: matvec_launch<float, 128, 1, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 4: matvec_launch<float, 128, 4, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 5: matvec_launch<float, 128, 4, false>(g, links, kappa, states, ptrs, nslots, s); break;
            case 6: matvec_launch<float, 128, 5, false>(g, links, kappa, states, ptrs, nslots, s); break;
            case 7: matvec_launch<float, 128, 3, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 8: matvec_launch<float, 256, 2, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 9: matvec_launch<float, 64, 8, false>(g, links, kappa, states, ptrs, nslots, s); break;
            case 10: matvec_group_launch<8, 3>(g, links, kappa, states, ptrs, nslots, s); break;
            case 11: matvec_group_launch<8, 2>(g, links, kappa, states, ptrs, nslots, s); break;
            case 12: matvec_group_launch<16, 1>(g, links, kappa, states, ptrs, nslots, s); break;
            case 13: matvec_launch<float, 256, 3, false, 4>(g, links, kappa, states, ptrs, nslots, s); break;
            case 14: matvec_launch<float, 256, 2, true, 4>(g, links, kappa, states, ptrs, nslots, s); break;
            case 15: matvec_launch<float, 128, 4, true, 2>(g, links, kappa, states, ptrs, nslots, s); break;
            case 16: matvec_launch<float, 256, 3, false, 0, 4>(g, links, kappa, states, ptrs, nslots, s); break;
            case 17: matvec_launch<float, 128, 4, true, 0, 4>(g, links, kappa, states, ptrs, nslots, s); break;
            case 18: matvec_launch<float, 256, 2, true, 0, 2>(g, links, kappa, states, ptrs, nslots, s); break;
            // t march over 8 x 8 x BZ bricks (SPT consecutive t-planes per block)
            case 19: matvec_launch<float, 256, 1, true, 4, 8, false, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 20: matvec_launch<float, 256, 2, true, 4, 4, false, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 21: matvec_launch<float, 256, 1, false, 4, 8, false, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 22: matvec_launch<float, 256, 2, false, 4, 8, false, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 23: matvec_launch<float, 128, 2, true, 2, 8, false, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 24: matvec_launch<float, 256, 1, true, 4, 16, false, true>(g, links, kappa, states, ptrs, nslots, s); break;
            default: matvec_launch<float, 128, 1, false>(g, links, kappa, states, ptrs, nslots, s); break;
        }
    }
    count_launches(1);
    return cudaGetLastError();
}

// The gamma5 variant's operator (A p only, sigma with phat = gamma5 p): the
// one-operator shapes of the list above (per-site threads, no operator pairing).
bool matvec_g5_variant_ok(const Geom& g, int v) {
    switch (v) {
        case 0: case 1: case 2: case 5: case 6: case 9: case 16: return true;
        case 13: case 21: case 22: return brick_ok(g, 4);
        default: return false;
    }
}

cudaError_t launch_bicg_matvec_g5(const Geom& g, const void* links, double kappa, int prec, SlotState* states,
                                  const SlotPtrs* ptrs, int nslots, cudaStream_t s, int variant,
                                  int kmax) {
    if (prec == 0) {
        if (site_threads(g.V, kmax, 128) == 32) matvec_launch<double, 32, 8, false, 0, 1, true>(g, links, kappa, states, ptrs, nslots, s);
        else matvec_launch<double, 128, 1, false, 0, 1, true>(g, links, kappa, states, ptrs, nslots, s);
    } else {
        switch (variant) {
            case 1: matvec_launch<float, 128, 6, false, 0, 1, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 2: matvec_launch<float, 256, 3, false, 0, 1, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 5: matvec_launch<float, 128, 4, false, 0, 1, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 6: matvec_launch<float, 128, 5, false, 0, 1, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 9: matvec_launch<float, 64, 8, false, 0, 1, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 13: matvec_launch<float, 256, 3, false, 4, 1, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 16: matvec_launch<float, 256, 3, false, 0, 4, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 21: matvec_launch<float, 256, 1, false, 4, 8, true, true>(g, links, kappa, states, ptrs, nslots, s); break;
            case 22: matvec_launch<float, 256, 2, false, 4, 8, true, true>(g, links, kappa, states, ptrs, nslots, s); break;
            default: matvec_launch<float, 128, 1, false, 0, 1, true>(g, links, kappa, states, ptrs, nslots, s); break;
        }
    }
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_bicg_update(int prec, SlotState* states, const SlotPtrs* ptrs, int nslots, size_t N, cudaStream_t s,
                               int kmax) {
    dim3 grid(red_blocks(N / 2), nslots);
    const int t = site_threads(N / 2, kmax, BL_THREADS);
    if (prec == 0) update_kernel<double><<<t == 32 ? dim3(blas_blocks(N / 2 * (BL_THREADS / 32)), nslots) : grid, t, 0, s>>>(states, ptrs, N);
    else update_kernel<float><<<grid, BL_THREADS, 0, s>>>(states, ptrs, N);
    count_launches(1);
    return cudaGetLastError();
}

// FP64 true-residual shapes (threads, blocks per SM): FP64 arithmetic runs at a
// small fraction of the FP32 rate, so occupancy (latency hiding for the FP64
// pipe) decides; the library times them at init.
template <int THREADS, int MINB>
static void true_resid_launch(const Geom& g, const void* links64, double kappa, SlotState* states,
                              const SlotPtrs* ptrs, int nslots, cudaStream_t s) {
    int nb = div_up((size_t)g.V, THREADS);
    if (nb > PARTIAL_STRIDE / 2) nb = PARTIAL_STRIDE / 2;
    true_resid_kernel<THREADS, MINB><<<dim3(nb, nslots), THREADS, 0, s>>>(g, links64, kappa, states, ptrs);
}
int true_resid_variants() { return 4; }
cudaError_t launch_true_resid(int variant, const Geom& g, const void* links64, double kappa, SlotState* states,
                              const SlotPtrs* ptrs, int nslots, cudaStream_t s) {
    switch (variant) {
        case 1: true_resid_launch<128, 3>(g, links64, kappa, states, ptrs, nslots, s); break;
        case 2: true_resid_launch<128, 4>(g, links64, kappa, states, ptrs, nslots, s); break;
        case 3: true_resid_launch<64, 6>(g, links64, kappa, states, ptrs, nslots, s); break;
        default: true_resid_launch<128, 1>(g, links64, kappa, states, ptrs, nslots, s); break;
    }
    count_launches(1);
    return cudaGetLastError();
}

template <typename S, int THREADS, int MINB, int PHASE>
static void stab_matvec_launch(const Geom& g, const void* links, double kappa, SlotState* states,
                               const SlotPtrs* ptrs, int nslots, cudaStream_t s) {
    int nb = div_up((size_t)g.V, (size_t)THREADS * 2);
    if (nb > PARTIAL_STRIDE / 2) nb = PARTIAL_STRIDE / 2;
    stab_matvec_kernel<S, THREADS, MINB, PHASE><<<nb * nslots, THREADS, 0, s>>>(g, links, kappa, states, ptrs, nslots);
}

cudaError_t launch_stab_step(const Geom& g, const void* links, double kappa, int prec, SlotState* states,
                             const SlotPtrs* ptrs, int nslots, size_t N, cudaStream_t s) {
    dim3 grid(blas_blocks(N / 2), nslots);
    if (prec == 0) {
        stab_dir_kernel<double><<<grid, BL_THREADS, 0, s>>>(states, ptrs, N);
        stab_matvec_launch<double, 128, 1, 1>(g, links, kappa, states, ptrs, nslots, s);
        stab_s_kernel<double><<<grid, BL_THREADS, 0, s>>>(states, ptrs, N);
        stab_matvec_launch<double, 128, 1, 2>(g, links, kappa, states, ptrs, nslots, s);
        stab_update_kernel<double><<<grid, BL_THREADS, 0, s>>>(states, ptrs, N);
    } else {
        stab_dir_kernel<float><<<grid, BL_THREADS, 0, s>>>(states, ptrs, N);
        stab_matvec_launch<float, 128, 4, 1>(g, links, kappa, states, ptrs, nslots, s);
        stab_s_kernel<float><<<grid, BL_THREADS, 0, s>>>(states, ptrs, N);
        stab_matvec_launch<float, 128, 4, 2>(g, links, kappa, states, ptrs, nslots, s);
        stab_update_kernel<float><<<grid, BL_THREADS, 0, s>>>(states, ptrs, N);
    }
    count_launches(5);
    return cudaGetLastError();
}

cudaError_t launch_bicg_direction(int prec, SlotState* states, const SlotPtrs* ptrs, int nslots, size_t N,
                                  cudaStream_t s) {
    dim3 grid(blas_blocks(N / 2), nslots);
    const int t = site_threads(N / 2, nslots, BL_THREADS);
    if (prec == 0) direction_kernel<double><<<t == 32 ? dim3(blas_blocks(N / 2 * (BL_THREADS / 32)), nslots) : grid, t, 0, s>>>(states, ptrs, N);
    else direction_kernel<float><<<grid, BL_THREADS, 0, s>>>(states, ptrs, N);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_bicg_finish(const Geom& g, const void* links64, double kappa, int prec, SlotState* states,
                               const SlotPtrs* ptrs, int nslots, size_t N, cudaStream_t s, int ru_variant, int eo) {
    dim3 g2(blas_blocks(N / 2), nslots);
    if (prec == 0) fold_kernel<double><<<g2, BL_THREADS, 0, s>>>(states, ptrs, N);
    else fold_kernel<float><<<g2, BL_THREADS, 0, s>>>(states, ptrs, N);
    count_launches(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (eo) return launch_eo_true_resid(g, links64, kappa, states, ptrs, nslots, s);
    return launch_true_resid(ru_variant, g, links64, kappa, states, ptrs, nslots, s);
}

template <typename S, int RMAX>
static void window_gemm_launch(SlotState* states, const SlotPtrs* ptrs, int nslots, size_t N, cudaStream_t s) {
    constexpr int threads = WG_T * ((RMAX + WG_K - 1) / WG_K);
    int nb = div_up(N, (size_t)WG_E * WG_T);
    if (nb > 2 * 152) nb = 2 * 152;
    if (nb > PARTIAL_STRIDE / RMAX) nb = PARTIAL_STRIDE / RMAX;
    window_gemm_kernel<S, RMAX><<<dim3(nb, 2 * nslots), threads, 0, s>>>(states, ptrs, N);
}

template <typename S>
static cudaError_t window_gemm_dispatch(int rmax_needed, SlotState* states, const SlotPtrs* ptrs, int nslots,
                                        size_t N, cudaStream_t s) {
    if (rmax_needed <= 8) window_gemm_launch<S, 8>(states, ptrs, nslots, N, s);
    else if (rmax_needed <= 16) window_gemm_launch<S, 16>(states, ptrs, nslots, N, s);
    else if (rmax_needed <= 24) window_gemm_launch<S, 24>(states, ptrs, nslots, N, s);
    else if (rmax_needed <= 32) window_gemm_launch<S, 32>(states, ptrs, nslots, N, s);
    else return cudaErrorInvalidValue;
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_window_gemm(int prec, int two_nev, SlotState* states, const SlotPtrs* ptrs, int nslots, size_t N,
                               cudaStream_t s) {
    if (prec == 0) return window_gemm_dispatch<double>(two_nev, states, ptrs, nslots, N, s);
    return window_gemm_dispatch<float>(two_nev, states, ptrs, nslots, N, s);
}

}  // namespace lqcd
