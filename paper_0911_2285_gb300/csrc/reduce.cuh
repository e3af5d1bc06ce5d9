// Per-slot two-level reductions shared by the lattice kernels.
#pragma once
#include "fp64.cuh"
#include "kernels.cuh"

namespace lqcd {

constexpr int RED_MAX_THREADS = 256;   // blocks that reduce have at most this many threads

__device__ __forceinline__ double2* part(const SlotPtrs& P, int kind) { return P.partials + (size_t)kind * PARTIAL_STRIDE; }

// NR numbers per lane summed over the warp: each of the first steps halves the numbers
// that a lane holds, the lane's bit says which half it keeps; lane l returns the sum
// number l / (32 / NR). NR = 4: 6 additions where the sums one by one take 20, in FP64 each
// of them 64 clocks of its pipe.
template <int NR, typename T> __device__ __forceinline__ T lane_sums(const T (&r)[NR]) {
    static_assert(NR == 2 || NR == 4, "numbers per lane");
    const int lane = threadIdx.x & 31;
    const bool u16 = lane & 16, u8 = lane & 8;
    T t;
    if constexpr (NR == 4) {
        const T a = (u16 ? r[2] : r[0]) + __shfl_xor_sync(0xffffffffu, u16 ? r[0] : r[2], 16);
        const T b = (u16 ? r[3] : r[1]) + __shfl_xor_sync(0xffffffffu, u16 ? r[1] : r[3], 16);
        t = (u8 ? b : a) + __shfl_xor_sync(0xffffffffu, u8 ? a : b, 8);
    } else {
        t = (u16 ? r[1] : r[0]) + __shfl_xor_sync(0xffffffffu, u16 ? r[0] : r[1], 16);
        t += __shfl_xor_sync(0xffffffffu, t, 8);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}
__device__ __forceinline__ double wid(float a) { return widen(a); }
__device__ __forceinline__ double wid(double a) { return a; }
// Sums of NV complex values over the block, valid in thread 0: over a warp in the precision
// of v, across the warps in FP64. FP32 across the warps as well would leave the rounding of
// one number per block, and red_blocks has few blocks: rms error of a squared norm on the
// half lattice of 16^3 x 32 (random fields, the order of the sums restated in numpy) 2.5e-9,
// 1.1e-9 with the 1216 blocks of blas_blocks, this way 0.7e-9. smem: 2 NV doubles per warp.
template <int NV, typename C>
__device__ __forceinline__ void block_sum_wide(const C (&v)[NV], double2 (&out)[NV], double* smem) {
    using T = decltype(v[0].x + v[0].x);
    constexpr int NR = 2 * NV;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T r[NR];
#pragma unroll
    for (int i = 0; i < NV; ++i) { r[2 * i] = v[i].x; r[2 * i + 1] = v[i].y; }
    const double t = wid(lane_sums<NR, T>(r));
    __syncthreads();
    if (lane % (32 / NR) == 0) smem[w * NR + lane / (32 / NR)] = t;
    __syncthreads();
    if (w == 0) {
        double s = lane < nw * NR ? smem[lane] : 0.0;   // number l % NR of warp l / NR: at most 8 warps of 4
#pragma unroll
        for (int o = 16; o >= NR; o >>= 1)
            if (o < nw * NR) s += __shfl_xor_sync(0xffffffffu, s, o);
#pragma unroll
        for (int i = 0; i < NV; ++i)
            out[i] = make_double2(__shfl_sync(0xffffffffu, s, 2 * i), __shfl_sync(0xffffffffu, s, 2 * i + 1));
    }
}

// Sum NV complex values per block into part[kind][block*NV + i]; in the last
// block returns true with tot[] = sum over blocks (thread 0 only). The sum over a
// warp runs in the precision of v (FP32 for the mixed solver), the sums across
// warps and blocks in FP64.
template <int NV, typename C>
__device__ bool reduce_slot(const SlotPtrs& P, int kind, C (&v)[NV], double2 (&tot)[NV], unsigned nblocks,
                            unsigned bid) {
    __shared__ double2 smd[(RED_MAX_THREADS / 32) * NV];   // blockDim.x <= RED_MAX_THREADS
    double2 bs[NV];
    block_sum_wide<NV>(v, bs, reinterpret_cast<double*>(smd));
    double2* pp = part(P, kind);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) pp[(size_t)bid * NV + i] = bs[i];
    }
    bool last = last_block(P.counters + kind, nblocks);
    if (last) {
        // The last block adds the partials in a fixed order (deterministic): thread t
        // takes the real number t % (2 NV) of every block whose index is
        // t / (2 NV) modulo the threads per number, then a fixed tree. One FP64 sum
        // per thread and step: an FP64 addition takes 64 cycles here, and the tail of
        // each reduction is a chain of them.
        constexpr int NR = 2 * NV;
        static_assert(NR == 2 || NR == 4, "numbers per block");
        const int q = threadIdx.x % NR, per = blockDim.x / NR;
        const double* pd = reinterpret_cast<const double*>(pp);
        double a0 = 0.0, a1 = 0.0;
        unsigned b = threadIdx.x / NR;
        for (; b + per < nblocks; b += 2 * per) {
            a0 += __ldcg(pd + (size_t)b * NR + q);
            a1 += __ldcg(pd + (size_t)(b + per) * NR + q);
        }
        if (b < nblocks) a0 += __ldcg(pd + (size_t)b * NR + q);
        a0 += a1;
#pragma unroll
        for (int o = 16; o >= NR; o >>= 1) a0 += __shfl_xor_sync(0xffffffffu, a0, o);
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
        double* sd = reinterpret_cast<double*>(smd);
        if (lane < NR) sd[w * NR + lane] = a0;
        __syncthreads();
        if (w == 0) {
            // lane l: number l % NR of warp l / NR (at most 8 warps x 4 numbers)
            double t = lane < nw * NR ? sd[lane] : 0.0;
#pragma unroll
            for (int o = 16; o >= NR; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
#pragma unroll
            for (int i = 0; i < NV; ++i)
                tot[i] = make_double2(__shfl_sync(0xffffffffu, t, 2 * i), __shfl_sync(0xffffffffu, t, 2 * i + 1));
        }
    }
    return last;
}

// Per-thread sums accumulate in the storage precision (FP32 for the mixed solver:
// FP64 arithmetic runs at a small fraction of the FP32 rate on this GPU and would
// bound these bandwidth kernels).
template <typename S> struct Acc {
    cplx<S> z;      // complex sum
    S a, b;         // two real sums
    __device__ __forceinline__ Acc() : z(mk<S>(S(0), S(0))), a(S(0)), b(S(0)) {}
    __device__ __forceinline__ void to(cplx<S> (&v)[2]) const { v[0] = z; v[1] = mk<S>(a, b); }
};
template <typename C> __device__ __forceinline__ auto abs2(C a) -> decltype(a.x) { return a.x * a.x + a.y * a.y; }

constexpr double BREAK_TOL = 1e-14;

// End of an operator launch for one slot (one thread): sigma = (phat, A p), the scales
// of its breakdown test (p2 = |phat|^2, ap2 = |A p|^2) and alpha = rho / sigma.
static __device__ __noinline__ void finish_sigma(SlotState& st, double2 sigma, double p2, double ap2, int products) {
    st.sigma = sigma;
    st.phat_norm = sqrt_fp64(p2);
    st.ap_norm = sqrt_fp64(ap2);
    st.matvecs += products;
    if (!abs_at_least(sigma, BREAK_TOL, st.phat_norm, st.ap_norm) || (sigma.x == 0.0 && sigma.y == 0.0))
        st.status = ST_BREAKDOWN;
    else
        st.alpha = cdiv_fp64(st.rho, sigma);
}

}  // namespace lqcd
