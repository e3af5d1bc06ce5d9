// Inner-product matrices of FP32 fields,
//   C[i][j] = sum_e conj(X_i(e)) Y_j(e),   i < a, j < b,
// N complex numbers per field: the Galerkin projections of the deflation and of the
// eigenspace growth (Alg. Incremental eigBiCG: U_l^H r, U_l^H A U_r and the oblique
// orthogonalisation of new Ritz vectors).
//
// What bounds it: X is read once from HBM (80 fields of 24^3 x 64: 6.8 GB, 1.0 ms at
// the measured copy rate) and every element takes 4 a b multiply-adds (80 x 8:
// 2560, 0.70 ms on the FP32 pipe). A tcgen05 form (3xTF32, 128-row A tiles for N = 16
// columns) spent its time on shared memory: each tile written by TMA, read and
// split, written twice and read three times by narrow MMAs, 3.8 ms; here a byte is
// written once by TMA and read once per 4 x 8 block of C, and the products are full
// FP32. Measured 80 x 8 at N = 10.6 M: 3.8 -> 1.35 ms; 40 x 8 at N = 1.6 M: 0.61 -> 0.12.
// The copies alone take 0.99 ms, the multiply-adds and loads alone 1.3: what is left is
// the FP32 pipe at about half its rate (register-bank conflicts of three-operand
// multiply-adds; packed f32x2 ones need the operands duplicated by moves: 1.50 ms).
//
// Layout: a warp keeps a 4 x 8 block of complex sums in 64 registers per lane; a
// lane takes one of every 32 elements of a chunk (one 8-byte load per field row: 12
// loads, 24 cycles of shared memory, per 128 multiply-adds, 32 cycles of the SM's
// FP32 pipe; with two elements per load the operands do not fit the registers). A block's warps are GI such blocks over the same staged
// 64-element chunk (up to 80 X fields against 8 Y fields), times EG chunks where that leaves
// warps over: 20 warps, five on each quarter of the SM. (8 x 8 blocks on ten warps:
// three of them on two of the quarters, 168 registers and spills, 1.9 ms.) One TMA
// tensor copy per operand and chunk into a ring of stages; rows past a or b and
// elements past N arrive as zeros. More than 8 Y fields: one launch per 8.
//
// Precision: FP32 multiply-adds over 32 elements per lane (a longer FP32 run loses
// accuracy with its square root), then a pairwise FP32 sum over the lanes of the
// warp, then FP64.
#include <cuda.h>

#include "async.cuh"
#include "fp64.cuh"
#include "kernels.cuh"

namespace lqcd {
namespace {

constexpr int DT_E = 64;              // elements per chunk
constexpr int DT_I = 4, DT_J = 8;     // block of C per warp
constexpr int DT_ACC = 2 * DT_I * DT_J;
constexpr int DT_WARPS = 20;          // warps per block at most
constexpr int DT_FLUSH = 16;          // chunks (32 elements per lane) summed in FP32
constexpr int DT_STAGES = 6;
constexpr int DT_EG = 8;              // chunks per stage at most
constexpr size_t DT_RING = 200 * 1024;
constexpr int DT_ROW = 2 * DT_E;      // floats per staged row

struct DotsPlan {
    int GI, EG, ny, stages, nx;   // ny: groups of DT_I GI X rows; nx: blocks along the elements
    size_t stage_floats() const { return (size_t)EG * (DT_I * GI + DT_J) * DT_ROW; }
    size_t smem() const { return stages * stage_floats() * sizeof(float) + 128; }
};
DotsPlan plan_dots(int a, size_t N, int nsm) {
    DotsPlan p;
    const int ni = (a + DT_I - 1) / DT_I;
    p.ny = (ni + DT_WARPS - 1) / DT_WARPS;
    p.GI = (ni + p.ny - 1) / p.ny;
    p.EG = DT_WARPS / p.GI;
    if (p.EG > DT_EG) p.EG = DT_EG;
    const size_t chunks = (N + DT_E - 1) / DT_E;
    if ((size_t)p.EG > chunks) p.EG = (int)chunks;
    p.nx = nsm / p.ny > 1 ? nsm / p.ny : 1;
    const size_t most = (chunks + p.EG - 1) / p.EG;
    if ((size_t)p.nx > most) p.nx = (int)most;
    p.stages = (int)(DT_RING / (p.stage_floats() * sizeof(float)));
    if (p.stages > DT_STAGES) p.stages = DT_STAGES;
    return p;
}

__device__ __forceinline__ void arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// One halving step of the sums over the lanes of a warp: HALF values stay per lane.
template <int HALF, int BIT> __device__ __forceinline__ void halve(float (&v)[DT_ACC], int lane) {
    const bool up = lane & BIT;
#pragma unroll
    for (int k = 0; k < HALF; ++k) {
        const float keep = up ? v[HALF + k] : v[k], send = up ? v[k] : v[HALF + k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, BIT);
    }
}

// Grid (nx, ny). part: [nx * EG][a][b] FP64 partial sums.
__global__ void __launch_bounds__(32 * DT_WARPS, 1)
    dots_kernel(const __grid_constant__ CUtensorMap mx, const __grid_constant__ CUtensorMap my, DotsPlan pl, int a, int b,
                long long chunks, double2* part, int* err) {
    extern __shared__ unsigned char smem_raw[];
    float* ring = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    __shared__ uint64_t full[DT_STAGES], empty[DT_STAGES];
    __shared__ int abort_s, nit_s;
    __shared__ unsigned issued[DT_STAGES];   // copies started per stage
    __shared__ double2 sums[32 * DT_WARPS];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int S = pl.stages;
    const int rows = DT_I * pl.GI + DT_J;                  // staged rows per chunk
    // All blocks walk the fields side by side, EG chunks each per step: the live part of
    // every field stays within a page or two.
    const long long c0 = (long long)blockIdx.x * pl.EG, cstep = (long long)gridDim.x * pl.EG;
    const int nit = chunks > c0 ? (int)((chunks - c0 + cstep - 1) / cstep) : 0;
    if (tid == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], blockDim.x >> 5); issued[s] = 0; }
        abort_s = 0;
        mbar_init_fence();
    }
    __syncthreads();
    const int row0 = blockIdx.y * DT_I * pl.GI;
    // The copies of an iteration, by one thread.
    auto issue = [&](int it, int s) {
        ++issued[s];
        const int c = (int)c0 + it * (int)cstep;
        const int nv = (int)chunks - c < pl.EG ? (int)chunks - c : pl.EG;
        mbar_arrive_expect_tx(&full[s], (unsigned)(nv * rows) * DT_ROW * 4u);
        for (int e = 0; e < nv; ++e) {
            float* dst = ring + (s * pl.EG + e) * rows * DT_ROW;
            tma_load_2d(dst, &mx, (c + e) * DT_ROW, row0, &full[s]);
            tma_load_2d(dst + DT_I * pl.GI * DT_ROW, &my, (c + e) * DT_ROW, 0, &full[s]);
        }
    };
    if (tid == 0)
        for (int it = 0; it < S && it < nit; ++it) issue(it, it);
    const int eg = warp / pl.GI, ig = warp % pl.GI;

    float acc[DT_ACC];
    double2* sum = &sums[tid];   // in shared memory: 96 registers per thread, 88 of them sums and operands
    *sum = make_double2(0.0, 0.0);
#pragma unroll
    for (int k = 0; k < DT_ACC; ++k) acc[k] = 0.f;
    // Sums over the lanes: each step halves the values a lane holds, the lane's bit
    // selects which half it keeps; after five steps lane l holds complex sum l of the
    // block, added in FP64.
    auto flush = [&] {
        halve<32, 16>(acc, lane);
        halve<16, 8>(acc, lane);
        halve<8, 4>(acc, lane);
        halve<4, 2>(acc, lane);
        halve<2, 1>(acc, lane);
        *sum = *sum + make_double2(widen(acc[0]), widen(acc[1]));
#pragma unroll
        for (int k = 0; k < DT_ACC; ++k) acc[k] = 0.f;
    };
    const int nw = blockDim.x >> 5;
    int s = 0, turn = warp;
    unsigned ph = 0;
    const float2* xs = reinterpret_cast<const float2*>(ring) + (eg * rows + DT_I * ig) * DT_E + lane;
    const int yoff = DT_I * (pl.GI - ig) * DT_E, step = pl.EG * rows * DT_E;   // in float2
    const int miss = nit > 0 && c0 + (nit - 1) * cstep + eg >= chunks;   // no chunk for this warp in the last iteration
    if (tid == 0) nit_s = nit;   // read by the turns only
    __syncthreads();
    for (int rem = nit; rem > 0; --rem) {   // counted down: one register less
        // The stage of the iteration before last is refilled; the warps take turns, so that
        // no warp falls behind by the copies' instructions (always warp 0: 1.86 ms).
        if (--turn < 0) {
            turn += nw;
            const int n = *(volatile int*)&nit_s, it = n - rem;
            if (lane == 0 && it > 1 && it - 2 + S < n) {
                const int r = s < 2 ? s + S - 2 : s - 2;
                if (mbar_wait(&empty[r], s < 2 ? ph ^ 1u : ph)) issue(it - 2 + S, r);
                else *(volatile int*)&abort_s = 1;
            }
            __syncwarp();
        }
        // A wait that gave up ends the block: the other warps' waits on that stage or on
        // this warp's arrivals run out as well.
        if (!__all_sync(0xffffffffu, mbar_wait(&full[s], ph))) {
            if (lane == 0) *(volatile int*)&abort_s = 1;
            break;
        }
        if (rem > miss) {
#pragma unroll 1
            for (int h = 0; h < DT_E; h += 32) {
                float2 x[DT_I];
#pragma unroll
                for (int i = 0; i < DT_I; ++i) x[i] = xs[i * DT_E + h];
#pragma unroll
                for (int j = 0; j < DT_J; ++j) {
                    const float2 y = xs[yoff + j * DT_E + h];
#pragma unroll
                    for (int i = 0; i < DT_I; ++i) {
                        float& re = acc[(i * DT_J + j) * 2];
                        float& im = acc[(i * DT_J + j) * 2 + 1];
                        re = fmaf(x[i].x, y.x, re); im = fmaf(x[i].x, y.y, im);
                        re = fmaf(x[i].y, y.y, re); im = fmaf(-x[i].y, y.x, im);
                    }
                }
            }
        }
        __syncwarp();
        if (lane == 0) arrive(&empty[s]);
        if ((rem & (DT_FLUSH - 1)) == 0) flush();
        xs += step;
        if (++s == S) { s = 0; ph ^= 1u; xs -= S * step; }
    }
    flush();
    __syncthreads();
    if (*(volatile int*)&abort_s) {
        if (tid == 0) {
            atomicExch(err, 1);
            for (int s = 0; s < S; ++s)   // copies in flight land before the block exits
                if (issued[s]) mbar_drain(&full[s], (issued[s] - 1) & 1u);
        }
        return;
    }
    const int i = row0 + DT_I * ig + lane / DT_J, j = lane % DT_J;
    if (i < a && j < b) part[(((size_t)blockIdx.x * pl.EG + eg) * a + i) * b + j] = *sum;
}

// C[i][j] (or its conjugate into C[j][i]) = sum over the np partials, one warp each; zero
// after a wait that gave up (some partials are then from an earlier call).
__global__ void __launch_bounds__(128) dots_reduce_kernel(int a, int b, int np, const double2* part, double2* Cm, int ldc,
                                                          int conj_store, const int* err) {
    const int q = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (q >= a * b) return;
    double2 s0 = make_double2(0.0, 0.0), s1 = s0;
    int p = lane;
    for (; p + 32 < np; p += 64) {
        s0 = s0 + part[(size_t)p * a * b + q];
        s1 = s1 + part[(size_t)(p + 32) * a * b + q];
    }
    if (p < np) s0 = s0 + part[(size_t)p * a * b + q];
    s0 = warp_sum(s0 + s1);
    if (*(const volatile int*)err) s0 = make_double2(0.0, 0.0);
    if (lane == 0) {
        const int i = q / b, j = q % b;
        if (conj_store) Cm[(size_t)j * ldc + i] = conj_(s0);
        else Cm[(size_t)i * ldc + j] = s0;
    }
}

cudaError_t device_sms(int* nsm) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    return e == cudaSuccess ? cudaDeviceGetAttribute(nsm, cudaDevAttrMultiProcessorCount, dev) : e;
}

// a or b consecutive fields of N complex FP32 numbers as a 2-D tensor of floats.
bool encode_fields(CUtensorMap* m, const void* base, int fields, size_t N, int box_rows) {
    const uint64_t dims[2] = {(uint64_t)(2 * N), (uint64_t)fields}, strides[1] = {(uint64_t)(8 * N)};
    const uint32_t box[2] = {(uint32_t)DT_ROW, (uint32_t)box_rows};
    return encode_tensor_map_f32(m, base, 2, dims, strides, box);
}

}  // namespace

// TMA: 16-byte aligned rows; 31-bit coordinates.
bool dots_supported(int a, const void* X, const void* Y, size_t N) {
    return a > 0 && N > 0 && N % 2 == 0 && 2 * N + DT_ROW < ((size_t)1 << 31) && ((uintptr_t)X & 15) == 0 &&
           ((uintptr_t)Y & 15) == 0 && tensor_maps_available();
}

size_t dots_scratch(int a, int b, size_t N) {
    int nsm = 0;
    if (device_sms(&nsm) != cudaSuccess) return 0;
    const DotsPlan p = plan_dots(a, N, nsm);
    return (size_t)p.nx * p.EG * a * (b < DT_J ? b : DT_J);
}

cudaError_t launch_dots(int a, const void* X, int b, const void* Y, size_t N, double2* Cm, int ldc, int conj_store,
                        double2* scratch, size_t scratch_elems, int* err, cudaStream_t st) {
    if (a <= 0 || b <= 0) return cudaSuccess;
    if (!dots_supported(a, X, Y, N)) return cudaErrorInvalidValue;
    int nsm = 0;
    cudaError_t e = device_sms(&nsm);
    // the device's limit, set per call: a few hundred nanoseconds, and right on every device
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(dots_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(DT_RING + 128));
    if (e != cudaSuccess) return e;
    const DotsPlan p = plan_dots(a, N, nsm);
    for (int j0 = 0; j0 < b; j0 += DT_J) {
        const int bb = b - j0 < DT_J ? b - j0 : DT_J;
        if ((size_t)p.nx * p.EG * a * bb > scratch_elems) return cudaErrorInvalidValue;
        CUtensorMap mx, my;
        const char* Yj = reinterpret_cast<const char*>(Y) + (size_t)j0 * N * 8;
        if (!encode_fields(&mx, X, a, N, DT_I * p.GI) || !encode_fields(&my, Yj, bb, N, DT_J)) return cudaErrorInvalidValue;
        dots_kernel<<<dim3(p.nx, p.ny), 32 * p.GI * p.EG, p.smem(), st>>>(
            mx, my, p, a, bb, (long long)((N + DT_E - 1) / DT_E), scratch, err);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        double2* Cj = conj_store ? Cm + (size_t)j0 * ldc : Cm + j0;
        dots_reduce_kernel<<<(a * bb + 3) / 4, 128, 0, st>>>(a, bb, p.nx * p.EG, scratch, Cj, ldc, conj_store, err);
        count_launches(2);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t set_wait_cycles_dots(long long cycles) { return set_wait_cycles_here(cycles); }

}  // namespace lqcd
