// FP64 helpers with short dependent chains, and the barrier of cooperative launches (k_dense.cu,
// k_eigen.cu).
#pragma once

#include "wt_internal.cuh"

namespace wt {

// 1 / sqrt(x) from the FP32 value by one third-order step, y <- y + y e (1/2 + 3/8 e) with e = 1 - x y^2 (the
// binomial series: e of 2^-21 leaves 2^-64), x normalised by its exponent: within 1.23 x 2^-53 over all
// exponents; zero, subnormal, negative, infinite x and NaN by CUDA's own root and division.  A chain of
// five FP64 operations, each of which costs a warp 64 cycles of GB300's FP64 units; Newton's two steps
// take eight.
__device__ __forceinline__ double rsqrt_newton(double x) {
    const int hi = __double2hiint(x), ex = hi >> 20;            // negative for a negative x
    if (ex <= 0 || ex == 0x7ff) return 1.0 / sqrt(x);
    const int e = (ex - 1023) & ~1;                            // x = m 2^e, 1 <= m < 4
    const double m = __hiloint2double(hi - (e << 20), __double2loint(x));
    double y = (double)rsqrtf((float)m);
    const double c = fma(-m * y, y, 1.0);
    y = fma(y * c, fma(0.375, c, 0.5), y);
    return __hiloint2double(__double2hiint(y) - ((e / 2) << 20), __double2loint(y));
}
// 1 / x likewise, y <- y + y (e + e^2) with e = 1 - x y: within 1.0 x 2^-53.
__device__ __forceinline__ double rcp_newton(double x) {
    const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
    if (ex <= 2 || ex >= 0x7fd) return 1.0 / x;
    const int e = ex - 1023;
    const double m = __hiloint2double(hi - (e << 20), __double2loint(x));
    double y = (double)__frcp_rn((float)m);
    const double c = fma(-m, y, 1.0);
    y = fma(y, fma(c, c, c), y);
    return __hiloint2double(__double2hiint(y) - (e << 20), __double2loint(y));
}

// Sums of a, b and c over the warp: lanes 0, 8 and 16 return those of a, b and c (the two first steps halve
// the values a lane carries: six FP64 additions a lane instead of fifteen).
__device__ __forceinline__ double warp_sum3(double a, double b, double c) {
    const int lane = threadIdx.x & 31;
    // lanes below 16 go on with a and b, the others with c
    const bool up = lane & 16;
    const double s0 = up ? a : c, s1 = up ? b : 0.0;
    double x = (up ? c : a) + __shfl_xor_sync(0xffffffffu, s0, 16);
    double y = (up ? 0.0 : b) + __shfl_xor_sync(0xffffffffu, s1, 16);
    // lanes with bit 3 go on with b
    const bool hi = lane & 8;
    double v = (hi ? y : x) + __shfl_xor_sync(0xffffffffu, hi ? x : y, 8);
#pragma unroll
    for (int o = 4; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Barrier of the co-resident blocks of a cooperative launch: `round` counts them from 1.  bar:
// kBarrierWords words, zeroed before the launch (a counter that every block adds to, and a word that says
// that a block has given up, after two seconds: error word set, and everybody leaves).  A flag per block,
// every block polling all of them, measured slower (152 blocks: 3 us more).
constexpr unsigned long long kGridWaitNs = 2000000000ull;
constexpr int kBarrierWords = 2;
__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned round, int* err) {
    __syncthreads();
    __shared__ int ok_sh;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        const unsigned want = round * gridDim.x;
        auto count = [&] {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            return v;
        };
        volatile unsigned* gone = bar + 1;
        int ok = 1;
        if (count() < want) {
            unsigned long long t0, t;
            asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
            while (count() < want) {
                asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
                if (t - t0 > 20000 && *gone) { ok = 0; break; }
                if (t - t0 > kGridWaitNs) {
                    *gone = 1;
                    atomicMax(err, (int)DERR_TIMEOUT);
                    ok = 0;
                    break;
                }
            }
        }
        ok_sh = ok;
    }
    __syncthreads();
    return ok_sh != 0;
}

// Blocks of `kernel` that can be resident at once on the current device.
template <class K>
int coresident_blocks(K* kernel, int threads, size_t smem) {
    int dev = 0, n_sm = 0, per = 0;
    WT_CUDA(cudaGetDevice(&dev));
    WT_CUDA(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev));
    WT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem));
    return n_sm * per;
}

}  // namespace wt
