// Eq. 1 (Ramo-Shockley-Riegler convolution) against carrier tracks, direct
// form on the stored FP32 field H[t][c][x][y][z]:
//   Q(tau_m) = sum_{m' <= m, m' < n_steps} W(x_m', (m - m' + 1/2) dt) . v_m' dt
//   i(tau_m) = -(q / V_w) (Q(tau_m) - Q(tau_{m-1})) / dt
// W between grid points: trilinear (periodic x, y; z clamped to the first and
// last grid planes); between time samples: linear in t, W(0) = 0, held after
// the last sample.  One block per track: the dot products W(x_m', t_n) . v_m'
// at the time samples are staged in shared memory for a chunk of steps, then
// every output time accumulates its lags: the FP64 field in FP64; the FP32
// field as current increments, FP32 within a chunk and FP64 across chunks.
#include "wt_internal.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

namespace wt {

struct Eq1Lag {
    int n;          // lower time sample
    float w0, w1;   // weights of samples n and n+1
};
// FP64 weights, for the FP64 field of the loss
struct Eq1Lag64 {
    int n;
    double w0, w1;
};

constexpr int EQ1_MC = 16;   // track steps per chunk

// Current increments of one chunk of track steps (FP32 field): for output m,
//   D(m) = Q(tau_m) - Q(tau_{m-1}) = sum_j [g_j(m - m'_j) - g_j(m - m'_j - 1)] dt,
// g_j(L) = W(x_j, (L + 1/2) dt) . v_j (linear in time between the staged samples f[j][n],
// g_j(-1) = 0), summed in FP32 over the chunk's steps (at most EQ1_MC terms, each a difference of
// neighbouring lags, so nothing large cancels) and carried across chunks in FP64: one FP64
// addition per output and chunk instead of FP64 products per lag (GB300's FP64 rate is low).
__device__ __forceinline__ float eq1_interp(const float* __restrict__ fj, int nt, Eq1Lag lg) {
    return fmaf(lg.w0, fj[lg.n], lg.w1 * fj[min(lg.n + 1, nt - 1)]);
}
// f: [mc] rows of stride ld, nt the clamp of sample n + 1; outputs m < c0 take nothing
// from this chunk, so the threads start at c0.
__device__ __forceinline__ void eq1_increments(const float* __restrict__ f, int ld, int nt, int mc, int c0, int n_out,
                                               const Eq1Lag* __restrict__ lags, double* __restrict__ D) {
    for (int m = c0 + threadIdx.x; m < n_out; m += blockDim.x) {
        const int jmax = min(mc - 1, m - c0);
        if (jmax < 0) continue;
        // step j sees lag L = m - c0 - j; the entry of lag L - 1 is the next step's entry of lag L
        int L = m - c0;
        Eq1Lag hi = lags[L];
        float d = 0.f;
        for (int j = 0; j <= jmax; ++j, --L) {
            const float* fj = f + j * ld;
            const float g_hi = eq1_interp(fj, nt, hi);
            if (L == 0) {
                d += g_hi;
                break;
            }
            const Eq1Lag lo = lags[L - 1];
            d += g_hi - eq1_interp(fj, nt, lo);
            hi = lo;
        }
        D[m] += (double)d;
    }
}

// Cell and weights of one track step, and W(x, t_n) . v from a stored field.
template <class T>
struct Eq1Cell {
    T vx = 0, vy = 0, vz = 0, wx = 0, wy = 0, wz = 0;
    size_t a00 = 0, a01 = 0, a10 = 0, a11 = 0;
    __device__ __forceinline__ void set(T x, T y, T z, int Nx, int Ny, int Nz, T inv_hx, T inv_hy, T inv_hz) {
        const T fx = x * inv_hx, fy = y * inv_hy;
        T fz = z * inv_hz - (T)0.5;
        fz = fz < (T)0 ? (T)0 : (fz > (T)(Nz - 1) ? (T)(Nz - 1) : fz);
        const T flx = floor(fx), fly = floor(fy);
        const int k0 = min((int)floor(fz), Nz - 2);
        wx = fx - flx;
        wy = fy - fly;
        wz = fz - (T)k0;
        const int i0 = ((int)flx % Nx + Nx) % Nx, j0 = ((int)fly % Ny + Ny) % Ny;
        const int i1 = (i0 + 1) % Nx, j1 = (j0 + 1) % Ny;
        a00 = ((size_t)i0 * Ny + j0) * Nz + k0;
        a01 = ((size_t)i0 * Ny + j1) * Nz + k0;
        a10 = ((size_t)i1 * Ny + j0) * Nz + k0;
        a11 = ((size_t)i1 * Ny + j1) * Nz + k0;
    }
    __device__ __forceinline__ bool moving() const { return vx != 0 || vy != 0 || vz != 0; }
    // hb: the three component planes of one time sample
    __device__ __forceinline__ T dot(const T* __restrict__ hb, size_t npts) const {
        const T one = 1;
        T w[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const T* h = hb + (size_t)c * npts;
            const T v00 = (one - wz) * h[a00] + wz * h[a00 + 1];
            const T v01 = (one - wz) * h[a01] + wz * h[a01 + 1];
            const T v10 = (one - wz) * h[a10] + wz * h[a10 + 1];
            const T v11 = (one - wz) * h[a11] + wz * h[a11 + 1];
            w[c] = (one - wx) * ((one - wy) * v00 + wy * v01) + wx * ((one - wy) * v10 + wy * v11);
        }
        return w[0] * vx + w[1] * vy + w[2] * vz;
    }
};

// G[step][n] = W(x_step, t_n) . v_step for all steps of all tracks, eight time samples a thread (one
// 32-byte sector of G).  What bounds it are the sectors drawn from L2: a step of an inclined track lies
// in a cell of its own, 12 sectors a sample (49 GB for 1e6 steps x 128 samples of a 96 x 96 x 192
// field), so the steps of a large call are taken in the order of their cells: a warp's 32 steps then
// share the sectors of a few neighbouring cells.  That field and those steps: 16.0 ms with a block per
// track, 4.55 ms a time plane at a time in the tracks' order, 1.16 ms in the cells' order (the sort
// 0.055 ms).
constexpr int kStageTimes = 8;
struct Eq1Steps {
    const float *x, *y, *z, *vx, *vy, *vz;
    const unsigned* order;               // the step whose row of G a position fills (NULL: its own)
    size_t n;
};
__global__ void __launch_bounds__(256, 4) eq1_stage_kernel(const float* __restrict__ H, int Nx, int Ny, int Nz,
                                                        float inv_hx, float inv_hy, float inv_hz, Eq1Steps st, int nu,
                                                        int ldg, float* __restrict__ G) {
    const size_t s = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= st.n) return;
    const size_t npts = (size_t)Nx * Ny * Nz;
    Eq1Cell<float> c;
    c.vx = st.vx[s];
    c.vy = st.vy[s];
    c.vz = st.vz[s];
    c.set(st.x[s], st.y[s], st.z[s], Nx, Ny, Nz, inv_hx, inv_hy, inv_hz);
    const int n0 = blockIdx.y * kStageTimes;
    float r[kStageTimes] = {};
    if (c.moving()) {
        // no branch between the samples, so that their loads overlap; the ones past nu read the last plane
#pragma unroll
        for (int i = 0; i < kStageTimes; ++i) r[i] = c.dot(H + (size_t)min(n0 + i, nu - 1) * 3 * npts, npts);
#pragma unroll
        for (int i = 0; i < kStageTimes; ++i)
            if (n0 + i >= nu) r[i] = 0.f;
    }
    float4* g = reinterpret_cast<float4*>(G + (st.order ? (size_t)st.order[s] : s) * ldg + n0);
    g[0] = make_float4(r[0], r[1], r[2], r[3]);
    g[1] = make_float4(r[4], r[5], r[6], r[7]);
}

// Order of the steps by their cells (counting sort): a bin is eight cells along z, one 32-byte sector of
// each component plane; resting steps, which read nothing, have the last bin to themselves.  The order
// within a bin is that of the atomics: it moves no value.
__device__ __forceinline__ unsigned eq1_bin(const Eq1Steps& st, size_t s, int Nx, int Ny, int Nz, float inv_hx,
                                            float inv_hy, float inv_hz, unsigned n_bins) {
    Eq1Cell<float> c;
    c.vx = st.vx[s];
    c.vy = st.vy[s];
    c.vz = st.vz[s];
    if (!c.moving()) return n_bins - 1;
    c.set(st.x[s], st.y[s], st.z[s], Nx, Ny, Nz, inv_hx, inv_hy, inv_hz);
    const size_t col = c.a00 / Nz;
    return (unsigned)(col * ((Nz + 7) / 8) + (c.a00 - col * Nz) / 8);
}
__global__ void __launch_bounds__(256) eq1_count_kernel(Eq1Steps st, int Nx, int Ny, int Nz, float inv_hx, float inv_hy,
                                                        float inv_hz, unsigned n_bins, unsigned* __restrict__ count,
                                                        unsigned* __restrict__ rank) {
    const size_t s = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s < st.n) rank[s] = atomicAdd(count + eq1_bin(st, s, Nx, Ny, Nz, inv_hx, inv_hy, inv_hz, n_bins), 1u);
}
// Exclusive sums within stretches of kScan bins (in place), and each stretch's total.
constexpr int kScan = 4096;
__device__ __forceinline__ unsigned block_exclusive(unsigned v, unsigned* warp_tot, unsigned* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[w] = x;
    __syncthreads();
    if (w == 0) {
        unsigned t = warp_tot[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        warp_tot[lane] = t;
    }
    __syncthreads();
    *total = warp_tot[31];
    const unsigned base = w ? warp_tot[w - 1] : 0u;
    __syncthreads();
    return base + x - v;
}
__global__ void __launch_bounds__(1024) eq1_scan_kernel(unsigned* __restrict__ count, unsigned n_bins,
                                                        unsigned* __restrict__ total) {
    __shared__ unsigned wt[32];
    const unsigned b0 = blockIdx.x * kScan + 4 * threadIdx.x;
    unsigned v[4], sum = 0, all;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[i] = b0 + i < n_bins ? count[b0 + i] : 0u;
        sum += v[i];
    }
    unsigned at = block_exclusive(sum, wt, &all);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (b0 + i < n_bins) count[b0 + i] = at;
        at += v[i];
    }
    if (threadIdx.x == 0) total[blockIdx.x] = all;
}
__global__ void __launch_bounds__(1024) eq1_scan_totals_kernel(unsigned* __restrict__ total, int n) {
    __shared__ unsigned wt[32];
    unsigned carry = 0;
    for (int k0 = 0; k0 < n; k0 += 1024) {
        const int k = k0 + threadIdx.x;
        unsigned all;
        const unsigned at = block_exclusive(k < n ? total[k] : 0u, wt, &all);
        if (k < n) total[k] = carry + at;
        carry += all;
    }
}
__global__ void __launch_bounds__(256) eq1_order_kernel(Eq1Steps st, int Nx, int Ny, int Nz, float inv_hx, float inv_hy,
                                                        float inv_hz, unsigned n_bins,
                                                        const unsigned* __restrict__ count,
                                                        const unsigned* __restrict__ total,
                                                        const unsigned* __restrict__ rank, float* __restrict__ sorted,
                                                        unsigned* __restrict__ order) {
    const size_t s = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= st.n) return;
    const unsigned b = eq1_bin(st, s, Nx, Ny, Nz, inv_hx, inv_hy, inv_hz, n_bins);
    const size_t at = (size_t)count[b] + total[b / kScan] + rank[s];
    order[at] = (unsigned)s;
    sorted[at] = st.x[s];
    sorted[st.n + at] = st.y[s];
    sorted[2 * st.n + at] = st.z[s];
    sorted[3 * st.n + at] = st.vx[s];
    sorted[4 * st.n + at] = st.vy[s];
    sorted[5 * st.n + at] = st.vz[s];
}

// Workspace of the staged form: per step a row of G, its sorted copy, its place and its rank; the bins.
static int eq1_ldg(int nu) { return (nu + kStageTimes - 1) / kStageTimes * kStageTimes; }
static size_t eq1_bins(int Nx, int Ny, int Nz) { return (size_t)Nx * Ny * ((Nz + 7) / 8) + 1; }
static size_t eq1_bin_bytes(size_t bins) { return (bins + (bins + kScan - 1) / kScan) * sizeof(unsigned); }
static size_t eq1_step_bytes(int nu) { return (size_t)(eq1_ldg(nu) + 8) * sizeof(float); }
size_t eq1_stage_bytes(size_t steps, int nu, int Nx, int Ny, int Nz) {
    return steps * eq1_step_bytes(nu) + eq1_bin_bytes(eq1_bins(Nx, Ny, Nz));
}
// Whether the staged form pays, kept: its workspace is there already.  From 2^20 values on (2^19 with more than
// 64 samples); below, where a track has so many values that its one block takes long over them: one track
// of 50 steps, 200 samples 132 -> 56 us, 100 of them 296 -> 119 us, 64 samples 73 -> 54 us; with 300 tracks
// the blocks fill the chip and it takes four times the values (31 steps, 128 samples: 188 us without, 211
// with).  Few samples are not worth an allocation of 0.25 ms below 2^24 values: 1 000 tracks x 1 000 steps, 12
// samples 522 us without, 758 with.
bool eq1_staged(int n_tracks, int n_steps, int nu, bool kept) {
    const size_t per = (size_t)n_steps * nu, all = per * n_tracks;
    if (nu > 65535 || (!kept && nu < 32 && all < ((size_t)1 << 24))) return false;
    return all >= (nu > 64 ? (size_t)1 << 19 : (size_t)1 << 20) || per >= (n_tracks <= 200 ? 1000 : 4000);
}
// The sort pays for itself when there is a step for every eighth sector (a sector serves four cells), from
// 2^21 values on (below, its launches take longer than the sectors it saves).  96 x 96 x 192, 128 samples:
// 1e5 steps 982 -> 442 us, 4e4 steps 452 -> 375 us, 2e4 steps 226 -> 267 us (not sorted).  A field of at most 4 096
// bins stays in L1: 16 x 16 x 32, 3e5 steps x 12 samples 263 us, sorted 310.
static bool eq1_sort(size_t steps, int nu, size_t bins) {
    return 8 * steps >= bins && steps * nu >= ((size_t)1 << 21) && bins > 4096 && bins < ((size_t)1 << 31);
}

// T: field type; L: lag table entry; TO: current type.  nu: time samples the lag table reads
// (samples n >= nu are never staged).  G: the dot products of eq1_stage_kernel, or NULL to take them
// here (a call that may not allocate, the FP64 field, few steps): lanes over track steps, warps over
// time samples, a lane keeping its step's cell for all samples, so that neighbouring steps share
// sectors (lanes over time samples: every read a sector of its own).
// 1e4 tracks x 100 steps, 96 x 96 x 192, 128 samples: 38.1 ms with lanes over samples, 16.0 with lanes
// over steps, 1.6 through G.  A stage holds `steps` steps (32, or 16 where 32 rows of samples
// do not fit, or the power of two that holds all of them), accumulated 16 at a time.
template <class T, class L, class TO>
__global__ void __launch_bounds__(256) eq1_kernel(const T* __restrict__ H, int Nx, int Ny, int Nz, int nt, int nu,
                                                  T inv_hx, T inv_hy, T inv_hz,
                                                  const float* __restrict__ X, const float* __restrict__ Y,
                                                  const float* __restrict__ Z, const float* __restrict__ VX,
                                                  const float* __restrict__ VY, const float* __restrict__ VZ,
                                                  const float* __restrict__ qtrack, float qconst, int n_steps,
                                                  int n_out, double dt, double inv_vw, int steps, int ld,
                                                  const float* __restrict__ G, int ldg,
                                                  const L* __restrict__ lags, TO* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* f = reinterpret_cast<T*>(smem_raw);                               // [steps][ld]
    double* Q = reinterpret_cast<double*>(smem_raw + (((size_t)steps * ld * sizeof(T) + 15) & ~(size_t)15));   // [n_out]
    const int tr = blockIdx.x;
    const size_t npts = (size_t)Nx * Ny * Nz;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int per = 32 / steps;                                          // time samples per warp and turn
    for (int m = threadIdx.x; m < n_out; m += blockDim.x) Q[m] = 0.0;
    for (int s0 = 0; s0 < n_steps; s0 += steps) {
        const int j = lane % steps;
        const bool in = s0 + j < n_steps;
        Eq1Cell<T> cell;
        const size_t s = (size_t)tr * n_steps + s0 + j;
        if (in && !G) {
            cell.vx = VX[s];
            cell.vy = VY[s];
            cell.vz = VZ[s];
            cell.set((T)X[s], (T)Y[s], (T)Z[s], Nx, Ny, Nz, inv_hx, inv_hy, inv_hz);
        }
        __syncthreads();
        if (G) {
            const float* g = G + ((size_t)tr * n_steps + s0) * ldg;
            for (int q = warp; q < min(steps, n_steps - s0); q += nwarps)
                for (int n = lane; n < nu; n += 32) f[q * ld + n] = (T)g[(size_t)q * ldg + n];
        } else {
            for (int n = warp * per + lane / steps; n < nu; n += nwarps * per)
                if (in) f[j * ld + n] = cell.moving() ? cell.dot(H + (size_t)n * 3 * npts, npts) : (T)0;
        }
        __syncthreads();
        for (int c0 = s0; c0 < min(n_steps, s0 + steps); c0 += EQ1_MC) {
            const int mc = min(EQ1_MC, n_steps - c0);
            const T* fc = f + (size_t)(c0 - s0) * ld;
            if constexpr (std::is_same<T, float>::value) {
                // FP32 field: increments D(m) = Q(tau_m) - Q(tau_{m-1}) over dt, accumulated in Q; a
                // thread keeps its outputs across the chunks, shifted by EQ1_MC, so order them
                eq1_increments(fc, ld, nt, mc, c0, n_out, lags, Q);
                __syncthreads();
            } else {
                for (int m = threadIdx.x; m < n_out; m += blockDim.x) {
                    double q = 0.0;
                    const int jmax = min(mc - 1, m - c0);
                    for (int j = 0; j <= jmax; ++j) {
                        const L lg = lags[m - (c0 + j)];
                        q += (double)lg.w0 * (double)fc[j * ld + lg.n] +
                             (double)lg.w1 * (double)fc[j * ld + min(lg.n + 1, nt - 1)];
                    }
                    Q[m] += q * dt;
                }
            }
        }
    }
    __syncthreads();
    const float qc = qtrack ? qtrack[tr] : qconst;
    for (int m = threadIdx.x; m < n_out; m += blockDim.x) {
        // FP32 field: Q holds the increments already (the dt of Q and of the derivative cancel)
        const double dq = std::is_same<T, float>::value ? Q[m] * dt : Q[m] - (m ? Q[m - 1] : 0.0);
        out[(size_t)tr * n_out + m] = (TO)(-(double)qc * inv_vw * dq / dt);
    }
}

template <class T, class L, class TO>
static void eq1_launch_t(cudaStream_t s, const T* H, int Nx, int Ny, int Nz, int nt, double Lx, double Ly, double Lz,
                         const float* x, const float* y, const float* z, const float* vx, const float* vy,
                         const float* vz, const float* q, float qconst, int n_tracks, int n_steps, int n_out,
                         double dt, double v_w, const void* lags, int nu, TO* out, const float* G = nullptr) {
    if (nu < 1 || nu > nt) fail(WT_ERR_ARG, "eq1: bad count of time samples in use");
    // the limit of accepted sizes: 16 rows of nt samples and the outputs in 200 KB
    if ((((size_t)EQ1_MC * nt * sizeof(T) + 15) & ~(size_t)15) + (size_t)n_out * sizeof(double) > 200 * 1024)
        fail(WT_ERR_UNSUPPORTED, "eq1: n_t or n_out too large for shared memory");
    // rows of the staged samples: an odd stride (lanes store down a column); nu + 1 entries may be read
    const int ld = (std::min(nt, nu + 1)) | 1;
    auto bytes = [&](int steps) {
        return (((size_t)steps * ld * sizeof(T) + 15) & ~(size_t)15) + (size_t)n_out * sizeof(double);
    };
    // 32 steps per stage while four blocks fit an SM (or 16 would not give more); a power of two that holds
    // the steps where they are fewer, so that all lanes have a time sample to take (one step, 200 samples: 55 us
    // with 32, 41 with one; 100 tracks x 4 steps: 139 and 61)
    int steps = bytes(32) <= 56 * 1024 ? 32 : 16;
    while (steps / 2 >= n_steps) steps /= 2;
    const size_t sh = bytes(steps);
    allow_dyn_smem(eq1_kernel<T, L, TO>, sh);
    eq1_kernel<T, L, TO><<<n_tracks, 256, sh, s>>>(H, Nx, Ny, Nz, nt, nu, (T)(Nx / Lx), (T)(Ny / Ly), (T)(Nz / Lz), x, y,
                                                   z, vx, vy, vz, q, qconst, n_steps, n_out, dt, 1.0 / v_w, steps, ld,
                                                   G, eq1_ldg(nu), static_cast<const L*>(lags),
                                                   out);
    WT_LAUNCH("eq1");
}
void eq1_launch(cudaStream_t s, const float* H, int Nx, int Ny, int Nz, int nt, double Lx, double Ly, double Lz,
                const float* x, const float* y, const float* z, const float* vx, const float* vy, const float* vz,
                const float* q, float qconst, int n_tracks, int n_steps, int n_out, double dt, double v_w,
                const void* lags, int nu, float* out, unsigned char* ws, size_t ws_bytes) {
    // ws: workspace (NULL: none) for the dot products of as many whole tracks at a time
    const size_t bins = eq1_bins(Nx, Ny, Nz), fixed = eq1_bin_bytes(bins);
    const int per = !ws || ws_bytes <= fixed ? 0 :
        (int)std::min<size_t>(n_tracks, (ws_bytes - fixed) / (eq1_step_bytes(nu) * n_steps));
    if (per < 1) {
        eq1_launch_t<float, Eq1Lag, float>(s, H, Nx, Ny, Nz, nt, Lx, Ly, Lz, x, y, z, vx, vy, vz, q, qconst, n_tracks,
                                           n_steps, n_out, dt, v_w, lags, nu, out);
        return;
    }
    const float ix = (float)(Nx / Lx), iy = (float)(Ny / Ly), iz = (float)(Nz / Lz);
    const int ldg = eq1_ldg(nu);
    for (int t0 = 0; t0 < n_tracks; t0 += per) {
        const int n = std::min(per, n_tracks - t0);
        const size_t o = (size_t)t0 * n_steps, steps = (size_t)n * n_steps;
        const unsigned blocks = (unsigned)((steps + 255) / 256);
        float* G = reinterpret_cast<float*>(ws);
        Eq1Steps st{x + o, y + o, z + o, vx + o, vy + o, vz + o, nullptr, steps};
        if (eq1_sort(steps, nu, bins)) {
            float* sorted = G + steps * ldg;
            unsigned* order = reinterpret_cast<unsigned*>(sorted + 6 * steps);
            unsigned *rank = order + steps, *count = rank + steps, *total = count + bins;
            const int stretches = (int)((bins + kScan - 1) / kScan);
            WT_CUDA(cudaMemsetAsync(count, 0, bins * sizeof(unsigned), s));
            eq1_count_kernel<<<blocks, 256, 0, s>>>(st, Nx, Ny, Nz, ix, iy, iz, (unsigned)bins, count, rank);
            eq1_scan_kernel<<<stretches, 1024, 0, s>>>(count, (unsigned)bins, total);
            eq1_scan_totals_kernel<<<1, 1024, 0, s>>>(total, stretches);
            eq1_order_kernel<<<blocks, 256, 0, s>>>(st, Nx, Ny, Nz, ix, iy, iz, (unsigned)bins, count, total, rank,
                                                    sorted, order);
            WT_LAUNCH("eq1_order");
            st = Eq1Steps{sorted, sorted + steps, sorted + 2 * steps, sorted + 3 * steps, sorted + 4 * steps,
                          sorted + 5 * steps, order, steps};
        }
        eq1_stage_kernel<<<dim3(blocks, ldg / kStageTimes), 256, 0, s>>>(H, Nx, Ny, Nz, ix, iy, iz, st, nu, ldg, G);
        WT_LAUNCH("eq1_stage");
        eq1_launch_t<float, Eq1Lag, float>(s, H, Nx, Ny, Nz, nt, Lx, Ly, Lz, x + o, y + o, z + o, vx + o, vy + o, vz + o,
                                           q ? q + t0 : nullptr, qconst, n, n_steps, n_out, dt, v_w, lags, nu,
                                           out + (size_t)t0 * n_out, G);
    }
}
// FP64 field (plain path): interpolation, time weights and currents in FP64 (lags: FP64 table).
void eq1_launch64(cudaStream_t s, const double* H, int Nx, int Ny, int Nz, int nt, double Lx, double Ly, double Lz,
                  const float* x, const float* y, const float* z, const float* vx, const float* vy, const float* vz,
                  const float* q, float qconst, int n_tracks, int n_steps, int n_out, double dt, double v_w,
                  const void* lags, int nu, double* out) {
    eq1_launch_t<double, Eq1Lag64, double>(s, H, Nx, Ny, Nz, nt, Lx, Ly, Lz, x, y, z, vx, vy, vz, q, qconst,
                                           n_tracks, n_steps, n_out, dt, v_w, lags, nu, out);
}
// Eq. 1 straight from the rank-r form of the FP32 field, H[t][c][p] = sum_m W[t][m] E[c][m][p]
// (the representation the tensor-core expansion writes out): the staged dot products are
// W(x_j, t_n) . v_j = sum_m W[t_n][m] (E_m(x_j) . v_j), the interpolation being linear, so per
// track step the r basis fields are interpolated once instead of the field at every time
// sample (r x 24 gathers from E instead of n_t x 24 from H).  Lags, accumulation and currents
// as in eq1_kernel.  The basis fields are read point-major, Ep[p][c][32] (eq1_point_major): one
// warp per track step, a lane per basis field, so that each of the 24 corner-component reads is
// one 128-byte line, and the two z neighbours of a corner are adjacent lines.
// f[j][n] = sum_m W[t_n][m] sv[m][j] for n < nu, j < mc: NB time samples (nq apart, so that a warp
// reads consecutive words of Wt) by four steps per thread; Wt rows hold NB nq >= nu samples, the
// ones past nu zero.
template <int NB>
__device__ __forceinline__ void eq1_stage_product(const float* __restrict__ sv, const float* __restrict__ Wt, int r,
                                                  int nq, int nu, int mc, float* __restrict__ f) {
    const int ng = (mc + 3) >> 2, ldw = NB * nq;
    for (int e = threadIdx.x; e < nq * ng; e += blockDim.x) {
        const int n0 = e % nq, j0 = 4 * (e / nq);
        float acc[NB][4] = {};
        for (int m = 0; m < r; ++m) {
            const float4 s4 = *reinterpret_cast<const float4*>(sv + m * EQ1_MC + j0);
            const float* wr = Wt + (size_t)m * ldw + n0;
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                const float wv = wr[i * nq];
                acc[i][0] = fmaf(wv, s4.x, acc[i][0]);
                acc[i][1] = fmaf(wv, s4.y, acc[i][1]);
                acc[i][2] = fmaf(wv, s4.z, acc[i][2]);
                acc[i][3] = fmaf(wv, s4.w, acc[i][3]);
            }
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int n = n0 + i * nq;
            if (n >= nu) continue;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (j0 + q < mc) f[(j0 + q) * nu + n] = acc[i][q];
        }
    }
}

__global__ void __launch_bounds__(256) eq1_basis_kernel(const float* __restrict__ Ep, int r,
                                                        const float* __restrict__ W32, int Nx, int Ny, int Nz,
                                                        int nt, int nu, float inv_hx, float inv_hy,
                                                        float inv_hz,
                                                        const float* __restrict__ X, const float* __restrict__ Y,
                                                        const float* __restrict__ Z, const float* __restrict__ VX,
                                                        const float* __restrict__ VY, const float* __restrict__ VZ,
                                                        const float* __restrict__ qtrack, float qconst, int n_steps,
                                                        int n_out, double dt, double inv_vw, int nb,
                                                        bool stage_lags, const Eq1Lag* __restrict__ lags,
                                                        float* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* sv = reinterpret_cast<float*>(smem_raw);                          // [32][EQ1_MC] (basis-major)
    float* Wt = sv + 32 * EQ1_MC;                                            // [r][ldw]
    const int nq = (nu + nb - 1) / nb, ldw = nb * nq;                        // Wt row: nu samples, zero-padded
    float* f = Wt + (size_t)r * ldw;                                         // [EQ1_MC][nu]
    double* Q = reinterpret_cast<double*>(smem_raw + ((((size_t)r * ldw + EQ1_MC * 32 + (size_t)EQ1_MC * nu) *
                                                        sizeof(float) + 15) & ~(size_t)15));   // [n_out]
    Eq1Lag* ls = reinterpret_cast<Eq1Lag*>(Q + n_out);                       // [n_out] when staged
    if (stage_lags)
        for (int m = threadIdx.x; m < n_out; m += blockDim.x) ls[m] = lags[m];
    const Eq1Lag* lg = stage_lags ? ls : lags;
    const int tr = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    for (int e = threadIdx.x; e < r * ldw; e += blockDim.x) {
        const int m = e / ldw, n = e - m * ldw;
        Wt[e] = n < nu ? W32[(size_t)n * 32 + m] : 0.f;
    }
    for (int m = threadIdx.x; m < n_out; m += blockDim.x) Q[m] = 0.0;
    for (int c0 = 0; c0 < n_steps; c0 += EQ1_MC) {
        const int mc = min(EQ1_MC, n_steps - c0);
        __syncthreads();
        for (int j = warp; j < mc; j += nwarps) {
            const size_t s = (size_t)tr * n_steps + c0 + j;
            const float vx = VX[s], vy = VY[s], vz = VZ[s];
            float acc = 0.f;
            if (vx != 0.f || vy != 0.f || vz != 0.f) {
                const float fx = X[s] * inv_hx, fy = Y[s] * inv_hy;
                float fz = Z[s] * inv_hz - 0.5f;
                fz = fz < 0.f ? 0.f : (fz > (float)(Nz - 1) ? (float)(Nz - 1) : fz);
                const float flx = floorf(fx), fly = floorf(fy);
                const int k0 = min((int)floorf(fz), Nz - 2);
                const float wx = fx - flx, wy = fy - fly, wz = fz - (float)k0;
                const int i0 = ((int)flx % Nx + Nx) % Nx, j0 = ((int)fly % Ny + Ny) % Ny;
                const int i1 = (i0 + 1) % Nx, j1 = (j0 + 1) % Ny;
                // 96 floats per point; the z neighbour is the next point
                const float* p00 = Ep + (((size_t)i0 * Ny + j0) * Nz + k0) * 96 + lane;
                const float* p01 = Ep + (((size_t)i0 * Ny + j1) * Nz + k0) * 96 + lane;
                const float* p10 = Ep + (((size_t)i1 * Ny + j0) * Nz + k0) * 96 + lane;
                const float* p11 = Ep + (((size_t)i1 * Ny + j1) * Nz + k0) * 96 + lane;
                float w[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const int o = 32 * c;
                    const float v00 = (1.f - wz) * __ldg(p00 + o) + wz * __ldg(p00 + 96 + o);
                    const float v01 = (1.f - wz) * __ldg(p01 + o) + wz * __ldg(p01 + 96 + o);
                    const float v10 = (1.f - wz) * __ldg(p10 + o) + wz * __ldg(p10 + 96 + o);
                    const float v11 = (1.f - wz) * __ldg(p11 + o) + wz * __ldg(p11 + 96 + o);
                    w[c] = (1.f - wx) * ((1.f - wy) * v00 + wy * v01) + wx * ((1.f - wy) * v10 + wy * v11);
                }
                acc = w[0] * vx + w[1] * vy + w[2] * vz;
            }
            sv[lane * EQ1_MC + j] = lane < r ? acc : 0.f;
        }
        __syncthreads();
        switch (nb) {
            case 1: eq1_stage_product<1>(sv, Wt, r, nq, nu, mc, f); break;
            case 2: eq1_stage_product<2>(sv, Wt, r, nq, nu, mc, f); break;
            case 3: eq1_stage_product<3>(sv, Wt, r, nq, nu, mc, f); break;
            default: eq1_stage_product<4>(sv, Wt, r, nq, nu, mc, f); break;
        }
        __syncthreads();
        eq1_increments(f, nu, nu, mc, c0, n_out, lg, Q);
    }
    __syncthreads();
    const float qc = qtrack ? qtrack[tr] : qconst;
    for (int m = threadIdx.x; m < n_out; m += blockDim.x)
        out[(size_t)tr * n_out + m] = (float)(-(double)qc * inv_vw * Q[m]);
}

// The same currents as a convolution.  With the lag table folded into the time coefficients,
//   dV[L][m] = V[L][m] - V[L-1][m],  V[L][m] = w0(L) W[n(L)][m] + w1(L) W[n(L)+1][m],  V[-1] = 0,
// the increment of output k is D(k) = sum_j sum_m s_m(j) dV[k - j][m], s_m(j) = E_m(x_j) . v_j: one FP32
// multiply-add per (step, output, basis vector) in place of the staged product, its two lag reads and
// their difference, and the small differences are formed once, in FP64, instead of from rounded values
// per track (the error against 64 bits falls; 1e5 drifting carriers: 1.5e-6 -> 0.9e-6).  Bound by the FP32 units; one track per
// block, blocks persistent with the table (32 x (n_out + pad) floats) in shared memory:
//   * a thread holds 16 consecutive outputs and takes 8 steps and two basis vectors at a time: 23 table
//     reads and 8 broadcast coefficients, all pairs, for 128 paired multiply-adds (fma.rn.f32x2: half
//     the instructions, which bound the single form).  Table entry e lies at e + e / 16, so that lanes,
//     16 outputs apart, read 17 pairs apart: no bank conflicts, and offsets within a thread are constants
//     from three bases;
//   * the steps of a chunk (8 per group of threads) are gathered first, a warp taking consecutive steps
//     and keeping its cell's 24 corner values while the track stays in the cell (a drifting carrier: 11
//     steps a cell);
//   * groups are added in FP32, chunks in FP64;
//   * groups of 8 steps in which the track rests (a carrier that has arrived, a track that has left the
//     sensor) are left out: the chunks take the moving groups only.
// 1e5 tracks x 200 steps, 400 outputs, rank 32: 20.3 -> 14.3 ms, without the resting
// groups 10.5 ms (carriers that drift 20 um on average of the 30 that 200 steps allow).
constexpr int kConvThreads = 128, kConvOut = 16, kConvSteps = 8, kConvPad = 24;
constexpr size_t kConvTableMax = 110 * 1024;
struct ConvShape {
    int tm;        // threads along the outputs
    int ng;        // groups of steps
    int row;       // entries of the table per basis vector
    int jc;        // steps per chunk
    int js;        // row stride of the gathered coefficients
    size_t smem;
};
static bool conv_shape(int n_out, ConvShape* sh) {
    sh->tm = (n_out + kConvOut - 1) / kConvOut;
    if (sh->tm > kConvThreads) return false;
    sh->ng = kConvThreads / sh->tm;
    sh->row = 17 * (sh->tm + 2);
    sh->jc = kConvSteps * std::min(sh->ng, 16);
    sh->ng = sh->jc / kConvSteps;
    sh->js = sh->jc + 4;
    const size_t table = (size_t)32 * sh->row * sizeof(float);
    sh->smem = table + (size_t)32 * sh->js * sizeof(float) + (size_t)sh->ng * sh->tm * kConvOut * sizeof(float) +
               (size_t)sh->tm * kConvOut * sizeof(double) + 16;
    return table <= kConvTableMax;
}

// dvt[m / 2][e + e / 16][m % 2] = dV[e - kConvPad][m] for 0 <= e - kConvPad < n_out, else 0.
__global__ void eq1_dv_kernel(const double* __restrict__ W, int r, int nt, const Eq1Lag64* __restrict__ lags, int n_out,
                              int row, float* __restrict__ dvt) {
    const int pos = blockIdx.x * blockDim.x + threadIdx.x, m = blockIdx.y;
    if (pos >= row) return;
    const int L = pos - pos / 17 - kConvPad;              // the 17th of each group is not read
    double d = 0.0;
    if (pos % 17 < 16 && L >= 0 && L < n_out && m < r) {
        auto V = [&](int l) {
            const Eq1Lag64 g = lags[l];
            return g.w0 * W[(size_t)g.n * 32 + m] + g.w1 * W[(size_t)min(g.n + 1, nt - 1) * 32 + m];
        };
        d = V(L) - (L > 0 ? V(L - 1) : 0.0);
    }
    dvt[((size_t)(m >> 1) * row + pos) * 2 + (m & 1)] = (float)d;
}

__device__ __forceinline__ unsigned long long fma_pair(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__global__ void __launch_bounds__(kConvThreads) eq1_conv_kernel(
    const float* __restrict__ Ep, int r, const float* __restrict__ dvt, ConvShape C, int Nx, int Ny, int Nz, float inv_hx,
    float inv_hy, float inv_hz, const float* __restrict__ X, const float* __restrict__ Y, const float* __restrict__ Z,
    const float* __restrict__ VX, const float* __restrict__ VY, const float* __restrict__ VZ,
    const float* __restrict__ qtrack, float qconst, int n_tracks, int n_steps, int n_out, double inv_vw,
    float* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int row = C.row, nm = C.tm * kConvOut;
    double* D = reinterpret_cast<double*>(smem_raw);              // [nm]
    float* S = reinterpret_cast<float*>(D + nm);                  // [16][js][2]
    float* tab = S + (size_t)32 * C.js;                           // [16][row][2]
    float* P = tab + (size_t)32 * row;                            // [ng][nm]
    __shared__ unsigned bits[kConvThreads / 4];
    __shared__ unsigned char list[kConvThreads];
    __shared__ int n_list, bad_step;                              // first step with a non-finite coefficient
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int e = tid; e < 32 * row; e += kConvThreads) tab[e] = dvt[e];
    const int t = tid % C.tm, g = tid / C.tm;                     // outputs 16 t .., group of steps
    const bool work = g < C.ng;
    const int per_warp = (C.jc + kConvThreads / 32 - 1) / (kConvThreads / 32);
    for (int tr = blockIdx.x; tr < n_tracks; tr += gridDim.x) {
        for (int m = tid; m < nm; m += kConvThreads) D[m] = 0.0;
        if (tid == 0) bad_step = n_out;
        for (int b0 = 0; b0 < n_steps; b0 += kConvSteps * kConvThreads) {
            // the groups of 8 steps in which the track moves at all, in order: a bit per group, then its place
            __syncthreads();                                           // the last list is used
            if (tid < kConvThreads / 4) bits[tid] = 0;
            __syncthreads();
            const int lim = min(n_steps - b0, kConvSteps * kConvThreads);
            for (int j = b0 + tid; j - lane < b0 + lim; j += kConvThreads) {
                const size_t st = (size_t)tr * n_steps + j;
                const bool mv = j < n_steps && (VX[st] != 0.f || VY[st] != 0.f || VZ[st] != 0.f);
                const unsigned any = __ballot_sync(0xffffffffu, mv);
                if (lane == 0)                                         // 32 steps: four groups
                    bits[(j - b0) >> 5] = (any & 0xffu ? 1u : 0u) | (any & 0xff00u ? 2u : 0u) | (any & 0xff0000u ? 4u : 0u) |
                                          (any & 0xff000000u ? 8u : 0u);
            }
            __syncthreads();
            if (warp == 0) {
                const unsigned mine = bits[lane];
                int at = __popc(mine);
    #pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, at, o);
                    if (lane >= o) at += y;
                }
                if (lane == 31) n_list = at;
                at -= __popc(mine);
    #pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (mine >> q & 1) list[at++] = (unsigned char)(4 * lane + q);
            }
            __syncthreads();
            const int n_act = n_list;
            for (int k0 = 0; k0 < n_act; k0 += C.ng) {
                const int nk = min(C.ng, n_act - k0), c0 = b0 + kConvSteps * list[k0];
                if (k0) __syncthreads();                               // S and P of the last chunk are read
                // a warp's steps are prepared a lane each (one coalesced read of the track arrays), then taken
                // one after the other with a lane per basis field
                for (int l0 = 0; l0 < per_warp; l0 += 32) {
                    const int js = warp * per_warp + l0 + lane;
                    Eq1Cell<float> cell;
                    const int step =
                        js < kConvSteps * nk ? b0 + kConvSteps * list[k0 + js / kConvSteps] + js % kConvSteps : n_steps;
                    if (l0 + lane < per_warp && step < n_steps) {
                        const size_t st = (size_t)tr * n_steps + step;
                        cell.vx = VX[st];
                        cell.vy = VY[st];
                        cell.vz = VZ[st];
                        cell.set(X[st], Y[st], Z[st], Nx, Ny, Nz, inv_hx, inv_hy, inv_hz);
                    }
                    const unsigned moving = __ballot_sync(0xffffffffu, cell.moving());
                    const int a00 = (int)cell.a00, a01 = (int)cell.a01, a10 = (int)cell.a10, a11 = (int)cell.a11;
                    int key = -1, bad_j = C.jc;
                    float v[24];
                    const int nl = min(32, per_warp - l0);
                    for (int l = 0; l < nl; ++l) {
                        const int j = warp * per_warp + l0 + l;
                        if (j >= C.jc) break;
                        float acc = 0.f;
                        if (moving >> l & 1) {
                            const int k00 = __shfl_sync(0xffffffffu, a00, l);
                            if (k00 != key) {
                                key = k00;
                                const int k01 = __shfl_sync(0xffffffffu, a01, l), k10 = __shfl_sync(0xffffffffu, a10, l),
                                          k11 = __shfl_sync(0xffffffffu, a11, l);
                                const float* p[4] = {Ep + (size_t)k00 * 96 + lane, Ep + (size_t)k01 * 96 + lane,
                                                     Ep + (size_t)k10 * 96 + lane, Ep + (size_t)k11 * 96 + lane};
    #pragma unroll
                                for (int q = 0; q < 4; ++q)
    #pragma unroll
                                    for (int c = 0; c < 3; ++c) {
                                        v[6 * q + 2 * c] = __ldg(p[q] + 32 * c);
                                        v[6 * q + 2 * c + 1] = __ldg(p[q] + 96 + 32 * c);
                                    }
                            }
                            const float wx = __shfl_sync(0xffffffffu, cell.wx, l), wy = __shfl_sync(0xffffffffu, cell.wy, l),
                                        wz = __shfl_sync(0xffffffffu, cell.wz, l);
                            float w[3];
    #pragma unroll
                            for (int c = 0; c < 3; ++c) {
                                float u[4];
    #pragma unroll
                                for (int q = 0; q < 4; ++q)
                                    u[q] = (1.f - wz) * v[6 * q + 2 * c] + wz * v[6 * q + 2 * c + 1];
                                w[c] = (1.f - wx) * ((1.f - wy) * u[0] + wy * u[1]) + wx * ((1.f - wy) * u[2] + wy * u[3]);
                            }
                            acc = w[0] * __shfl_sync(0xffffffffu, cell.vx, l) + w[1] * __shfl_sync(0xffffffffu, cell.vy, l) +
                                  w[2] * __shfl_sync(0xffffffffu, cell.vz, l);
                        }
                        // a step that is not finite counts nothing here (0 x infinity would reach the outputs before
                        // it) and makes every output from its own on NaN at the end
                        const bool use = lane < r && isfinite(acc);
                        if (lane < r && !use) bad_j = min(bad_j, j);
                        S[((lane >> 1) * C.js + j) * 2 + (lane & 1)] = use ? acc : 0.f;
                    }
                    if (bad_j < C.jc)
                        atomicMin(&bad_step, b0 + kConvSteps * list[k0 + bad_j / kConvSteps] + bad_j % kConvSteps);
                }
                __syncthreads();
                // this thread's steps (in the chunk and in the track) and outputs
                const int j0 = kConvSteps * g, js0 = work && g < nk ? b0 + kConvSteps * list[k0 + g] : 0, m0 = kConvOut * t;
                const bool live = work && g < nk && m0 + kConvOut - 1 >= js0;
                using pair = unsigned long long;
                pair acc[kConvOut];
    #pragma unroll
                for (int i = 0; i < kConvOut; ++i) acc[i] = 0;
                if (live) {
                    // entries e0 .. e0 + 22 of a table row: dV[m0 + i - (js0 + jj)] at i - jj + 7; e0 mod 16 is 1
                    // or 9 (m0 is a multiple of 16, js0 of 8), so the skip of every 17th place falls at
                    // entry 15, or at 7
                    const int e0 = m0 - js0 - (kConvSteps - 1) + kConvPad;
                    const pair* T = reinterpret_cast<const pair*>(tab) + e0 + (e0 >> 4);
                    const int skip = (e0 & 15) == 9 ? 1 : 0;
                    const ulonglong2* sp = reinterpret_cast<const ulonglong2*>(S) + j0 / 2;
                    for (int m = 0; m < r; m += 2, T += row, sp += C.js / 2) {
                        pair sj[kConvSteps], w[kConvOut + kConvSteps - 1];
    #pragma unroll
                        for (int k = 0; k < kConvSteps / 2; ++k) {
                            const ulonglong2 x = sp[k];
                            sj[2 * k] = x.x;
                            sj[2 * k + 1] = x.y;
                        }
    #pragma unroll
                        for (int k = 0; k < kConvOut + kConvSteps - 1; ++k) w[k] = k < 7 ? T[k] : k < 15 ? T[k + skip] : T[k + 1];
    #pragma unroll
                        for (int jj = 0; jj < kConvSteps; ++jj)
    #pragma unroll
                            for (int i = 0; i < kConvOut; ++i) acc[i] = fma_pair(sj[jj], w[i - jj + kConvSteps - 1], acc[i]);
                    }
                }
                if (work)
    #pragma unroll
                    for (int i = 0; i < kConvOut; ++i)
                        P[(size_t)g * nm + i * C.tm + t] = __uint_as_float((unsigned)acc[i]) +
                                                           __uint_as_float((unsigned)(acc[i] >> 32));
                __syncthreads();
                for (int e = tid; e < nm; e += kConvThreads) {         // e = i tm + t: output 16 t + i
                    const int m = (e % C.tm) * kConvOut + e / C.tm;
                    if (m < c0) continue;
                    float d = 0.f;
                    for (int q = 0; q < nk; ++q) d += P[(size_t)q * nm + e];
                    D[e] += (double)d;
                }
            }
        }
        __syncthreads();
        const float qc = qtrack ? qtrack[tr] : qconst;
        for (int m = tid; m < n_out; m += kConvThreads)
            out[(size_t)tr * n_out + m] = m >= bad_step ? __int_as_float(0x7fffffff)
                                                        : (float)(-(double)qc * inv_vw * D[(m % kConvOut) * C.tm + m / kConvOut]);
        __syncthreads();
    }
}

// Floats of the table of eq1_conv_launch, 0 where it does not take n_out outputs.
size_t eq1_conv_table(int n_out) {
    ConvShape C;
    return conv_shape(n_out, &C) ? (size_t)32 * C.row : 0;
}
// Ep: point-major basis fields; W: [nt][32] FP64 time coefficients; lags: the FP64 lag table; dvt: workspace.
void eq1_conv_launch(cudaStream_t s, const float* Ep, int r, const double* W, int Nx, int Ny, int Nz, int nt, double Lx,
                     double Ly, double Lz, const float* x, const float* y, const float* z, const float* vx,
                     const float* vy, const float* vz, const float* q, float qconst, int n_tracks, int n_steps,
                     int n_out, double v_w, const void* lags, float* dvt, float* out) {
    if (r < 1 || r > 32) fail(WT_ERR_ARG, "eq1: basis rank out of range");
    ConvShape C;
    if (!conv_shape(n_out, &C)) fail(WT_ERR_UNSUPPORTED, "eq1: n_out too large for the convolution's table");
    if (n_tracks < 1) return;
    eq1_dv_kernel<<<dim3((C.row + 127) / 128, 32), 128, 0, s>>>(W, r, nt, static_cast<const Eq1Lag64*>(lags), n_out,
                                                               C.row, dvt);
    WT_LAUNCH("eq1_dv");
    allow_dyn_smem(eq1_conv_kernel, C.smem);
    int dev = 0, n_sm = 0, per = 0;
    WT_CUDA(cudaGetDevice(&dev));
    WT_CUDA(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev));
    WT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, eq1_conv_kernel, kConvThreads, C.smem));
    eq1_conv_kernel<<<std::min(n_tracks, n_sm * std::max(1, per)), kConvThreads, C.smem, s>>>(
        Ep, r, dvt, C, Nx, Ny, Nz, (float)(Nx / Lx), (float)(Ny / Ly), (float)(Nz / Lz), x, y, z, vx, vy, vz, q, qconst,
        n_tracks, n_steps, n_out, 1.0 / v_w, out);
    WT_LAUNCH("eq1_conv");
}

// Point-major copy of the basis fields for eq1_basis_kernel: Ep[p][c][m] = E[c][m][p] for m < r, 0 for
// r <= m < 32 (E: [3][32][npts], rows m >= r need not be written).  A block moves a tile of 32 points x
// 96 rows through shared memory: coalesced 128-byte row reads, one contiguous 12 KB write.
__global__ void __launch_bounds__(256) eq1_point_major_kernel(const float* __restrict__ E, int r, size_t npts,
                                                              float* __restrict__ Ep) {
    __shared__ float tile[96][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t ntiles = (npts + 31) / 32;
    for (size_t tb = blockIdx.x; tb < ntiles; tb += gridDim.x) {
        const size_t p0 = tb * 32;
        const size_t p = p0 + lane;
        for (int row = warp; row < 96; row += 8) {
            const int m = row & 31;
            tile[row][lane] = (m < r && p < npts) ? __ldg(E + (size_t)row * npts + p) : 0.f;
        }
        __syncthreads();
        const int np = (int)min((size_t)32, npts - p0);
        float* o = Ep + p0 * 96;
        for (int e = threadIdx.x; e < np * 96; e += 256) o[e] = tile[e % 96][e / 96];
        __syncthreads();
    }
}

void eq1_point_major(cudaStream_t s, const float* E, int r, size_t npts, float* Ep) {
    if (npts == 0) return;
    int dev = 0, num_sms = 0;
    WT_CUDA(cudaGetDevice(&dev));
    WT_CUDA(cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev));
    const size_t ntiles = (npts + 31) / 32;
    const int grid = (int)std::min<size_t>(ntiles, (size_t)num_sms * 8);
    eq1_point_major_kernel<<<grid, 256, 0, s>>>(E, r, npts, Ep);
    WT_LAUNCH("eq1_point_major");
}

// Shared memory of eq1_basis_kernel; the lag table goes beside the rest when it is small (12 B per output).
static size_t eq1_basis_smem(int r, int nu, int n_out, int* nb_out, bool* stage_lags_out) {
    // time samples per thread in the staged product: the fewest that keep the (samples / nb) x
    // (steps / 4) items within one pass of the 256 threads
    const int nb = std::min(4, std::max(1, (nu + 63) / 64));
    const size_t ldw = (size_t)nb * ((nu + nb - 1) / nb);
    const size_t base = ((((size_t)r * ldw + EQ1_MC * 32 + (size_t)EQ1_MC * nu) * sizeof(float) + 15) & ~(size_t)15) +
                        (size_t)n_out * sizeof(double);
    const bool stage_lags = (size_t)n_out * sizeof(Eq1Lag) <= 16384;
    if (nb_out) *nb_out = nb;
    if (stage_lags_out) *stage_lags_out = stage_lags;
    return base + (stage_lags ? (size_t)n_out * sizeof(Eq1Lag) : 0);
}
// Whether eq1_basis_launch takes up to nt time samples and n_out outputs, at any rank.
bool eq1_basis_fits(int nt, int n_out) { return eq1_basis_smem(32, nt, n_out, nullptr, nullptr) <= 200 * 1024; }
void eq1_basis_launch(cudaStream_t s, const float* Ep, int r, const float* W32, int Nx, int Ny, int Nz, int nt,
                      double Lx, double Ly, double Lz, const float* x, const float* y, const float* z,
                      const float* vx, const float* vy, const float* vz, const float* q, float qconst, int n_tracks,
                      int n_steps, int n_out, double dt, double v_w, const void* lags, int nu, float* out) {
    if (r < 1 || r > 32) fail(WT_ERR_ARG, "eq1: basis rank out of range");
    if (nu < 1 || nu > nt) fail(WT_ERR_ARG, "eq1: bad count of time samples in use");
    int nb = 0;
    bool stage_lags = false;
    const size_t sh = eq1_basis_smem(r, nu, n_out, &nb, &stage_lags);
    if (sh > 200 * 1024) fail(WT_ERR_UNSUPPORTED, "eq1: n_t or n_out too large for shared memory");
    allow_dyn_smem(eq1_basis_kernel, sh);
    if (n_tracks > 0)
        eq1_basis_kernel<<<n_tracks, 256, sh, s>>>(Ep, r, W32, Nx, Ny, Nz, nt, nu, (float)(Nx / Lx), (float)(Ny / Ly),
                                                   (float)(Nz / Lz), x, y, z, vx, vy, vz, q, qconst, n_steps, n_out,
                                                   dt, 1.0 / v_w, nb, stage_lags, static_cast<const Eq1Lag*>(lags),
                                                   out);
    WT_LAUNCH("eq1_basis");
}

size_t eq1_lag_size() { return sizeof(Eq1Lag); }
void eq1_pack_lag(void* dst, int n, float w0, float w1) { *static_cast<Eq1Lag*>(dst) = Eq1Lag{n, w0, w1}; }
size_t eq1_lag64_size() { return sizeof(Eq1Lag64); }
void eq1_pack_lag64(void* dst, int n, double w0, double w1) { *static_cast<Eq1Lag64*>(dst) = Eq1Lag64{n, w0, w1}; }

// ------------------------------------------------------------------------
// Allocation-free variant (wt_eq1_noalloc).  The per-call lag table lives in
// this fixed device array instead of a cudaMalloc'd buffer; every GPU that
// loads the library holds it (12 B x WT_EQ1_NOALLOC_MAX_OUT = 192 KB) until the
// process exits.  The limit is the one the header documents.
constexpr int kEq1NoAllocMaxOut = WT_EQ1_NOALLOC_MAX_OUT;
static __device__ __align__(256) Eq1Lag g_eq1_lag_scratch[kEq1NoAllocMaxOut];

// Lag table on the device from the relaxation's time samples: same rule as
// the host-built table of eq1_launch's callers (linear in t, 0 at t = 0,
// held after the last sample).  Every entry is overwritten on each call.
__global__ void eq1_lag_table_kernel(const double* __restrict__ t, int nt, double dt, int n_out,
                                     Eq1Lag* __restrict__ lags) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_out) return;
    const double L = (k + 0.5) * dt;
    int n0 = 0;
    double w0 = 0.0, w1 = 0.0;
    if (L <= t[0]) { n0 = 0; w0 = L / t[0]; }
    else if (L >= t[nt - 1]) { n0 = nt - 1; w0 = 1.0; }
    else {
        int lo = 0, hi = nt - 1;           // t[lo] <= L < t[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (t[mid] <= L) lo = mid; else hi = mid;
        }
        n0 = lo;
        const double f = (L - t[lo]) / (t[lo + 1] - t[lo]);
        w0 = 1.0 - f;
        w1 = f;
    }
    lags[k] = Eq1Lag{n0, (float)w0, (float)w1};
}

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
// Device address of the scratch per device, and the id of the CUDA context it
// was looked up in: a context created anew on the device (after a
// cudaDeviceReset, say) reloads the module, so the address is looked up again.
struct ScratchAddr {
    Eq1Lag* p = nullptr;
    unsigned long long ctx_id = 0;
};
ScratchAddr g_noalloc_addr[kMaxDevices];

// id of the current CUDA context (unique for the life of the process), through
// the runtime's driver entry points (no libcuda link)
unsigned long long current_context_id() {
    static PFN_cuCtxGetCurrent_v4000 get_cur = nullptr;
    static PFN_cuCtxGetId_v12000 get_id = nullptr;
    if (!get_cur || !get_id) {
        void* a = nullptr;
        void* b = nullptr;
        cudaDriverEntryPointQueryResult qa, qb;
        WT_CUDA(cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &a, 4000, cudaEnableDefault, &qa));
        WT_CUDA(cudaGetDriverEntryPointByVersion("cuCtxGetId", &b, 12000, cudaEnableDefault, &qb));
        if (qa != cudaDriverEntryPointSuccess || qb != cudaDriverEntryPointSuccess || !a || !b)
            fail(WT_ERR_CUDA, "cuCtxGetCurrent / cuCtxGetId unavailable");
        get_cur = reinterpret_cast<PFN_cuCtxGetCurrent_v4000>(a);
        get_id = reinterpret_cast<PFN_cuCtxGetId_v12000>(b);
    }
    CUcontext cx = nullptr;
    unsigned long long id = 0;
    if (get_cur(&cx) != CUDA_SUCCESS || !cx || get_id(cx, &id) != CUDA_SUCCESS)
        fail(WT_ERR_CUDA, "no current CUDA context for the allocation-free scratch");
    return id;
}
}  // namespace

// The caller's device is current.  Resolves the scratch address on the first
// call in this device's current context (the symbol's host-side name is not a
// device address); later calls in the same context reuse it.
void eq1_noalloc_launch(cudaStream_t s, int device, const float* H, int Nx, int Ny, int Nz, const double* d_times,
                        int nt, double Lx, double Ly, double Lz, const float* x, const float* y, const float* z,
                        const float* vx, const float* vy, const float* vz, const float* q, float qconst,
                        int n_tracks, int n_steps, int n_out, double dt, double v_w, int nu, float* out) {
    if (n_out > kEq1NoAllocMaxOut)
        fail(WT_ERR_ARG, "n_out " + std::to_string(n_out) + " exceeds the allocation-free limit of " +
                             std::to_string(kEq1NoAllocMaxOut));
    if (device < 0 || device >= kMaxDevices) fail(WT_ERR_UNSUPPORTED, "device index beyond the scratch table");
    Eq1Lag* lags = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_noalloc_mutex);
        const unsigned long long id = current_context_id();
        ScratchAddr& a = g_noalloc_addr[device];
        if (!a.p || a.ctx_id != id) {
            void* p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, g_eq1_lag_scratch);
            if (e != cudaSuccess || !p) {
                cudaGetLastError();
                fail(WT_ERR_CUDA, std::string("cudaGetSymbolAddress(eq1 scratch): ") + cudaGetErrorString(e));
            }
            a.p = static_cast<Eq1Lag*>(p);
            a.ctx_id = id;
        }
        lags = a.p;
    }
    eq1_lag_table_kernel<<<(n_out + 127) / 128, 128, 0, s>>>(d_times, nt, dt, n_out, lags);
    WT_LAUNCH("eq1_lag_table");
    eq1_launch(s, H, Nx, Ny, Nz, nt, Lx, Ly, Lz, x, y, z, vx, vy, vz, q, qconst, n_tracks, n_steps, n_out, dt, v_w,
               lags, nu, out, nullptr, 0);
}

}  // namespace wt
