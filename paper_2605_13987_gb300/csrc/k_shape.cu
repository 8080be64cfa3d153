// Front-end shaping of Eq. 1 currents: CR-(RC)^n impulse response of unit
// area, h(t) = (t / tau)^n e^(-t / tau) / (n! tau), convolved on the output
// grid by the rectangle rule, v_m = G sum_k h(k dt) dt i_(m-k) + sigma w_m
// (the paper names the electronics' response as a step of the signal chain
// without a transfer function; this is its parameterised form).
#include "wt_internal.cuh"

#include <algorithm>
#include <cmath>

namespace wt {

// The sampled response is t^n e^-t on a grid, so the convolution is a recursion: with a = e^{-dt/tau}
// and S_k[m] = sum_j C(j, k) a^j i_(m-j),
//   S_k[m] = a (S_k[m-1] + S_{k-1}[m-1])   (k = 0: S_0[m] = a S_0[m-1] + i_m),
// and j^n = sum_k S2(n, k) k! C(j, k) (Stirling numbers of the second kind) gives
//   v_m = sum_k c_k S_k[m],  c_k = G dt / (n! tau) (dt / tau)^n S2(n, k) k!.
// Every coefficient is positive, so nothing cancels that does not cancel in the sum itself.  3 n + 2
// FP64 operations per sample instead of one per tap (the FP64 units bound both: 20 000 tracks x 200
// samples, order 2: 3.15 -> 0.21 ms).  One lane per track, tiles of 32 tracks x 32 samples through shared
// memory for coalesced rows.  Taps beyond (n + 60) tau, which the definition drops, are below e^-50 of
// the peak and stay in.  A track with an infinity or a NaN in it is convolved tap by tap instead (the
// recursion would carry it past the last tap).
constexpr int kShapeWarps = 4;
struct ShapeCoef {
    double c[21];
};

// one track by its taps, from the last sample down (cur may be v)
__device__ void shape_taps(const float* __restrict__ noise, const float* x, int n_out, int n_taps, double dt,
                           double tau, int order, double scale, double noise_rms, float* v, int lane) {
    for (int m0 = (n_out - 1) & ~31; m0 >= 0; m0 -= 32) {
        const int m = m0 + lane;
        double acc = 0.0;
        if (m < n_out) {
            const int kmax = min(m, n_taps - 1);
            for (int k = 0; k <= kmax; ++k) {
                const double t = k * dt / tau;
                acc = fma(scale * pow(t, (double)order) * exp(-t), (double)x[m - k], acc);
            }
            if (noise) acc += noise_rms * (double)noise[m];
        }
        __syncwarp();
        if (m < n_out) v[m] = (float)acc;
    }
}

// Few tracks: one block per track, the taps (FP64) and the track's currents in shared memory, threads
// over output samples.  The recursion takes its samples one after the other, about 0.7 us each
// (order 2) whatever the count of tracks, so it needs enough of them (see shape_launch).
__global__ void shape_direct_kernel(const float* cur, int n_out, int n_taps, double dt, double tau, int order,
                                    double scale, double noise_rms, const float* __restrict__ noise, float* v) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* taps = reinterpret_cast<double*>(smem_raw);
    float* row = reinterpret_cast<float*>(taps + n_taps);
    const size_t tr = blockIdx.x;
    for (int k = threadIdx.x; k < n_taps; k += blockDim.x) {
        const double x = k * dt / tau;
        taps[k] = scale * pow(x, (double)order) * exp(-x);        // scale = G dt / (n! tau)
    }
    for (int m = threadIdx.x; m < n_out; m += blockDim.x) row[m] = cur[tr * n_out + m];
    __syncthreads();
    for (int m = threadIdx.x; m < n_out; m += blockDim.x) {
        double acc = 0.0;
        const int kmax = min(m, n_taps - 1);
        for (int k = 0; k <= kmax; ++k) acc = fma(taps[k], (double)row[m - k], acc);
        if (noise) acc += noise_rms * (double)noise[tr * n_out + m];
        v[tr * n_out + m] = (float)acc;
    }
}

// N: order, or -1 for orders above 4 (states in an array of 21)
template <int N>
__global__ void __launch_bounds__(32 * kShapeWarps) shape_kernel(const float* cur, int n_tracks,
                                                                 int n_out, int n_taps, double dt, double tau,
                                                                 int order_arg, double scale, ShapeCoef C, double a,
                                                                 double noise_rms, const float* __restrict__ noise,
                                                                 float* v) {
    __shared__ float xin[kShapeWarps][32][33];
    __shared__ double xout[kShapeWarps][32][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int order = N >= 0 ? N : order_arg;
    const long long t0 = ((long long)blockIdx.x * kShapeWarps + w) * 32;
    if (t0 >= n_tracks) return;
    const int nt = (int)min((long long)32, n_tracks - t0);
    constexpr int NS = N >= 0 ? N + 1 : 21;
    double S[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) S[k] = 0.0;
    unsigned bad = 0;                                    // tracks with an infinity or a NaN, by lane
    if (cur == v)                                        // known before the first store only where it matters
        for (int r = 0; r < nt; ++r) {
            bool b = false;
            for (int m = lane; m < n_out; m += 32) b = b || !isfinite(cur[(size_t)(t0 + r) * n_out + m]);
            if (__any_sync(0xffffffffu, b)) bad |= 1u << r;
        }
    bool mine = false;
    for (int m0 = 0; m0 < n_out; m0 += 32) {
        const int m = m0 + lane;
        __syncwarp();
#pragma unroll 8
        for (int r = 0; r < nt; ++r) xin[w][r][lane] = m < n_out ? cur[(size_t)(t0 + r) * n_out + m] : 0.f;
        __syncwarp();
        const int nm = min(32, n_out - m0);
        if (lane < nt) {
#pragma unroll 4
            for (int q = 0; q < nm; ++q) {
                const float xf = xin[w][lane][q];
                mine = mine || !isfinite(xf);
                double acc;
                if constexpr (N >= 0) {
#pragma unroll
                    for (int k = N; k > 0; --k) S[k] = a * (S[k] + S[k - 1]);
                    S[0] = fma(a, S[0], (double)xf);
                    acc = C.c[0] * S[0];
#pragma unroll
                    for (int k = 1; k <= N; ++k) acc = fma(C.c[k], S[k], acc);
                } else {
                    acc = 0.0;
#pragma unroll
                    for (int k = NS - 1; k > 0; --k)
                        if (k <= order) S[k] = a * (S[k] + S[k - 1]);
                    S[0] = fma(a, S[0], (double)xf);
#pragma unroll
                    for (int k = 0; k < NS; ++k)
                        if (k <= order) acc = fma(C.c[k], S[k], acc);
                }
                xout[w][lane][q] = acc;
            }
        }
        __syncwarp();
        if (m < n_out)
#pragma unroll 8
            for (int r = 0; r < nt; ++r) {
                if (bad >> r & 1) continue;
                const size_t at = (size_t)(t0 + r) * n_out + m;
                double acc = xout[w][r][lane];
                if (noise) acc += noise_rms * (double)noise[at];
                v[at] = (float)acc;
            }
    }
    bad |= __ballot_sync(0xffffffffu, mine);
    __syncwarp();
    for (; bad; bad &= bad - 1) {
        const size_t at = (size_t)(t0 + __ffs(bad) - 1) * n_out;
        shape_taps(noise ? noise + at : nullptr, cur + at, n_out, n_taps, dt, tau, order, scale, noise_rms, v + at, lane);
    }
}

void shape_launch(cudaStream_t s, const float* cur, int n_tracks, int n_out, double dt, double tau, int order,
                  double gain, double noise_rms, const float* noise, float* v) {
    // taps beyond t = (order + 60) tau are below e^-50 of the peak and are dropped
    const double span = (order + 60.0) * tau / dt;
    const int n_taps = (int)std::max(1.0, std::min((double)n_out, std::ceil(span)));
    double fact = 1.0;
    for (int k = 2; k <= order; ++k) fact *= k;
    const double scale = gain * dt / (fact * tau);
    ShapeCoef C{};
    double s2[21] = {1.0}, kf = 1.0;                      // S2(n, k), n growing to order
    for (int n = 1; n <= order; ++n) {
        for (int k = n; k > 0; --k) s2[k] = k * s2[k] + s2[k - 1];
        s2[0] = 0.0;
    }
    const double step = std::pow(dt / tau, order);
    for (int k = 0; k <= order; ++k) {
        if (k > 1) kf *= k;
        C.c[k] = scale * step * s2[k] * kf;
    }
    const double a = std::exp(-dt / tau);
    const int blocks = (n_tracks + 32 * kShapeWarps - 1) / (32 * kShapeWarps);
    // Estimated times in us, fitted to orders 0-20, 50-2 000 samples and 1-20 000 tracks: tap by tap a
    // block's own chain or all multiply-adds at 1.4e11/s and 24 ns a block; the recursion its chain of
    // samples (0.5 us and 0.11 per order; 3.3 us in the array form) and 16 ps a sample.  Order 2, 200
    // samples: 31 us against 142 at 152 tracks, 250 against 142 at 1 500.
    const double nn = n_out, mean_taps = n_taps >= n_out ? 0.5 * nn : n_taps * (1.0 - 0.5 * n_taps / nn);
    const double t_direct = std::max(std::ceil(nn / 256) * n_taps * 0.13, n_tracks * (0.024 + nn * mean_taps / 1.4e5));
    const double t_rec = nn * (order <= 4 ? 0.5 + 0.11 * order : 3.3) + 1.6e-5 * nn * n_tracks;
    // (dt / tau)^n, which the recursion's coefficients hold, must be a normal number (order 20: dt / tau of 1e-15 to
    // 1e15); the taps hold it times a power of the lag and e^-t
    if (n_tracks > 0 && (t_direct <= t_rec || !std::isnormal(step))) {
        const size_t sh = (size_t)n_taps * sizeof(double) + (size_t)n_out * sizeof(float);
        allow_dyn_smem(shape_direct_kernel, sh);
        shape_direct_kernel<<<n_tracks, 256, sh, s>>>(cur, n_out, n_taps, dt, tau, order, scale, noise_rms, noise, v);
    } else if (n_tracks > 0) {
#define WT_SHAPE(N)                                                                                               \
    shape_kernel<N><<<blocks, 32 * kShapeWarps, 0, s>>>(cur, n_tracks, n_out, n_taps, dt, tau, order, scale, C, a, \
                                                        noise_rms, noise, v)
        switch (order) {
            case 0: WT_SHAPE(0); break;
            case 1: WT_SHAPE(1); break;
            case 2: WT_SHAPE(2); break;
            case 3: WT_SHAPE(3); break;
            case 4: WT_SHAPE(4); break;
            default: WT_SHAPE(-1); break;
        }
#undef WT_SHAPE
    }
    WT_LAUNCH("shape");
}

}  // namespace wt
