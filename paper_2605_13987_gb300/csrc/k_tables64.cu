// FP64 field of many time samples from per-column lateral tables (Sec. 3's translated
// fundamental-solution chunks in spectral form, FP64):
//   T_c[a][kz][xy] = pref w_a(kz) sum over the lateral band of component a's factor at (x - x_c, y - y_c),
//       a = x, y: w = 1 (kz = 0) or 2;  a = z: w = 2 kz
//   R[a][kz][t][xy] = sum_c Zc[t][c][kz] T_c[a][kz][xy]
//   H[t][a][xy][z]  = sum_kz R[a][kz][t][xy] cos or sin(kz z)        (a product, on the tensor cores)
// The lateral transforms are taken once per context instead of once per time sample, and the z series,
// a double-length complex FFT of FP64 units' speed per line before, is a product with N_z x N_z cosines.
// 3 x 3 cell, 60 x 60 x 120, 64 samples: 26.3 -> 5.8 ms (the combination's 18 FP64 multiply-adds per
// value take 2.4 of it); the tables take 2.5 ms once.
#include "wt_internal.cuh"

#include <algorithm>

namespace wt {

// F[(x, u, f)][mx] at the grid's x: f = 0 wx cos(kx dx), 1: 2 kx sin(kx dx).
__global__ void t64_xfactor_kernel(const double* __restrict__ ux, int nx, int n_ux, double Lx, double* __restrict__ F) {
    const int hx = nx / 2;
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)nx * n_ux * hx) return;
    const int mx = (int)(e % hx);
    const size_t xu = e / hx;
    const double rel = (double)(xu / n_ux) / nx - ux[xu % n_ux] / Lx;
    double sn, cs;
    sincospi(2.0 * mx * rel, &sn, &cs);
    F[(2 * xu) * hx + mx] = (mx ? 2.0 : 1.0) * cs;
    F[(2 * xu + 1) * hx + mx] = 2.0 * (2.0 * kPi * mx / Lx) * sn;
}

// Y[c][f][my][y]: f = 0 wy cos(ky dy), 1: 2 ky sin(ky dy).
__global__ void t64_yfactor_kernel(const double* __restrict__ col_y, int n_cols, int ny, double Ly,
                                   double* __restrict__ Y) {
    const int hy = ny / 2;
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)n_cols * hy * ny) return;
    const int y = (int)(e % ny), my = (int)(e / ny % hy), c = (int)(e / ny / hy);
    double sn, cs;
    sincospi(2.0 * my * ((double)y / ny - col_y[c] / Ly), &sn, &cs);
    double* o = Y + ((size_t)c * 2 * hy + my) * ny + y;
    o[0] = (my ? 2.0 : 1.0) * cs;
    o[(size_t)hy * ny] = 2.0 * (2.0 * kPi * my / Ly) * sn;
}

// One block per (x, kz chunk, column): threads over y, the chunk's k_x sums in shared memory.
constexpr int kT64Z = 8;
__global__ void __launch_bounds__(128) t64_build_kernel(const double* __restrict__ Y, const int* __restrict__ col_u,
                                                        int n_ux, int nx, int ny, int nz, double Lz, double pref, const double* __restrict__ G,
                                                        double* __restrict__ T) {
    extern __shared__ double sh[];                 // [hy][kT64Z] x (cos and sin part of G)
    const int hy = ny / 2, x = blockIdx.x, kz0 = blockIdx.y * kT64Z, c = blockIdx.z;
    const int nk = min(kT64Z, nz - kz0);
    double* gc = sh;
    double* gs = sh + (size_t)hy * kT64Z;
    const double* g = G + 2 * ((size_t)x * n_ux + col_u[c]) * hy * nz;
    for (int e = threadIdx.x; e < hy * kT64Z; e += blockDim.x) {
        const int my = e / kT64Z, k = e % kT64Z;
        gc[e] = k < nk ? g[(size_t)my * nz + kz0 + k] : 0.0;
        gs[e] = k < nk ? g[(size_t)(hy + my) * nz + kz0 + k] : 0.0;
    }
    __syncthreads();
    const size_t nxy = (size_t)nx * ny;
    for (int y = threadIdx.x; y < ny; y += blockDim.x) {
        const double* yf = Y + (size_t)c * 2 * hy * ny + y;
        double ax[kT64Z] = {}, ay[kT64Z] = {}, a0[kT64Z] = {};
        for (int my = 0; my < hy; ++my) {
            const double cy = yf[(size_t)my * ny], sy = yf[(size_t)(hy + my) * ny];
#pragma unroll
            for (int k = 0; k < kT64Z; ++k) {
                ax[k] = fma(cy, gs[my * kT64Z + k], ax[k]);
                ay[k] = fma(sy, gc[my * kT64Z + k], ay[k]);
                a0[k] = fma(cy, gc[my * kT64Z + k], a0[k]);
            }
        }
        for (int k = 0; k < nk; ++k) {
            const int kz = kz0 + k;
            double* o = T + ((size_t)c * 3 * nz + kz) * nxy + (size_t)x * ny + y;
            const double w = pref * (kz ? 2.0 : 1.0);
            o[0] = w * ax[k];
            o[(size_t)nz * nxy] = w * ay[k];
            o[(size_t)2 * nz * nxy] = pref * 2.0 * (kPi * kz / Lz) * a0[k];
        }
    }
}

// CS[z][kz] = cos(kz z), then sin(kz z).
__global__ void t64_series_kernel(int nz, double* __restrict__ CS) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nz * nz) return;
    const int z = e / nz, kz = e % nz;
    double sn, cs;
    sincospi((double)kz * (2 * z + 1) / (2.0 * nz), &sn, &cs);
    CS[e] = cs;
    CS[(size_t)nz * nz + e] = sn;
}

// R[a][kz][t][xy] for nb time samples, kB of them per thread and pass; grid (xy, kz, a).  The FP64 units
// bound it, so kB is the one of 2, 4, 8, 12, 16 that leaves the fewest samples of a pass empty (18 columns,
// 128 x 128 x 256, three samples at a time: 5.8 ms with kB = 16, 1.45 with 4) among those whose coefficients
// of all columns fit a block's shared memory (16 up to 1 600 columns).
template <int kB>
__global__ void __launch_bounds__(128) t64_combine_kernel(const double* __restrict__ T, const double* __restrict__ Zc,
                                                          int n_cols, int nz, size_t nxy, int nb,
                                                          double* __restrict__ R) {
    extern __shared__ __align__(16) double zs[];   // [n_cols][kB]
    const int kz = blockIdx.y, a = blockIdx.z;
    const size_t xy = (size_t)blockIdx.x * 128 + threadIdx.x;
    const bool in = xy < nxy;
    const double* t = T + ((size_t)a * nz + kz) * nxy + (in ? xy : 0);
    double* r = R + ((size_t)a * nz + kz) * nb * nxy + (in ? xy : 0);
    for (int b0 = 0; b0 < nb; b0 += kB) {
        __syncthreads();
        for (int e = threadIdx.x; e < n_cols * kB; e += 128) {
            const int b = b0 + e % kB;
            zs[e] = b < nb ? Zc[((size_t)b * n_cols + e / kB) * nz + kz] : 0.0;
        }
        __syncthreads();
        if (!in) continue;
        double acc[kB];
#pragma unroll
        for (int b = 0; b < kB; ++b) acc[b] = 0.0;
#pragma unroll 2
        for (int c = 0; c < n_cols; ++c) {
            const double v = t[(size_t)c * 3 * nz * nxy];
#pragma unroll
            for (int b = 0; b < kB; ++b) acc[b] = fma(zs[c * kB + b], v, acc[b]);
        }
#pragma unroll
        for (int b = 0; b < kB; ++b)
            if (b0 + b < nb) r[(size_t)(b0 + b) * nxy] = acc[b];
    }
}

constexpr size_t kT64Coefs = 200 * 1024;
static int t64_pass(int nb, int n_cols) {
    int best = 2;
    for (int q : {4, 8, 12, 16})
        if ((size_t)n_cols * q * sizeof(double) <= kT64Coefs && (nb + q - 1) / q * q <= (nb + best - 1) / best * best) best = q;
    return best;
}
// Whether the combination takes so many columns.
bool t64_takes(int n_cols) { return (size_t)n_cols * 2 * sizeof(double) <= kT64Coefs; }
template <int kB>
static void t64_combine(cudaStream_t s, const double* T, const double* Zc, int n_cols, int nz, size_t nxy, int nb,
                        double* R) {
    const size_t sh = (size_t)n_cols * kB * sizeof(double);
    allow_dyn_smem(t64_combine_kernel<kB>, sh);
    t64_combine_kernel<kB><<<dim3((unsigned)((nxy + 127) / 128), nz, 3), 128, sh, s>>>(T, Zc, n_cols, nz, nxy, nb, R);
    WT_LAUNCH("t64_combine");
}

// Tables T [n_cols][3][Nz][Nx Ny] and the series matrices CS [2][Nz][Nz].  hux: distinct column x, hcu[c]
// which one column c has; F, G, Y: work buffers of Nx n_ux Nx, Nx n_ux Ny Nz and n_cols Ny Ny
// values.
void t64_build(cudaStream_t s, const double* ux, const int* col_u, const double* col_y, int n_cols, int n_ux, int Nx,
               int Ny, int Nz, double Lx, double Ly, double Lz, double pref, const double* invk2, double* F, double* G,
               double* Y, double* T, double* CS) {
    const int hx = Nx / 2, hy = Ny / 2;
    const size_t nf = (size_t)Nx * n_ux * hx;
    t64_xfactor_kernel<<<(unsigned)((nf + 255) / 256), 256, 0, s>>>(ux, Nx, n_ux, Lx, F);
    WT_LAUNCH("t64_xfactor");
    dgemm(s, false, false, 2 * Nx * n_ux, hy * Nz, hx, 1.0, F, hx, invk2, hy * Nz, 0.0, G, hy * Nz);
    const size_t ny = (size_t)n_cols * hy * Ny;
    t64_yfactor_kernel<<<(unsigned)((ny + 255) / 256), 256, 0, s>>>(col_y, n_cols, Ny, Ly, Y);
    WT_LAUNCH("t64_yfactor");
    const size_t sh = 2 * (size_t)hy * kT64Z * sizeof(double);
    allow_dyn_smem(t64_build_kernel, sh);
    t64_build_kernel<<<dim3(Nx, (Nz + kT64Z - 1) / kT64Z, n_cols), 128, sh, s>>>(Y, col_u, n_ux, Nx, Ny, Nz, Lz, pref, G, T);
    WT_LAUNCH("t64_build");
    t64_series_kernel<<<(Nz * Nz + 255) / 256, 256, 0, s>>>(Nz, CS);
    WT_LAUNCH("t64_series");
}

// Bytes of the products' workspace for nb time samples at a time.
size_t t64_work(int nb, int Nx, int Ny, int Nz) { return dgemm_tc_rows_bytes(nb * Nx * Ny, Nz, Nz); }

// H[t][a][xy][z] of nb time samples (out: the first one's) from Zc [nb][n_cols][Nz]; R: 3 Nz nb Nx Ny values.
void t64_fields(cudaStream_t s, const double* T, const double* CS, const double* Zc, int nb, int n_cols, int Nx, int Ny,
                int Nz, double* R, unsigned char* ws, int* d_err, double* out) {
    const size_t nxy = (size_t)Nx * Ny, npts = nxy * Nz;
    switch (t64_pass(nb, n_cols)) {
        case 2: t64_combine<2>(s, T, Zc, n_cols, Nz, nxy, nb, R); break;
        case 4: t64_combine<4>(s, T, Zc, n_cols, Nz, nxy, nb, R); break;
        case 8: t64_combine<8>(s, T, Zc, n_cols, Nz, nxy, nb, R); break;
        case 12: t64_combine<12>(s, T, Zc, n_cols, Nz, nxy, nb, R); break;
        default: t64_combine<16>(s, T, Zc, n_cols, Nz, nxy, nb, R);
    }
    const int M = (int)(nb * nxy);
    for (int a = 0; a < 3; ++a)
        dgemm_tc_rows(s, M, Nz, Nz, R + (size_t)a * Nz * M, M, CS + (a == 2 ? (size_t)Nz * Nz : 0), Nz,
                      out + (size_t)a * npts, Nz, (int)nxy, 3 * npts, ws, d_err);
}

}  // namespace wt
