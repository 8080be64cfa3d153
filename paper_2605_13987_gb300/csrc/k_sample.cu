// Exact FP64 point evaluation of the field (the band-limited spectral sum of
// the bulk extension, Abstract / Sec. 1, at arbitrary points):
//   W_x(p) = pref sum_c sum_mz w(mz) Zc(mz) cos(kz z_p) Lx(p - x_c; kz)
//   W_y(p) = pref sum_c sum_mz w(mz) Zc(mz) cos(kz z_p) Ly(p - x_c; kz)
//   W_z(p) = pref sum_c sum_mz Zc(mz) 2 kz sin(kz z_p) L0(p - x_c; kz)
// with the lateral sums over all (kx, ky) of the band:
//   Lx = sum kx sin(kx dx) cos(ky dy)/|k|^2, Ly = sum ky cos(kx dx) sin(ky dy)/|k|^2,
//   L0 = sum cos(kx dx) cos(ky dy)/|k|^2  (k = 0 excluded).
#include "wt_internal.cuh"

namespace wt {

// The sums factor by axis.  Columns share few distinct x coordinates (a 3 x 3 matrix's 18 columns: 6),
// so the k_x sums are taken once per (point, distinct x), as one FP64 product (on the tensor cores)
//   G[p][u][my][mz] = sum_mx F[p][u][mx] T[mx][my][mz],   F = wx cos(kx dx) and 2 kx sin(kx dx),
// the k_y sums and the z factors per (point, column, mz), and the sum over columns and mz for all times
// as another product.  500 points, 16 times, 18 columns, 64 x 64 x 128: 38.4 -> 1.1 ms of kernels.

// F[(p, u, f)][mx], f = 0: wx cos, 1: 2 kx sin.
__global__ void sample_xfactor_kernel(const double* __restrict__ pts, const double* __restrict__ ux, int n_pts,
                                      int n_ux, int hx, double Lx, double* __restrict__ F) {
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)n_pts * n_ux * hx) return;
    const int mx = (int)(e % hx);
    const size_t pu = e / hx;
    const double dx = pts[3 * (pu / n_ux)] - ux[pu % n_ux];
    double sn, cs;
    sincospi(2.0 * mx * dx / Lx, &sn, &cs);
    F[(2 * pu) * hx + mx] = (mx ? 2.0 : 1.0) * cs;
    F[(2 * pu + 1) * hx + mx] = 2.0 * (2.0 * kPi * mx / Lx) * sn;
}

// Lat[p][a][c][mz] = pref x (z factor of component a) x (k_y sum); a block per (point, column).
__global__ void __launch_bounds__(128) sample_lateral_kernel(const double* __restrict__ pts,
                                                             const double* __restrict__ col_xy,
                                                             const int* __restrict__ col_u, int n_cols, int n_ux,
                                                             int hy, int nz, double Ly, double Lz, double pref,
                                                             const double* __restrict__ G, double* __restrict__ Lat) {
    extern __shared__ double sh[];
    double* cy = sh;                       // wy cos(ky dy)
    double* sy = cy + hy;                  // 2 ky sin(ky dy)
    const int p = blockIdx.x, c = blockIdx.y;
    const double dy = pts[3 * p + 1] - col_xy[2 * c + 1], z = pts[3 * p + 2];
    for (int m = threadIdx.x; m < hy; m += blockDim.x) {
        double sn, cs;
        sincospi(2.0 * m * dy / Ly, &sn, &cs);
        cy[m] = (m ? 2.0 : 1.0) * cs;
        sy[m] = 2.0 * (2.0 * kPi * m / Ly) * sn;
    }
    __syncthreads();
    const double* gc = G + 2 * ((size_t)p * n_ux + col_u[c]) * hy * nz;
    const double* gs = gc + (size_t)hy * nz;
    for (int mz = threadIdx.x; mz < nz; mz += blockDim.x) {
        double ax = 0.0, ay = 0.0, a0 = 0.0;
        for (int my = 0; my < hy; ++my) {
            const double tc = gc[(size_t)my * nz + mz], ts = gs[(size_t)my * nz + mz];
            ax = fma(cy[my], ts, ax);
            ay = fma(sy[my], tc, ay);
            a0 = fma(cy[my], tc, a0);
        }
        double sn, cs;
        sincospi((double)mz * z / Lz, &sn, &cs);
        const double w = pref * (mz ? 2.0 : 1.0) * cs, ws = pref * 2.0 * (kPi * mz / Lz) * sn;
        double* o = Lat + (((size_t)p * 3) * n_cols + c) * nz + mz;
        const size_t st = (size_t)n_cols * nz;
        o[0] = w * ax;
        o[st] = w * ay;
        o[2 * st] = ws * a0;
    }
}

// Points of one chunk (n_pts of them) at all times: out[t][p][a].  ux: the distinct column x, col_u[c]
// which of them is column c's; F, G, Lat: work buffers of 2 n_pts n_ux hx, 2 n_pts n_ux hy nz and
// 3 n_pts n_cols nz values.
void sample_points(cudaStream_t s, const double* pts, int n_pts, const double* col_xy, const double* ux,
                   const int* col_u, int n_cols, int n_ux, int Nx, int Ny, int Nz, double Lx, double Ly, double Lz,
                   double pref, const double* T, const double* Zc, int n_t, double* F, double* G, double* Lat,
                   double* out) {
    const int hx = Nx / 2, hy = Ny / 2;
    const size_t nf = (size_t)n_pts * n_ux * hx;
    sample_xfactor_kernel<<<(unsigned)((nf + 255) / 256), 256, 0, s>>>(pts, ux, n_pts, n_ux, hx, Lx, F);
    WT_LAUNCH("sample_xfactor");
    dgemm(s, false, false, 2 * n_pts * n_ux, hy * Nz, hx, 1.0, F, hx, T, hy * Nz, 0.0, G, hy * Nz);
    sample_lateral_kernel<<<dim3(n_pts, n_cols), 128, 2 * (size_t)hy * sizeof(double), s>>>(
        pts, col_xy, col_u, n_cols, n_ux, hy, Nz, Ly, Lz, pref, G, Lat);
    WT_LAUNCH("sample_lateral");
    dgemm(s, false, true, n_t, 3 * n_pts, n_cols * Nz, 1.0, Zc, n_cols * Nz, Lat, n_cols * Nz, 0.0, out, 3 * n_pts);
}

}  // namespace wt
