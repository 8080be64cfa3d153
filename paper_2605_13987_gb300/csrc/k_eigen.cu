// Symmetric eigendecomposition for the relaxation modes (the quasi-static
// relaxation of Sec. 3, solved exactly through its modes): FP64 throughout.
//
//   1. Householder tridiagonalisation Y = Q T Q^T, one reflector per column:
//      H_k = I - tau_k u_k u_k^T with u_k = [0 (k + 1 entries); v_k],
//      v_k[0] = 1.  Per step: the reflector, p = tau A22 v, w = p -
//      (tau p.v / 2) v, and the rank-two update A22 -= v w^T + w v^T, taken
//      with the next step's pass over A22.  v_k is kept in row k of A.
//   2. Divide and conquer on T (Cuppen's splitting): T = diag(T1', T2') +
//      |rho| s s^T with rho the coupling at the split, s = [e_last; sign(rho)
//      e_first] and T1', T2' the halves with |rho| taken off the touching
//      diagonal entries.  Leaves (<= 8 rows) by implicit QL with Wilkinson
//      shifts, one warp each.  A merge turns the halves' eigen-
//      decompositions into that of D + r z z^T (r = 2|rho|, |z| = 1):
//      deflation of negligible z entries and of close pairs of D (a Givens
//      rotation zeroes one z entry), the roots of the secular equation
//      1 + r sum_i z_i^2 / (d_i - lambda) = 0 (one warp per root, each root
//      held as the offset tau from its nearer pole so that every difference
//      d_i - lambda is formed without cancellation), the update vector
//      recomputed from the roots by Loewner's formula (Gu and Eisenstat), so
//      that the eigenvectors z^_i / (d_i - lambda_j) come out orthogonal to
//      working precision, and one GEMM per merge for the new eigenvectors.
//   3. Back-transformation V = H_0 H_1 ... H_{n-3} Z in blocks of 128
//      reflectors (compact WY form I - W T W^T, three GEMMs per block).
#include "coop.cuh"

#include <algorithm>
#include <cmath>
#include <vector>

namespace wt {

namespace {

// Largest leaf of the divide-and-conquer tree.  A leaf's QL iteration is a serial chain of about
// 2 K^2 rotations on one lane (32 rows: 0.9-2.4 ms); two more levels of merges cost less.
constexpr int kLeaf = 8;
constexpr int kWyBlock = 128;   // reflectors per back-transformation block (the products' K)
constexpr double kEps = 2.220446049250313e-16;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Block-wide sum (blockDim.x a multiple of 32); every thread gets the result.
__device__ double block_sum(double v, double* sh) {
    v = warp_sum(v);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    if (w == 0) {
        double t = l < (int)(blockDim.x >> 5) ? sh[l] : 0.0;
        t = warp_sum(t);
        if (l == 0) sh[32] = t;
    }
    __syncthreads();
    return sh[32];
}

// ------------------------------------------------------ tridiagonalisation
// All columns in one cooperative launch (one block per SM, rows dealt out cyclically).  Step k, with the
// vector u of step k - 1 (unscaled: H = 1 - t u u^T) and p = t A u in shared memory, A' = A - u p^T - c u^T,
// c = p - (t p.u) u:
//   every block forms row k of A' and the squares below its subdiagonal entry (the same work in every
//   block: 4 m operations, cheaper than a barrier);
//   four warps take a row i > k, a quarter of its entries each: A[i] = A'[i], and on the same pass
//   acc = A'[i] . A'[k].  A warp of its own meanwhile works out the reflector (beta, t); it enters
//   the product through its first entry only, u = A'[k] - beta e_{k+1}, so p_i = t (acc - beta A'[i][k+1]);
//   barrier; every block reads p.
// One barrier per column and one pass over the trailing block.  What bounds it: three FP64 operations per
// entry of the trailing block (2 per clock and SM: n^3 in all, 21 of the 43.5 ms at n = 2304; the four
// warps of a row sit on the four quarters of the SM, so that a few rows load them alike), and about six
// us a column of latency (barrier, loads, two sums).  Four launches a column: 94 ms at n = 2304; the same
// launch with normalised vectors, a warp per row: 46.7.
// p alternates between two buffers, so that a block still reading one is not overtaken.  The reflector of
// step k is written into row k one step later, when no block reads that row any more.
//
// The sums over vectors are taken by the first four warps only, one per SM quarter: a quarter does an FP64
// warp instruction in 64 cycles, so more warps add nothing to the sums and four times the shuffle steps
// to the reductions.
constexpr int kTrdThreads = 544, kTrdRowThreads = 512, kTrdVec = 128, kTrdRows = 64;
// sum over the first kTrdVec threads, for all threads of the block (red: 4 values)
__device__ __forceinline__ double trd_sum(double v, double* red) {
    if (threadIdx.x < kTrdVec) {
        v = warp_sum(v);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    }
    __syncthreads();
    return (red[0] + red[1]) + (red[2] + red[3]);
}
__global__ void __launch_bounds__(kTrdThreads, 1)
    trd_kernel(double* A, int n, double* __restrict__ d, double* __restrict__ e, double* __restrict__ tau_out,
               double* p, unsigned* bar, int* err) {
    extern __shared__ double sm[];
    double* u = sm;
    double* w = sm + n;                                  // p of the last step
    double* x = sm + 2 * (size_t)n;                      // row k, then the next u
    __shared__ double red[2][4];
    __shared__ double par[2];                            // t, scale of the last reflector
    __shared__ double part[kTrdRows][5];                 // per own row: sums of its quarters, entry k + 1
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nblk = gridDim.x, blk = blockIdx.x;
    const int vt = tid < kTrdVec ? tid : n;              // the vector threads' start
    for (int j = tid; j < n; j += kTrdThreads) { u[j] = 0.0; w[j] = 0.0; }
    if (tid == 0) { par[0] = 0.0; par[1] = 0.0; }
    double ref = 0.0;                                    // largest entry so far (scalar warp)
    __syncthreads();
    double al2 = 0.0;                                    // t (p . u) of the last step
    // p and row k of the last step's matrix into shared memory, then al2 (all threads; k: first index in use)
    auto take_p = [&](int k) {
        const double* pk = p + (size_t)((k - 1) & 1) * n;
        for (int j = k + tid; j < n; j += kTrdThreads) w[j] = __ldcg(pk + j);
    };
    auto sum_pu = [&](int k) {
        double sp = 0.0;
        for (int j = k + vt; j < n; j += kTrdVec) sp = fma(w[j], u[j], sp);
        al2 = par[0] * trd_sum(sp, red[0]);
    };
    for (int k = 0; k + 2 < n; ++k) {
        for (int j = k + tid; j < n; j += kTrdThreads) x[j] = __ldcg(A + (size_t)k * n + j);
        if (k > 0) take_p(k);
        __syncthreads();
        if (k > 0) sum_pu(k);
        const double scale = par[1];                     // of step k - 1
        {
            const double uk = u[k], ck = fma(-al2, uk, w[k]);
            double ss = 0.0;
            for (int j = k + vt; j < n; j += kTrdVec) {
                const double y = fma(-ck, u[j], fma(-uk, w[j], x[j]));
                x[j] = y;
                if (j >= k + 2) ss = fma(y, y, ss);
            }
            if (tid < kTrdVec) {
                ss = warp_sum(ss);
                if (lane == 0) red[1][warp] = ss;
            }
        }
        __syncthreads();
        const int first = k + 1 + ((blk - (k + 1)) % nblk + nblk) % nblk;
        double beta = 0.0;
        if (warp < kTrdRowThreads / 32) {
            // rows below k: quarter q of row first + r nblk
            const int q = warp & 3;
            for (int i = first + (warp >> 2) * nblk, r = warp >> 2; i < n; i += 4 * nblk, r += 4) {
                const double ui = u[i], ci = fma(-al2, ui, w[i]);
                double* row = A + (size_t)i * n;
                double acc = 0.0;
#pragma unroll 4
                for (int j = k + 1 + 32 * q + lane; j < n; j += 128) {
                    const double y = fma(-ci, u[j], fma(-ui, w[j], row[j]));
                    row[j] = y;
                    acc = fma(y, x[j], acc);
                    if (j == k + 1) part[r][4] = y;
                }
                acc = warp_sum(acc);
                if (lane == 0) part[r][q] = acc;
            }
            if (k > 0 && (k - 1) % nblk == blk)
                for (int j = k + tid; j < n; j += kTrdRowThreads)
                    A[(size_t)(k - 1) * n + j] = j == k ? 1.0 : u[j] * scale;
        } else if (lane == 0) {
            const double ss = (red[1][0] + red[1][1]) + (red[1][2] + red[1][3]), x0 = x[k + 1], dk = x[k];
            const double sq = fma(x0, x0, ss);
            double t = 0.0, sc = 0.0;
            beta = x0;
            // a row below 1e-100 of the entries so far couples nothing, and its square would leave the range
            if (ss > 0.0 && !(sq < 1e-200 * ref * ref)) {
                const double rq = rsqrt_newton(sq);
                beta = -copysign(sq * rq, x0);
                sc = rcp_newton(x0 - beta);
                t = fma(fabs(x0), rq, 1.0);                        // (beta - x0) / beta
            }
            ref = fmax(ref, fmax(fabs(dk), fabs(beta)));
            par[0] = t * sc * sc;
            par[1] = sc;
            red[0][0] = beta;
            if (blk == 0) {
                d[k] = dk;
                e[k] = beta;
                tau_out[k] = t;
            }
        }
        __syncthreads();
        beta = red[0][0];
        if (tid == kTrdRowThreads) x[k + 1] -= beta;               // the rows have been taken with row k itself
        const int i = first + tid * nblk;
        if (tid < kTrdRows && i < n)
            __stcg(p + (size_t)(k & 1) * n + i,
                   par[0] * fma(-beta, part[tid][4], (part[tid][0] + part[tid][1]) + (part[tid][2] + part[tid][3])));
        if (nblk > 1) {
            if (!grid_barrier(bar, k + 1, err)) return;
        } else {
            __syncthreads();
        }
        double* y = u;
        u = x;
        x = y;
    }
    // the last 2 x 2 block and the last reflector (its row was read before the last barrier)
    if (blk == 0) {
        if (n > 2) {
            take_p(n - 2);
            __syncthreads();
            sum_pu(n - 2);
            for (int j = n - 2 + tid; j < n; j += kTrdThreads)
                A[(size_t)(n - 3) * n + j] = j == n - 2 ? 1.0 : u[j] * par[1];
        }
        if (tid == 0) {
            const int a = n - 2, b = n - 1;
            auto at = [&](int i, int j) {
                return fma(-fma(-al2, u[i], w[i]), u[j], fma(-u[i], w[j], __ldcg(A + (size_t)i * n + j)));
            };
            if (n >= 2) {
                d[a] = at(a, a);
                e[a] = at(a, b);
                tau_out[a] = 0.0;
            }
            d[b] = at(b, b);
            e[b] = 0.0;
            tau_out[b] = 0.0;
        }
    }
}

// The same steps by four launches a column, for matrices whose three vectors do not fit shared memory:
// Reflector of step k from x = A[k][k+1 ..] (row k equals column k): H x = beta e_0.
__global__ void __launch_bounds__(1024) trd_house_kernel(double* A, int n, int k, double* vk, double* d, double* e,
                                                        double* tau) {
    __shared__ double sh[33];
    const int m = n - k - 1;
    double* row = A + (size_t)k * n + k + 1;
    double ss = 0.0;
    for (int i = 1 + threadIdx.x; i < m; i += blockDim.x) ss = fma(row[i], row[i], ss);
    ss = block_sum(ss, sh);
    const double x0 = row[0];
    double t = 0.0, beta = x0, scale = 0.0;
    if (ss > 0.0) {
        beta = -copysign(sqrt(fma(x0, x0, ss)), x0);
        t = (beta - x0) / beta;
        scale = 1.0 / (x0 - beta);
    }
    __syncthreads();                      // x0 read everywhere before row[0] is replaced
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        const double v = i == 0 ? 1.0 : row[i] * scale;
        vk[i] = v;
        row[i] = v;
    }
    if (threadIdx.x == 0) {
        d[k] = A[(size_t)k * n + k];
        e[k] = beta;
        tau[k] = t;
    }
}

// p = tau A22 v, one warp per row of the trailing block.
__global__ void __launch_bounds__(256) trd_symv_kernel(const double* __restrict__ A, int n, int k,
                                                      const double* __restrict__ v, const double* __restrict__ tau,
                                                      double* __restrict__ p) {
    const int m = n - k - 1;
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= m) return;
    const double* row = A + (size_t)(k + 1 + i) * n + k + 1;
    double acc = 0.0;
    for (int j = lane; j < m; j += 32) acc = fma(row[j], v[j], acc);
    acc = warp_sum(acc);
    if (lane == 0) p[i] = tau[k] * acc;
}

// w = p - (tau (p . v) / 2) v, in place on p (one block).
__global__ void __launch_bounds__(1024) trd_w_kernel(int n, int k, const double* __restrict__ v,
                                                    const double* __restrict__ tau, double* __restrict__ p) {
    __shared__ double sh[33];
    const int m = n - k - 1;
    double s = 0.0;
    for (int i = threadIdx.x; i < m; i += blockDim.x) s = fma(p[i], v[i], s);
    s = block_sum(s, sh);
    const double a = 0.5 * tau[k] * s;
    for (int i = threadIdx.x; i < m; i += blockDim.x) p[i] = fma(-a, v[i], p[i]);
}

// A22 -= v w^T + w v^T; four rows per block row.
__global__ void __launch_bounds__(256) trd_syr2_kernel(double* __restrict__ A, int n, int k,
                                                      const double* __restrict__ v, const double* __restrict__ w) {
    const int m = n - k - 1;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m) return;
    const double vj = v[j], wj = w[j];
    const int i1 = min(m, (int)blockIdx.y * 4 + 4);
    for (int i = blockIdx.y * 4; i < i1; ++i) {
        double* a = A + (size_t)(k + 1 + i) * n + k + 1 + j;
        const double t = __dadd_rn(__dmul_rn(v[i], wj), __dmul_rn(w[i], vj));
        *a = __dsub_rn(*a, t);
    }
}

__global__ void trd_tail_kernel(const double* A, int n, double* d, double* e, double* tau) {
    if (threadIdx.x) return;
    if (n >= 2) {
        d[n - 2] = A[(size_t)(n - 2) * n + n - 2];
        e[n - 2] = A[(size_t)(n - 2) * n + n - 1];
        tau[n - 2] = 0.0;
    }
    d[n - 1] = A[(size_t)(n - 1) * n + n - 1];
    e[n - 1] = 0.0;
    tau[n - 1] = 0.0;
}

// Small matrices (n <= kSmallTrd) in one block: the same four steps per column on a copy of A in
// shared memory (rows of pitch n), then A (reflectors in its rows), d, e, tau written back.
constexpr int kSmallTrd = 96;
__global__ void __launch_bounds__(1024) trd_small_kernel(double* A, int n, double* d, double* e, double* tau) {
    extern __shared__ double sm[];
    double* a = sm;                       // [n][n]
    double* v = a + (size_t)n * n;        // [n]
    double* p = v + n;                    // [n]
    __shared__ double red[33];
    __shared__ double par[3];             // tau, beta, scale
    for (int i = threadIdx.x; i < n * n; i += blockDim.x) a[i] = A[i];
    __syncthreads();
    for (int k = 0; k + 2 < n; ++k) {
        const int m = n - k - 1;
        double* row = a + (size_t)k * n + k + 1;
        double ss = 0.0;
        for (int i = 1 + threadIdx.x; i < m; i += blockDim.x) ss = fma(row[i], row[i], ss);
        ss = block_sum(ss, red);
        if (threadIdx.x == 0) {
            const double x0 = row[0];
            double t = 0.0, beta = x0, scale = 0.0;
            if (ss > 0.0) {
                beta = -copysign(sqrt(fma(x0, x0, ss)), x0);
                t = (beta - x0) / beta;
                scale = 1.0 / (x0 - beta);
            }
            par[0] = t;
            par[1] = beta;
            par[2] = scale;
            d[k] = a[(size_t)k * n + k];
            e[k] = beta;
            tau[k] = t;
        }
        __syncthreads();
        const double t = par[0], scale = par[2];
        for (int i = threadIdx.x; i < m; i += blockDim.x) {
            const double vi = i == 0 ? 1.0 : row[i] * scale;
            v[i] = vi;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < m; i += blockDim.x) row[i] = v[i];
        // p = tau A22 v, one thread per row
        for (int i = threadIdx.x; i < m; i += blockDim.x) {
            const double* r = a + (size_t)(k + 1 + i) * n + k + 1;
            double acc = 0.0;
            for (int j = 0; j < m; ++j) acc = fma(r[j], v[j], acc);
            p[i] = t * acc;
        }
        __syncthreads();
        double sv = 0.0;
        for (int i = threadIdx.x; i < m; i += blockDim.x) sv = fma(p[i], v[i], sv);
        sv = block_sum(sv, red);
        const double al = 0.5 * t * sv;
        for (int i = threadIdx.x; i < m; i += blockDim.x) p[i] = fma(-al, v[i], p[i]);
        __syncthreads();
        for (int idx = threadIdx.x; idx < m * m; idx += blockDim.x) {
            const int i = idx / m, j = idx % m;
            double* x = a + (size_t)(k + 1 + i) * n + k + 1 + j;
            *x = __dsub_rn(*x, __dadd_rn(__dmul_rn(v[i], p[j]), __dmul_rn(p[i], v[j])));
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        if (n >= 2) {
            d[n - 2] = a[(size_t)(n - 2) * n + n - 2];
            e[n - 2] = a[(size_t)(n - 2) * n + n - 1];
            tau[n - 2] = 0.0;
        }
        d[n - 1] = a[(size_t)(n - 1) * n + n - 1];
        e[n - 1] = 0.0;
        tau[n - 1] = 0.0;
    }
    for (int i = threadIdx.x; i < n * n; i += blockDim.x) A[i] = a[i];
}

// ------------------------------------------------------- divide and conquer
// Take |rho| off the diagonal entries on both sides of every split (one thread, in order).
__global__ void dc_split_kernel(double* d, const double* e, const int* splits, int n_splits) {
    if (threadIdx.x || blockIdx.x) return;
    for (int q = 0; q < n_splits; ++q) {
        const int s = splits[q];
        const double a = fabs(e[s - 1]);
        d[s - 1] -= a;
        d[s] -= a;
    }
}

// One warp per leaf: implicit QL with Wilkinson shifts (lane 0 runs the recurrence and records
// each sweep's rotations), all lanes rotate their rows of the leaf's eigenvector matrix.
// Output sorted ascending: lam[l0 + j], Q[(l0 + i) n + l0 + j].
__global__ void __launch_bounds__(128) dc_leaf_kernel(const double* __restrict__ d, const double* __restrict__ e,
                                                      const int* __restrict__ starts, int n_leaves, int n,
                                                      double* __restrict__ lam, double* __restrict__ Q, int* err) {
    __shared__ double Zs[4][32][kLeaf + 1];
    __shared__ double dd[4][kLeaf], ee[4][kLeaf], rc[4][kLeaf], rs[4][kLeaf];
    __shared__ int ctl[4][4];
    __shared__ int perm[4][kLeaf];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int leaf = blockIdx.x * 4 + w;
    if (leaf >= n_leaves) return;
    const int l0 = starts[leaf], K = starts[leaf + 1] - l0;
    double (*Z)[kLeaf + 1] = Zs[w];
    for (int j = 0; j < K; ++j) Z[lane][j] = (lane == j) ? 1.0 : 0.0;
    if (lane < K) {
        dd[w][lane] = d[l0 + lane];
        ee[w][lane] = lane < K - 1 ? e[l0 + lane] : 0.0;
    }
    __syncwarp();
    for (int l = 0; l < K; ++l) {
        int iter = 0;
        while (true) {
            if (lane == 0) {
                double* D = dd[w];
                double* E = ee[w];
                int m = l;
                for (; m < K - 1; ++m) {
                    const double s = fabs(D[m]) + fabs(D[m + 1]);
                    if (fabs(E[m]) <= kEps * s) break;
                }
                int lo = 0, hi = -1, done = (m == l);
                if (!done && ++iter > 60) {
                    atomicMax(err, (int)DERR_TIMEOUT);
                    done = 1;
                }
                if (!done) {
                    double g = (D[l + 1] - D[l]) / (2.0 * E[l]);
                    double r = hypot(g, 1.0);
                    g = D[m] - D[l] + E[l] / (g + copysign(r, g));
                    double s = 1.0, c = 1.0, p = 0.0;
                    int i = m - 1;
                    bool under = false;
                    for (; i >= l; --i) {
                        const double f = s * E[i], b = c * E[i];
                        r = hypot(f, g);
                        E[i + 1] = r;
                        if (r == 0.0) {
                            D[i + 1] -= p;
                            E[m] = 0.0;
                            under = true;
                            break;
                        }
                        s = f / r;
                        c = g / r;
                        g = D[i + 1] - p;
                        r = (D[i] - g) * s + 2.0 * c * b;
                        p = s * r;
                        D[i + 1] = g + p;
                        g = c * r - b;
                        rc[w][i] = c;
                        rs[w][i] = s;
                    }
                    if (!under) {
                        D[l] -= p;
                        E[l] = g;
                        E[m] = 0.0;
                    }
                    lo = under ? i + 1 : l;
                    hi = m - 1;
                }
                ctl[w][0] = done;
                ctl[w][1] = lo;
                ctl[w][2] = hi;
            }
            __syncwarp();
            const int done = ctl[w][0], lo = ctl[w][1], hi = ctl[w][2];
            if (done) break;
            if (lane < K)
                for (int i = hi; i >= lo; --i) {
                    const double c = rc[w][i], s = rs[w][i];
                    const double f = Z[lane][i + 1];
                    Z[lane][i + 1] = s * Z[lane][i] + c * f;
                    Z[lane][i] = c * Z[lane][i] - s * f;
                }
            __syncwarp();
        }
        __syncwarp();
    }
    if (lane == 0) {                      // ascending order (selection sort, K <= 32)
        for (int j = 0; j < K; ++j) perm[w][j] = j;
        for (int j = 0; j < K; ++j) {
            int b = j;
            for (int q = j + 1; q < K; ++q)
                if (dd[w][perm[w][q]] < dd[w][perm[w][b]]) b = q;
            const int t = perm[w][j];
            perm[w][j] = perm[w][b];
            perm[w][b] = t;
        }
    }
    __syncwarp();
    if (lane < K) {
        lam[l0 + lane] = dd[w][perm[w][lane]];
        for (int j = 0; j < K; ++j) Q[(size_t)(l0 + lane) * n + l0 + j] = Z[lane][perm[w][j]];
    }
}

// Per-merge scratch, all arrays indexed from the node's first row l.
struct DcWork {
    int* perm;        // sorted position -> index in the node (0 .. K-1)
    int* fcol;        // sorted position -> column of the gathered matrix ([non-deflated | deflated])
    int* rot_p;       // Givens rotations on gathered columns, in order
    int* rot_i;
    double* rot_c;
    double* rot_s;
    double* ds;       // sorted (and rotated) diagonal; deflated eigenvalues at their sorted positions
    double* delta;    // non-deflated poles (ascending), [Kp]
    double* zeta;     // their update vector entries
    int* org;         // root j: index of its pole of origin
    double* tau;      // root j: lambda_j - delta[org_j]
    double* zh;       // Loewner update vector
    double* root;     // lambda_j
    double* defl_val; // deflated eigenvalues in gathered-column order (column Kp + q)
    int* oper;        // final order: output column j <- gathered column oper[j]
    double* lam_out;
    int* node_kp;     // per node
    int* node_nrot;
    double* node_r;
};

struct DcNode {
    int l, mid, r;
};

// Exclusive prefix sum (or running maximum) over the block's per-thread values; blockDim.x = 1024.
__device__ __forceinline__ int block_scan(int v, bool maximum, int identity, int* sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x = maximum ? max(x, y) : x + y;
    }
    __syncthreads();
    if (lane == 31) sh[w] = x;
    __syncthreads();
    int base = identity;
    for (int q = 0; q < w; ++q) base = maximum ? max(base, sh[q]) : base + sh[q];
    const int up = __shfl_up_sync(0xffffffffu, x, 1);
    return lane == 0 ? base : (maximum ? max(base, up) : base + up);
}

// One block per merge node: the rank-one update vector, the merged order (each entry's rank by a
// binary search in the other half), deflation and the compaction of the non-deflated poles.  Two
// non-deflated neighbours are close when |x y (d_p - d_q)| <= tol (x^2 + y^2) (the coupling that the
// rotation would leave, without its square root); all pairs are looked at together, and only when one
// is close does thread 0 go through them in order, rotating.
constexpr int kPrepThreads = 1024;
__global__ void __launch_bounds__(kPrepThreads) dc_prep_kernel(const DcNode* __restrict__ nodes,
                                                               const double* __restrict__ e,
                                                               const double* __restrict__ lamA,
                                                               const double* __restrict__ QA, int n, DcWork W) {
    __shared__ int sh_i[32];
    __shared__ double sh_d[32];
    __shared__ int any_close, n_rot;
    const DcNode nd = nodes[blockIdx.x];
    const int l = nd.l, K = nd.r - nd.l, K1 = nd.mid - nd.l, tid = threadIdx.x;
    const double rho = e[nd.mid - 1];
    const double sg = rho < 0.0 ? -1.0 : 1.0;
    const double inv_sqrt2 = 0.70710678118654752440;
    const double r = 2.0 * fabs(rho);
    int* perm = W.perm + l;
    double* ds = W.ds + l;
    double* zs = W.zh + l;                 // update vector in merged order, until the Loewner pass overwrites it
    int* flag = W.oper + l;                // 1 = deflated (oper is written after the merge)
    const double* lam = lamA + l;
    if (tid == 0) { any_close = 0; n_rot = 0; }
    // a NaN has no rank: the positions that nobody takes then keep an index of the node
    for (int i = tid; i < K; i += kPrepThreads) {
        perm[i] = i;
        ds[i] = 0.0;
        zs[i] = 0.0;
    }
    __syncthreads();
    double dmax = 0.0;
    for (int i = tid; i < K; i += kPrepThreads) {
        const double x = lam[i];
        const bool a = i < K1;
        int lo = a ? K1 : 0, hi = a ? K : K1;
        const int base = lo;
        while (lo < hi) {                  // entries of the other half before x (ties: first half first)
            const int mid = (lo + hi) / 2;
            if (a ? lam[mid] < x : lam[mid] <= x) lo = mid + 1; else hi = mid;
        }
        const int q = (a ? i : i - K1) + (lo - base);
        perm[q] = i;
        ds[q] = x;
        zs[q] = inv_sqrt2 * (a ? QA[(size_t)(nd.mid - 1) * n + l + i] : sg * QA[(size_t)nd.mid * n + l + i]);
        dmax = fmax(dmax, fabs(x));
    }
    for (int o = 16; o; o >>= 1) dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    if ((tid & 31) == 0) sh_d[tid >> 5] = dmax;
    __syncthreads();
    for (int q = 0; q < kPrepThreads / 32; ++q) dmax = fmax(dmax, sh_d[q]);
    const double tol = 8.0 * kEps * fmax(dmax, r);
    // contiguous pieces of the merged order per thread from here on
    const int per = (K + kPrepThreads - 1) / kPrepThreads, q0 = min(K, tid * per), q1 = min(K, q0 + per);
    int last = -1;
    for (int q = q0; q < q1; ++q) {
        const int f = r * fabs(zs[q]) <= tol;
        flag[q] = f;
        if (!f) last = q;
    }
    int p = block_scan(last, true, -1, sh_i);       // last non-deflated entry before this piece
    __syncthreads();
    for (int q = q0; q < q1; ++q) {
        if (flag[q]) continue;
        if (p >= 0) {
            const double x = zs[p], y = zs[q];
            if (fabs(x * y * (ds[p] - ds[q])) <= tol * fma(x, x, y * y)) any_close = 1;
        }
        p = q;
    }
    __syncthreads();
    if (any_close && tid == 0) {
        int nrot = 0, pp = -1;
        for (int q = 0; q < K; ++q) {
            if (flag[q]) continue;
            if (pp >= 0) {
                const double x = zs[pp], y = zs[q], a = ds[pp], b = ds[q];
                if (fabs(x * y * (a - b)) <= tol * fma(x, x, y * y)) {
                    const double t = hypot(x, y);
                    const double c = y / t, s = x / t;
                    ds[pp] = c * c * a + s * s * b;
                    ds[q] = s * s * a + c * c * b;
                    zs[pp] = 0.0;
                    zs[q] = t;
                    flag[pp] = 1;
                    W.rot_p[l + nrot] = pp;
                    W.rot_i[l + nrot] = q;
                    W.rot_c[l + nrot] = c;
                    W.rot_s[l + nrot] = s;
                    ++nrot;
                }
            }
            pp = q;
        }
        n_rot = nrot;
    }
    __syncthreads();
    // compaction: non-deflated first (ascending), then deflated
    int live = 0;
    for (int q = q0; q < q1; ++q) live += !flag[q];
    int a = block_scan(live, false, 0, sh_i);
    __shared__ int kp_sh;
    if (tid == kPrepThreads - 1) kp_sh = a + live;
    __syncthreads();
    const int kp = kp_sh;
    for (int q = q0; q < q1; ++q) {
        if (!flag[q]) {
            W.delta[l + a] = ds[q];
            W.zeta[l + a] = zs[q];
            W.fcol[l + q] = a++;
        } else {
            const int b = q - a;           // deflated entries before this one
            W.defl_val[l + b] = ds[q];
            W.fcol[l + q] = kp + b;
        }
    }
    if (tid == 0) {
        W.node_kp[blockIdx.x] = kp;
        W.node_nrot[blockIdx.x] = n_rot;
        W.node_r[blockIdx.x] = r;
    }
}

// f(tau) = 1 + r sum_i zeta_i^2 / ((delta_i - delta_org) - tau), its derivative and the sum of its
// terms' sizes, summed by the 32 lanes of a warp (lane k takes the poles k, k + 32, ...).  The xor
// butterfly gives every lane the same bits, so the iteration that uses them stays uniform across the warp.
__device__ __forceinline__ void secular_f(const double* __restrict__ delta, const double* __restrict__ zeta, int kp,
                                          double dorg, double r, double tau, double* f, double* fp, double* size) {
    double s = 0.0, sp = 0.0, sa = 0.0;
    for (int i = threadIdx.x & 31; i < kp; i += 32) {
        const double q = rcp_newton((delta[i] - dorg) - tau);
        const double t = zeta[i] * zeta[i] * q;
        s += t;
        sa += fabs(t);
        sp = fma(t, q, sp);
    }
    s = warp_sum(s);
    sp = warp_sum(sp);
    sa = warp_sum(sa);
    *f = fma(r, s, 1.0);
    *fp = r * sp;
    *size = fma(r, sa, 1.0);
}

// The same in FP32 on differences taken in FP64 (their rounding is relative, so near poles keep their
// sign and size): two FP64 operations per pole instead of about fifteen.
__device__ __forceinline__ void secular_f32(const double* __restrict__ delta, const double* __restrict__ zeta, int kp,
                                            double dorg, double r, float tau, float* f, float* fp, float* size) {
    float s = 0.f, sp = 0.f, sa = 0.f;
    const float rf = (float)r;
    for (int i = threadIdx.x & 31; i < kp; i += 32) {
        const float q = __fdividef(1.f, (float)(delta[i] - dorg) - tau), z = (float)zeta[i];
        const float zq = z * z * rf * q;
        s += zq;
        sa += fabsf(zq);
        sp = fmaf(zq, q, sp);
    }
    for (int o = 16; o; o >>= 1) {
        sa += __shfl_xor_sync(0xffffffffu, sa, o);
        s += __shfl_xor_sync(0xffffffffu, s, o);
        sp += __shfl_xor_sync(0xffffffffu, sp, o);
    }
    *f = 1.f + s;
    *fp = sp;
    *size = 1.f + sa;
}

// Step of the secular iteration by R.-C. Li's fixed-weight rational interpolation (Solving secular
// equations stably and efficiently, 1993): the two poles next to the root keep their places, the one
// that tau is measured from its weight pw, and value and derivative of f are matched; a quadratic
// remains.  dj, dj1: distances to the poles left and right of the root (last root: to the last two
// poles).  Newton's step where that is not a step towards the root.
__device__ __forceinline__ double over(double a, double b) { return a * rcp_newton(b); }
__device__ __forceinline__ float over(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double root_of(double q) { return q > 0.0 ? q * rsqrt_newton(q) : 0.0; }
__device__ __forceinline__ float root_of(float q) { return sqrtf(q); }
template <class T>
__device__ __forceinline__ T secular_step(bool last, bool at_j, T f, T fp, T dj, T dj1, T pw) {
    const T c = last ? fabs(f - dj * (fp - pw) - dj1 * pw) : at_j ? f - dj1 * fp + pw : f - dj * fp - pw;
    const T a = (dj + dj1) * f - dj * dj1 * fp, b = dj * dj1 * f;
    const T sq = root_of(fabs(a * a - 4 * b * c));
    const T eta = last == (a >= 0) ? over(last ? a + sq : a - sq, 2 * c) : over(2 * b, last ? a - sq : a + sq);
    return f * eta < 0 ? eta : over(-f, fp);
}

// One warp per root (eight per block): bracket between the poles, steps kept inside the
// bracket, else bisection; stops when the bracket is at the rounding level of tau.  The first steps,
// to about 1e-5 of tau, run in FP32; they only choose where the FP64 iteration starts, whose bracket
// and stopping rules are its own.  Bound by the root that takes the most steps: with Newton's step,
// which crawls away from a pole, the last merge took 394 us at 127 roots and 3.48 ms at 2301; with the
// rational step 81 us and 0.73 ms.
__global__ void __launch_bounds__(256) dc_secular_kernel(const DcNode* __restrict__ nodes, DcWork W) {
    const DcNode nd = nodes[blockIdx.y];
    const int l = nd.l, kp = W.node_kp[blockIdx.y];
    const int j = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (j >= kp) return;                 // whole warps leave together
    const double r = W.node_r[blockIdx.y];
    const double* delta = W.delta + l;
    const double* zeta = W.zeta + l;
    int org;
    double lo, hi;
    if (j < kp - 1) {
        const double gap = delta[j + 1] - delta[j];
        double f, fp, size;
        secular_f(delta, zeta, kp, delta[j], r, 0.5 * gap, &f, &fp, &size);
        if (f > 0.0) { org = j; lo = 0.0; hi = 0.5 * gap; }
        else { org = j + 1; lo = -0.5 * gap; hi = 0.0; }
    } else {
        double zz = 0.0;
        for (int i = threadIdx.x & 31; i < kp; i += 32) zz = fma(zeta[i], zeta[i], zz);
        zz = warp_sum(zz);
        org = j;
        lo = 0.0;
        hi = r * zz;
    }
    const double dorg = delta[org];
    // the step's poles and weight, in units of g (the gap, or the last root's bracket)
    const bool last = j == kp - 1;
    const int jl = last ? max(0, j - 1) : j;
    const double pl = delta[jl] - dorg, pr = delta[min(jl + 1, kp - 1)] - dorg, g = last ? hi : pr - pl, ig = rcp_newton(g);
    const double pk = r * zeta[org] * zeta[org] * ig;
    double t = 0.5 * (lo + hi);
    {
        const float fpl = (float)(pl * ig), fpr = (float)(pr * ig), fg = (float)g, fig = (float)ig, fpk = (float)pk;
        float flo = (float)lo, fhi = (float)hi, x = (float)t;
        for (int it = 0; it < 24; ++it) {
            float f, fp, size;
            secular_f32(delta, zeta, kp, dorg, r, x, &f, &fp, &size);
            if (fabsf(f) <= 1e-6f * size) break;                   // FP32 rounding
            if (f > 0.f) fhi = x; else flo = x;
            const float dj = fpl - x * fig, dj1 = fpr - x * fig, dd = org == jl ? dj : dj1;
            float xn = kp > 1 ? x + fg * secular_step(last, org == jl, f, fp * fg, dj, dj1, __fdividef(fpk, dd * dd))
                              : x - f / fp;
            if (!(xn > flo && xn < fhi) || (fabsf(xn - x) > 0.5f * (fhi - flo) && it > 2)) xn = 0.5f * (flo + fhi);
            const bool close = fabsf(xn - x) <= 1e-5f * fabsf(x);
            x = xn;
            if (close || !isfinite(xn)) break;
        }
        if (isfinite(x) && (double)x > lo && (double)x < hi) t = (double)x;
    }
    for (int it = 0; it < 200; ++it) {
        double f, fp, size;
        secular_f(delta, zeta, kp, dorg, r, t, &f, &fp, &size);
        // f at its own rounding level (the sum of 32 lanes' partial sums): no step beyond this one is
        // more than noise, and Newton's would wander there until the bracket closed
        if (fabs(f) <= 2.0 * kEps * size) { lo = hi = t; break; }
        if (f > 0.0) hi = t; else lo = t;
        const double w = hi - lo;
        if (w <= 4.0 * kEps * fmax(fabs(lo), fabs(hi))) break;
        const double dj = (pl - t) * ig, dj1 = (pr - t) * ig, id = rcp_newton(org == jl ? dj : dj1);
        double tn = kp > 1 ? fma(g, secular_step(last, org == jl, f, fp * g, dj, dj1, pk * id * id), t)
                           : t - f / fp;
        if (!(tn > lo && tn < hi) || (fabs(tn - t) > 0.5 * w && it > 2)) tn = 0.5 * (lo + hi);
        // converged: the step is at the rounding level of tau (Newton may otherwise alternate
        // between neighbouring values until the iteration limit)
        if (fabs(tn - t) <= 2.0 * kEps * fabs(t)) { t = tn; break; }
        t = tn;
    }
    if ((threadIdx.x & 31) == 0) {
        W.org[l + j] = org;
        W.tau[l + j] = t;
        W.root[l + j] = dorg + t;
    }
}

// Loewner's formula: zh_i^2 = (lambda_last - delta_i) / r  prod_{j < i} (lambda_j - delta_i) / (delta_j - delta_i)
//                              prod_{i <= j < last} (lambda_j - delta_i) / (delta_{j+1} - delta_i)
// One warp per pole (eight per block): the lanes take the factors j, j + 32, ...
__global__ void __launch_bounds__(256) dc_loewner_kernel(const DcNode* __restrict__ nodes, DcWork W) {
    const DcNode nd = nodes[blockIdx.y];
    const int l = nd.l, kp = W.node_kp[blockIdx.y];
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= kp) return;
    const double r = W.node_r[blockIdx.y];
    const double* delta = W.delta + l;
    const int* org = W.org + l;
    const double* tau = W.tau + l;
    const double di = delta[i];
    double acc = lane == 0 ? ((delta[org[kp - 1]] - di) + tau[kp - 1]) / r : 1.0;
    for (int j = lane; j < kp - 1; j += 32) {
        const double num = (delta[org[j]] - di) + tau[j];
        const double den = j < i ? delta[j] - di : delta[j + 1] - di;
        acc *= num / den;
    }
    for (int o = 16; o; o >>= 1) acc *= __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) W.zh[l + i] = copysign(sqrt(fmax(acc, 0.0)), W.zeta[l + i]);
}

// Eigenvectors of D + r z z^T: column j = zh / (delta - lambda_j), normalised; written as rows of
// WT (WT[j][i]) for the GEMM.  One warp per root.
__global__ void __launch_bounds__(256) dc_vec_kernel(const DcNode* __restrict__ nodes, DcWork W, int n,
                                                     double* __restrict__ WT) {
    const DcNode nd = nodes[blockIdx.y];
    const int l = nd.l, kp = W.node_kp[blockIdx.y];
    const int j = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (j >= kp) return;
    const double* delta = W.delta + l;
    const double* zh = W.zh + l;
    const double dorg = delta[W.org[l + j]], t = W.tau[l + j];
    double* row = WT + (size_t)(l + j) * n + l;
    double ss = 0.0;
    for (int i = lane; i < kp; i += 32) {
        const double v = zh[i] / ((delta[i] - dorg) - t);
        row[i] = v;
        ss = fma(v, v, ss);
    }
    ss = warp_sum(ss);
    const double inv = 1.0 / sqrt(ss);
    for (int i = lane; i < kp; i += 32) row[i] *= inv;
}

// Gathered eigenvector matrix of the halves: G[row][fcol[q]] = QA[row][l + perm[q]], one warp per row.
__global__ void __launch_bounds__(256) dc_gather_kernel(const DcNode* __restrict__ nodes, DcWork W, int n,
                                                        const double* __restrict__ QA, double* __restrict__ G) {
    const DcNode nd = nodes[blockIdx.y];
    const int l = nd.l, K = nd.r - nd.l;
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row >= K) return;
    const double* src = QA + (size_t)(l + row) * n + l;
    double* dst = G + (size_t)(l + row) * n + l;
    for (int q = threadIdx.x & 31; q < K; q += 32) dst[W.fcol[l + q]] = src[W.perm[l + q]];
}

// The deflation rotations on the gathered columns, in order (few matrices have any).  One thread per row.
__global__ void __launch_bounds__(128) dc_rotate_kernel(const DcNode* __restrict__ nodes, DcWork W, int n,
                                                        double* __restrict__ G) {
    const DcNode nd = nodes[blockIdx.y];
    const int l = nd.l, K = nd.r - nd.l, nrot = W.node_nrot[blockIdx.y];
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    if (nrot == 0 || row >= K) return;
    double* dst = G + (size_t)(l + row) * n + l;
    for (int k = 0; k < nrot; ++k) {
        const int cp = W.fcol[l + W.rot_p[l + k]], ci = W.fcol[l + W.rot_i[l + k]];
        const double c = W.rot_c[l + k], s = W.rot_s[l + k];
        const double a = dst[cp], b = dst[ci];
        dst[cp] = c * a - s * b;
        dst[ci] = s * a + c * b;
    }
}

// New eigenvectors of the small nodes of a level in one launch: columns j < kp of X = G WT^T, the
// deflated ones copied.  32 x 32 tiles, grid (tiles, tiles, nodes), 2 x 2 outputs per thread.
constexpr int kMergeBatch = 256;        // largest node of the batched form
__global__ void __launch_bounds__(256) dc_merge_kernel(const DcNode* __restrict__ nodes, DcWork W, int n,
                                                       const double* __restrict__ G, const double* __restrict__ WT,
                                                       double* __restrict__ X) {
    const DcNode nd = nodes[blockIdx.z];
    const int l = nd.l, K = nd.r - nd.l, kp = W.node_kp[blockIdx.z];
    const int bm = blockIdx.y * 32, bn = blockIdx.x * 32;
    if (bm >= K || bn >= K) return;
    __shared__ double As[16][33], Bs[16][33];
    const size_t off = (size_t)l * n + l;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    double acc[2][2] = {};
    if (bn < kp)
        for (int k0 = 0; k0 < kp; k0 += 16) {
            for (int q = threadIdx.x; q < 512; q += 256) {
                const int m = q >> 4, k = q & 15;
                As[k][m] = (bm + m < K && k0 + k < kp) ? G[off + (size_t)(bm + m) * n + k0 + k] : 0.0;
                Bs[k][m] = (bn + m < kp && k0 + k < kp) ? WT[off + (size_t)(bn + m) * n + k0 + k] : 0.0;
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < 16; ++k)
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 2; ++j) acc[i][j] = fma(As[k][ty + 16 * i], Bs[k][tx + 16 * j], acc[i][j]);
            __syncthreads();
        }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int row = bm + ty + 16 * i, col = bn + tx + 16 * j;
            if (row >= K || col >= K) continue;
            const size_t at = off + (size_t)row * n + col;
            X[at] = col < kp ? acc[i][j] : G[at];
        }
}

// Final order of a node's eigenvalues: roots (ascending) merged with the deflated values, every entry
// by its rank.  One block per node.
__global__ void __launch_bounds__(kPrepThreads) dc_order_kernel(const DcNode* __restrict__ nodes, DcWork W) {
    const DcNode nd = nodes[blockIdx.x];
    const int l = nd.l, K = nd.r - nd.l, kp = W.node_kp[blockIdx.x];
    const int nd_ = K - kp;
    const double* dv = W.defl_val + l;
    const double* root = W.root + l;
    double* sorted = W.delta + l;          // the poles are not needed any more
    int* idx = W.perm + l;
    for (int q = threadIdx.x; q < nd_; q += kPrepThreads) {      // for the ranks that a NaN leaves open
        idx[q] = q;
        sorted[q] = 0.0;
    }
    for (int q = threadIdx.x; q < K; q += kPrepThreads) {
        W.oper[l + q] = q;
        W.lam_out[l + q] = 0.0;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < nd_; q += kPrepThreads) {
        const double x = dv[q];
        int rank = 0;
        for (int p = 0; p < nd_; ++p) rank += dv[p] < x || (dv[p] == x && p < q);
        sorted[rank] = x;
        idx[rank] = q;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < K; q += kPrepThreads) {
        const bool is_root = q < kp;
        const double x = is_root ? root[q] : sorted[q - kp];
        const double* other = is_root ? sorted : root;
        int lo = 0, hi = is_root ? nd_ : kp;
        while (lo < hi) {                  // ties: roots first
            const int mid = (lo + hi) / 2;
            if (is_root ? other[mid] < x : other[mid] <= x) lo = mid + 1; else hi = mid;
        }
        const int o = (is_root ? q : q - kp) + lo;
        W.lam_out[l + o] = x;
        W.oper[l + o] = is_root ? q : kp + idx[q - kp];
    }
}

// QB[row][l + j] = X[row][l + oper[j]], one thread per (row, column chunk).
__global__ void __launch_bounds__(256) dc_permute_kernel(const DcNode* __restrict__ nodes, DcWork W, int n,
                                                         const double* __restrict__ X, double* __restrict__ QB,
                                                         double* __restrict__ lamB) {
    const DcNode nd = nodes[blockIdx.z];
    const int l = nd.l, K = nd.r - nd.l;
    const int j = blockIdx.x * blockDim.x + threadIdx.x, row = blockIdx.y;
    if (j >= K || row >= K) return;
    QB[(size_t)(l + row) * n + l + j] = X[(size_t)(l + row) * n + l + W.oper[l + j]];
    if (row == 0) lamB[l + j] = W.lam_out[l + j];
}

// ------------------------------------------------------- back-transformation
// Rows k of Wt (nref x n): u_k (zeros up to column k, then v_k from row k of A).
__global__ void wy_rows_kernel(const double* __restrict__ A, int n, int nref, double* __restrict__ Wt) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (c >= n || k >= nref) return;
    Wt[(size_t)k * n + c] = c <= k ? 0.0 : A[(size_t)k * n + c];
}

// T (upper triangular, pitch kWyBlock) of H_{k0} ... H_{k0+nb-1} = I - W T W^T from S = Wt Wt^T:
// T[j][j] = tau_j, T[0:j, j] = -tau_j T[0:j, 0:j] S[0:j, j].  One block per group of reflectors (all
// groups in one launch), thread i holds row i of T in shared memory; four partial sums per entry.
__global__ void __launch_bounds__(kWyBlock) wy_t_kernel(const double* __restrict__ S_all, const double* __restrict__ tau,
                                                        int nref, double* __restrict__ T_all) {
    extern __shared__ double t[];                         // [kWyBlock][kWyBlock + 1]
    __shared__ double sj[kWyBlock];
    constexpr int P = kWyBlock + 1;
    const int k0 = blockIdx.x * kWyBlock, nb = min(kWyBlock, nref - k0), i = threadIdx.x;
    const double* S = S_all + (size_t)blockIdx.x * kWyBlock * kWyBlock;
    double* T = T_all + (size_t)blockIdx.x * kWyBlock * kWyBlock;
    for (int j = 0; j < nb; ++j) {
        const double tj = tau[k0 + j];
        __syncthreads();
        if (i < j) sj[i] = S[(size_t)i * kWyBlock + j];
        __syncthreads();
        double a[4] = {0.0, 0.0, 0.0, 0.0};
        if (i < j) {
            int q = i;
            for (; q + 3 < j; q += 4)
#pragma unroll
                for (int u = 0; u < 4; ++u) a[u] = fma(t[i * P + q + u], sj[q + u], a[u]);
            for (; q < j; ++q) a[0] = fma(t[i * P + q], sj[q], a[0]);
        }
        if (i < nb) t[i * P + j] = i < j ? -tj * ((a[0] + a[1]) + (a[2] + a[3])) : (i == j ? tj : 0.0);
    }
    __syncthreads();
    for (int j = 0; j < nb; ++j)
        if (i < nb) T[(size_t)j * kWyBlock + i] = t[j * P + i];
}

}  // namespace

// Eigendecomposition of the symmetric A (n x n row-major, destroyed): w ascending, V columns.
void sym_eig(cudaStream_t s, double* A, int n, double* w, double* V, int* d_err) {
    if (n <= 0) return;
    TBuf<double> d, e, tau, vk, p;
    TBuf<unsigned> bar;
    d.alloc(n);
    e.alloc(n);
    tau.alloc(n);
    vk.alloc(n);
    p.alloc(n);
    // 1. tridiagonalisation (small matrices in one block)
    if (n <= kSmallTrd) {
        const size_t sh = ((size_t)n * n + 2 * (size_t)n) * sizeof(double);
        allow_dyn_smem(trd_small_kernel, sh);
        trd_small_kernel<<<1, 1024, sh, s>>>(A, n, d.p, e.p, tau.p);
    } else {
        int dev = 0, n_sm = 0, optin = 0;
        WT_CUDA(cudaGetDevice(&dev));
        WT_CUDA(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev));
        WT_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
        const size_t sh = 3 * (size_t)n * sizeof(double);
        // about one row per warp: more blocks than that only lengthen the barrier
        int blocks = std::max(1, std::min(n_sm, (n + 7) / 8)), nn = n;
        if (sh + 4096 <= (size_t)optin && (n + blocks - 1) / blocks <= kTrdRows) {
            allow_dyn_smem(trd_kernel, sh);
            bar.alloc(kBarrierWords);
            bar.zero(s);
            p.alloc(2 * (size_t)n);
            void* args[] = {&A, &nn, &d.p, &e.p, &tau.p, &p.p, &bar.p, &d_err};
            WT_CUDA(cudaLaunchCooperativeKernel((const void*)trd_kernel, dim3(blocks), dim3(kTrdThreads), args, sh, s));
        } else {
            for (int k = 0; k + 2 < n; ++k) {
                const int m = n - k - 1;
                trd_house_kernel<<<1, 1024, 0, s>>>(A, n, k, vk.p, d.p, e.p, tau.p);
                trd_symv_kernel<<<(m + 7) / 8, 256, 0, s>>>(A, n, k, vk.p, tau.p, p.p);
                trd_w_kernel<<<1, 1024, 0, s>>>(n, k, vk.p, tau.p, p.p);
                trd_syr2_kernel<<<dim3((m + 255) / 256, (m + 3) / 4), 256, 0, s>>>(A, n, k, vk.p, p.p);
            }
            trd_tail_kernel<<<1, 32, 0, s>>>(A, n, d.p, e.p, tau.p);
        }
    }
    WT_LAUNCH("tridiagonalisation");
    vk.release();

    // 2. divide and conquer: tree by halving
    std::vector<int> leaves;            // starts, plus n
    std::vector<std::vector<DcNode>> levels;
    std::vector<int> splits;
    struct Item { int l, r, depth; };
    std::vector<Item> stack{{0, n, 0}};
    // every node is split down to the same depth (sizes of a level differ by one at most), so every
    // level merges all rows
    int depth = 0;
    while (((n - 1) >> depth) + 1 > kLeaf) ++depth;
    while (!stack.empty()) {
        const Item it = stack.back();
        stack.pop_back();
        if (it.depth == depth) {
            leaves.push_back(it.l);
            continue;
        }
        const int mid = it.l + (it.r - it.l) / 2;
        if ((int)levels.size() <= it.depth) levels.resize(it.depth + 1);
        levels[it.depth].push_back({it.l, mid, it.r});
        splits.push_back(mid);
        stack.push_back({it.l, mid, it.depth + 1});
        stack.push_back({mid, it.r, it.depth + 1});
    }
    std::sort(leaves.begin(), leaves.end());
    const int n_leaves = (int)leaves.size();
    leaves.push_back(n);
    TBuf<double> lamA, lamB, QA, QB, G;
    lamA.alloc(n);
    lamB.alloc(n);
    QA.alloc((size_t)n * n);
    QA.zero(s);
    if (!splits.empty()) {
        TBuf<int> dsp;
        dsp.upload(splits.data(), splits.size(), s);
        dc_split_kernel<<<1, 32, 0, s>>>(d.p, e.p, dsp.p, (int)splits.size());
        WT_LAUNCH("dc_split");
    }
    {
        TBuf<int> dst;
        dst.upload(leaves.data(), leaves.size(), s);
        dc_leaf_kernel<<<(n_leaves + 3) / 4, 128, 0, s>>>(d.p, e.p, dst.p, n_leaves, n, lamA.p, QA.p, d_err);
        WT_LAUNCH("dc_leaf");
    }
    if (!levels.empty()) {
        QB.alloc((size_t)n * n);
        G.alloc((size_t)n * n);
        QB.zero(s);
        TBuf<int> ibuf;
        TBuf<double> fbuf;
        ibuf.alloc((size_t)n * 8);
        fbuf.alloc((size_t)n * 12);
        TBuf<double> WT;
        WT.alloc((size_t)n * n);
        const size_t nn = n;
        DcWork Wk{};
        Wk.perm = ibuf.p;
        Wk.fcol = ibuf.p + nn;
        Wk.rot_p = ibuf.p + 2 * nn;
        Wk.rot_i = ibuf.p + 3 * nn;
        Wk.org = ibuf.p + 4 * nn;
        Wk.oper = ibuf.p + 5 * nn;
        Wk.node_kp = ibuf.p + 6 * nn;
        Wk.node_nrot = ibuf.p + 7 * nn;
        Wk.rot_c = fbuf.p;
        Wk.rot_s = fbuf.p + nn;
        Wk.ds = fbuf.p + 2 * nn;
        Wk.delta = fbuf.p + 3 * nn;
        Wk.zeta = fbuf.p + 4 * nn;
        Wk.tau = fbuf.p + 5 * nn;
        Wk.zh = fbuf.p + 6 * nn;
        Wk.root = fbuf.p + 7 * nn;
        Wk.defl_val = fbuf.p + 8 * nn;
        Wk.lam_out = fbuf.p + 9 * nn;
        Wk.node_r = fbuf.p + 10 * nn;
        TBuf<DcNode> dnodes;
        std::vector<DcNode> all;
        std::vector<size_t> level_at;
        for (const auto& nodes : levels) {
            level_at.push_back(all.size());
            all.insert(all.end(), nodes.begin(), nodes.end());
        }
        dnodes.upload(all.data(), all.size(), s);
        double *qa = QA.p, *qb = QB.p, *la = lamA.p, *lb = lamB.p;
        for (int lev = (int)levels.size() - 1; lev >= 0; --lev) {
            const std::vector<DcNode>& nodes = levels[lev];
            const int nn_ = (int)nodes.size();
            const DcNode* dn = dnodes.p + level_at[lev];
            int kmax = 0;
            for (const DcNode& nd : nodes) kmax = std::max(kmax, nd.r - nd.l);
            dc_prep_kernel<<<nn_, kPrepThreads, 0, s>>>(dn, e.p, la, qa, n, Wk);
            WT_LAUNCH("dc_prep");
            dc_secular_kernel<<<dim3((kmax + 7) / 8, nn_), 256, 0, s>>>(dn, Wk);
            WT_LAUNCH("dc_secular");
            dc_loewner_kernel<<<dim3((kmax + 7) / 8, nn_), 256, 0, s>>>(dn, Wk);
            WT_LAUNCH("dc_loewner");
            dc_vec_kernel<<<dim3((kmax + 7) / 8, nn_), 256, 0, s>>>(dn, Wk, n, WT.p);
            WT_LAUNCH("dc_vec");
            dc_gather_kernel<<<dim3((kmax + 7) / 8, nn_), 256, 0, s>>>(dn, Wk, n, qa, G.p);
            dc_rotate_kernel<<<dim3((kmax + 127) / 128, nn_), 128, 0, s>>>(dn, Wk, n, G.p);
            WT_LAUNCH("dc_gather");
            if (kmax <= kMergeBatch) {
                const int tiles = (kmax + 31) / 32;
                dc_merge_kernel<<<dim3(tiles, tiles, nn_), 256, 0, s>>>(dn, Wk, n, G.p, WT.p, qa);
                WT_LAUNCH("dc_merge");
            } else {
                std::vector<int> kp(nn_);
                WT_CUDA(cudaMemcpyAsync(kp.data(), Wk.node_kp, nn_ * sizeof(int), cudaMemcpyDeviceToHost, s));
                WT_CUDA(cudaStreamSynchronize(s));
                for (int q = 0; q < nn_; ++q) {
                    const DcNode& nd = nodes[q];
                    const int K = nd.r - nd.l, k1 = kp[q];
                    const size_t off = (size_t)nd.l * n + nd.l;
                    if (k1 > 0) dgemm(s, false, true, K, k1, k1, 1.0, G.p + off, n, WT.p + off, n, 0.0, qa + off, n);
                    if (K > k1) copy_block(s, G.p + off + k1, n, qa + off + k1, n, K, K - k1);
                }
            }
            dc_order_kernel<<<nn_, kPrepThreads, 0, s>>>(dn, Wk);
            WT_LAUNCH("dc_order");
            dc_permute_kernel<<<dim3((kmax + 255) / 256, kmax, nn_), 256, 0, s>>>(dn, Wk, n, qa, qb, lb);
            WT_LAUNCH("dc_permute");
            std::swap(qa, qb);
            std::swap(la, lb);
        }
        if (qa != QA.p) {
            copy_block(s, qa, n, QA.p, n, n, n);
            WT_CUDA(cudaMemcpyAsync(lamA.p, la, n * sizeof(double), cudaMemcpyDeviceToDevice, s));
        }
    }
    WT_CUDA(cudaMemcpyAsync(w, lamA.p, n * sizeof(double), cudaMemcpyDeviceToDevice, s));
    QB.release();
    G.release();

    // 3. back-transformation: V = H_0 ... H_{n-3} Z, blocks of reflectors from the last one down
    double* Z = QA.p;
    const int nref = std::max(0, n - 2);
    if (nref > 0) {
        TBuf<double> Wt, S, T, Y, Y2;
        const int nblk = (nref + kWyBlock - 1) / kWyBlock;
        constexpr size_t tt = (size_t)kWyBlock * kWyBlock;
        Wt.alloc((size_t)nref * n);
        S.alloc(nblk * tt);
        T.alloc(nblk * tt);
        Y.alloc((size_t)kWyBlock * n);
        Y2.alloc((size_t)kWyBlock * n);
        wy_rows_kernel<<<dim3((n + 255) / 256, nref), 256, 0, s>>>(A, n, nref, Wt.p);
        WT_LAUNCH("wy_rows");
        for (int bi = 0; bi < nblk; ++bi) {
            const int k0 = bi * kWyBlock, nb = std::min(kWyBlock, nref - k0), m = n - k0 - 1;
            const double* W0 = Wt.p + (size_t)k0 * n + k0 + 1;
            dgemm(s, false, true, nb, nb, m, 1.0, W0, n, W0, n, 0.0, S.p + bi * tt, kWyBlock);
        }
        const size_t sh = (size_t)kWyBlock * (kWyBlock + 1) * sizeof(double);
        allow_dyn_smem(wy_t_kernel, sh);
        wy_t_kernel<<<nblk, kWyBlock, sh, s>>>(S.p, tau.p, nref, T.p);
        WT_LAUNCH("wy_t");
        for (int bi = nblk - 1; bi >= 0; --bi) {
            const int k0 = bi * kWyBlock, nb = std::min(kWyBlock, nref - k0);
            const int m = n - k0 - 1;           // rows k0 + 1 .. n - 1
            const double* W0 = Wt.p + (size_t)k0 * n + k0 + 1;
            dgemm(s, false, false, nb, n, m, 1.0, W0, n, Z + (size_t)(k0 + 1) * n, n, 0.0, Y.p, n);
            dgemm(s, false, false, nb, n, nb, 1.0, T.p + bi * tt, kWyBlock, Y.p, n, 0.0, Y2.p, n);
            dgemm(s, true, false, m, n, nb, -1.0, W0, n, Y2.p, n, 1.0, Z + (size_t)(k0 + 1) * n, n);
        }
    }
    copy_block(s, Z, n, V, n, n, n);
    WT_CUDA(cudaStreamSynchronize(s));
}

}  // namespace wt
