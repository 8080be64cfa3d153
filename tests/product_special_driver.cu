// Products with infinities, NaN and subnormal entries: the tensor-core product against the FP64 kernel, entry
// by entry.  Prints, per layout, the entries whose kind (NaN, the sign of an infinity, finite) differs and the
// largest difference of finite entries over 2^-50 |a| |b| (norms of the row and the column).
#include "driver.cuh"

#include <cmath>
#include <random>
#include <vector>

using namespace wt;

int main() {
    const int M = 70, N = 90, K = 260;
    for (int form = 0; form < 4; ++form) {
        const bool ta = form & 1, tb = form & 2;
        std::mt19937_64 rng(3 + form);
        std::uniform_real_distribution<double> u(0.5, 1.5);
        const int lda = (ta ? M : K) + 1, ldb = (tb ? K : N) + 2;
        std::vector<double> A((size_t)(ta ? K : M) * lda), B((size_t)(tb ? N : K) * ldb), C0((size_t)M * N), C1, C2;
        auto a = [&](int i, int k) -> double& { return A[ta ? (size_t)k * lda + i : (size_t)i * lda + k]; };
        auto b = [&](int k, int j) -> double& { return B[tb ? (size_t)j * ldb + k : (size_t)k * ldb + j]; };
        for (int i = 0; i < M; ++i)
            for (int k = 0; k < K; ++k) a(i, k) = u(rng) * ((rng() & 1) ? 1 : -1);
        for (int k = 0; k < K; ++k)
            for (int j = 0; j < N; ++j) b(k, j) = u(rng) * ((rng() & 1) ? 1 : -1);
        for (double& x : C0) x = u(rng);
        a(3, 5) = INFINITY;                                  // signed infinities, zero x infinity, inf - inf
        b(5, 7) = 0.0;
        a(9, 11) = -INFINITY;
        a(9, 12) = -INFINITY;
        a(20, 100) = std::nan("");
        b(30, 4) = INFINITY;
        b(31, 6) = std::nan("");
        for (int k = 0; k < K; ++k) a(40, k) = 1e-310 * (k + 1);           // a subnormal row against large columns
        for (int k = 0; k < K; ++k) b(k, 50) *= 1e300;
        for (int k = 0; k < K; ++k) a(41, k) = k % 7 ? 1e-309 : 3e-308;    // subnormal entries among normal ones
        DBuf<double> dA, dB, dC;
        DBuf<int> err;
        const int zero = 0;
        err.upload(&zero, 1, 0);
        dA.upload(A.data(), A.size(), 0);
        dB.upload(B.data(), B.size(), 0);
        dC.upload(C0.data(), C0.size(), 0);
        C1.resize(C0.size());
        C2.resize(C0.size());
        bool taken;
        {
            CallMemory ws(err.p);
            taken = dgemm_tc(0, ta, tb, M, N, K, -1.0, dA.p, lda, dB.p, ldb, 1.0, dC.p, N, false);
        }
        dC.download(C1.data(), C1.size(), 0);
        dC.upload(C0.data(), C0.size(), 0);
        dgemm(0, ta, tb, M, N, K, -1.0, dA.p, lda, dB.p, ldb, 1.0, dC.p, N);      // no CallMemory: the FP64 kernel
        dC.download(C2.data(), C2.size(), 0);
        if (cudaDeviceSynchronize() != cudaSuccess || !taken) { std::printf("failed\n"); return 1; }
        int kinds = 0;
        double worst = 0.0;
        auto kind = [](double x) { return std::isnan(x) ? 3 : std::isinf(x) ? (x > 0 ? 1 : 2) : 0; };
        for (int i = 0; i < M; ++i)
            for (int j = 0; j < N; ++j) {
                const double x = C1[(size_t)i * N + j], y = C2[(size_t)i * N + j];
                if (kind(x) != kind(y)) { ++kinds; continue; }
                if (kind(x)) continue;
                double na = 0, nb = 0;
                for (int k = 0; k < K; ++k) { na = std::hypot(na, a(i, k)); nb = std::hypot(nb, b(k, j)); }
                worst = std::max(worst, std::fabs(x - y) / (std::ldexp(na * nb, -50) + std::ldexp(std::fabs(C0[(size_t)i * N + j]), -51)));
            }
        std::printf("%d %.3g\n", kinds, worst);
    }
    return 0;
}
