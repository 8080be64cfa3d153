// Test driver of the FP64 products (linked with the library's objects): one product per line of
// standard input, "ta tb M N K lower same special", checked on sampled entries (all of them up to
// 4096) against long double sums.  Prints "worst/bound untouched err" per line: the largest error
// over its bound, whether entries that must not change did not, and the device error word.
#include "../paper_2605_13987_gb300/csrc/wt_internal.cuh"

#include <algorithm>
#include <cmath>
#include <random>
#include <vector>

namespace wt {
void fail(wt_status c, const std::string& m) { throw Error{c, m}; }
void cuda_check(cudaError_t e, const char* w) {
    if (e != cudaSuccess) fail(WT_ERR_CUDA, std::string(w) + ": " + cudaGetErrorString(e));
}
}  // namespace wt
using namespace wt;

int main() {
    int ta, tb, M, N, K, lower, same, special;
    std::mt19937_64 rng(7);
    std::uniform_real_distribution<double> u(-1.0, 1.0);
    while (std::scanf("%d %d %d %d %d %d %d %d", &ta, &tb, &M, &N, &K, &lower, &same, &special) == 8) {
        const int ac = (ta ? M : K) + 3, bc = same ? ac : (tb ? K : N) + 5, ldc = N + 7;
        std::vector<double> A((size_t)(ta ? K : M) * ac), B((size_t)(tb ? N : K) * bc), C((size_t)M * ldc);
        for (double& x : A) x = u(rng) * std::exp(4.0 * u(rng));
        for (double& x : B) x = u(rng) * std::exp(4.0 * u(rng));
        for (double& x : C) x = u(rng);
        if (same) B = A;
        auto a = [&](int i, int k) -> double& { return A[ta ? (size_t)k * ac + i : (size_t)i * ac + k]; };
        auto b = [&](int k, int j) -> double& { return B[tb ? (size_t)j * bc + k : (size_t)k * bc + j]; };
        if (special) {                       // a zero row, tiny and huge rows, an infinity, one dominant entry
            for (int k = 0; k < K; ++k) { a(0, k) = 0.0; a(1, k) *= 1e-200; a(2, k) *= 1e150; b(k, 1) *= 1e-140; }
            a(3, K / 2) = INFINITY;
            a(4, K - 1) = 1e12;
        }
        DBuf<double> dA, dB, dC;
        DBuf<int> err;
        const int zero = 0;
        err.upload(&zero, 1, 0);
        dA.upload(A.data(), A.size(), 0);
        dB.upload(B.data(), B.size(), 0);
        dC.upload(C.data(), C.size(), 0);
        std::vector<double> R(C.size());
        bool taken;
        {
            CallMemory ws(err.p);
            taken = dgemm_tc(0, ta, tb, M, N, K, -1.0, dA.p, ac, same ? dA.p : dB.p, bc, 1.0, dC.p, ldc, lower);
        }
        dC.download(R.data(), R.size(), 0);
        int e = 0;
        err.download(&e, 1, 0);
        if (cudaDeviceSynchronize() != cudaSuccess || !taken) { std::printf("failed\n"); return 1; }
        double worst = 0.0;
        bool untouched = true;
        const bool all = (size_t)M * N <= 4096;
        for (int q = 0; q < (all ? M * N : 4096); ++q) {
            const int i = all ? q / N : (q < 64 ? M - 1 - q % std::min(M, 8) : (int)(rng() % M));
            const int j = all ? q % N : (q < 64 ? N - 1 - q / 8 % std::min(N, 8) : (int)(rng() % N));
            const double c0 = C[(size_t)i * ldc + j], got = R[(size_t)i * ldc + j];
            if (lower && j > i) { untouched = untouched && got == c0; continue; }
            long double s = 0, na = 0, nb = 0;
            for (int k = 0; k < K; ++k) {
                const long double x = a(i, k), y = b(k, j);
                s += x * y;
                na += x * x;
                nb += y * y;
            }
            if (special && i == 3) { if (std::isfinite(got)) worst = INFINITY; continue; }
            // rounding to integers of norm 2^58: at most half a unit per entry on either side; then the
            // conversion, the product by the scale and the addition to C round once each
            const long double bound = sqrtl(na * nb) * sqrtl((long double)K) * ldexpl(1.0L, -57) +
                                      4.0L * ldexpl(1.0L, -53) * (fabsl(s) + fabsl((long double)c0));
            worst = std::max(worst, (double)(fabsl((long double)got - (c0 - s)) / bound));
        }
        for (int i = 0; i < M; ++i)
            for (int j = N; j < ldc; ++j) untouched = untouched && R[(size_t)i * ldc + j] == C[(size_t)i * ldc + j];
        std::printf("%.6g %d %d\n", worst, untouched ? 1 : 0, e);
        std::fflush(stdout);
    }
    return 0;
}
