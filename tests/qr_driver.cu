// Column-pivoted QR of columns longer than a block's shared memory: prints the largest entry of R^T R - (M P)^T (M P)
// over the product of its columns' norms, and whether the diagonal of R falls.
#include "driver.cuh"

#include <cmath>
#include <random>
#include <vector>

using namespace wt;

int main() {
    int ns, nt;
    std::mt19937_64 rng(5);
    std::normal_distribution<double> g;
    while (std::scanf("%d %d", &ns, &nt) == 2) {
        std::vector<double> M((size_t)nt * ns), R((size_t)nt * nt);
        for (int j = 0; j < nt; ++j)
            for (int i = 0; i < ns; ++i) M[(size_t)j * ns + i] = g(rng) * std::pow(0.7, j) + (j ? 0.3 * M[(size_t)(j - 1) * ns + i] : 0.0);
        DBuf<double> dM, dR;
        DBuf<int> dp, err;
        const int zero = 0;
        err.upload(&zero, 1, 0);
        dM.upload(M.data(), M.size(), 0);
        dR.alloc(R.size());
        dp.alloc(nt);
        int steps;
        {
            CallMemory mem(err.p);
            steps = qrcp_r(0, dM.p, ns, nt, ns, dR.p, dp.p, err.p);
        }
        std::vector<int> p(nt);
        dR.download(R.data(), R.size(), 0);
        dp.download(p.data(), nt, 0);
        int e = 0;
        err.download(&e, 1, 0);
        if (cudaDeviceSynchronize() != cudaSuccess || e) { std::printf("failed\n"); return 1; }
        double worst = 0.0;
        bool falls = steps == nt;
        for (int i = 0; i < nt; ++i) {
            if (i) falls = falls && std::fabs(R[(size_t)i * nt + i]) <= std::fabs(R[(size_t)(i - 1) * nt + i - 1]) * (1 + 1e-12);
            for (int j = 0; j < nt; ++j) {
                long double s = 0, t = 0, ni = 0, nj = 0;
                for (int k = 0; k < nt; ++k) s += (long double)R[(size_t)k * nt + i] * R[(size_t)k * nt + j];
                for (int k = 0; k < ns; ++k) {
                    const long double x = M[(size_t)p[i] * ns + k], y = M[(size_t)p[j] * ns + k];
                    t += x * y;
                    ni += x * x;
                    nj += y * y;
                }
                worst = std::max(worst, (double)(std::fabs((double)(s - t)) / std::sqrt((double)(ni * nj))));
            }
        }
        std::printf("%.3g %d\n", worst, falls ? 1 : 0);
    }
    return 0;
}
