// One sweep of the one-sided Jacobi over two rows, a single rotation: prints what is left of their coupling
// (relative to their norms) over the rounding level of the dot product, for pairs of many ratios and angles.
#include "driver.cuh"

#include <cmath>
#include <random>
#include <vector>

using namespace wt;

int main() {
    const int n = 64;
    std::mt19937_64 rng(5);
    std::normal_distribution<double> g;
    std::uniform_real_distribution<double> u(0.0, 1.0);
    double worst = 0.0;
    for (int rep = 0; rep < 200; ++rep) {
        std::vector<double> A(2 * n);
        const double ratio = std::pow(10.0, -6.0 * u(rng)), mix = std::pow(10.0, -8.0 * u(rng)) * (rep % 2 ? 1 : -1);
        for (int k = 0; k < n; ++k) {
            A[k] = g(rng);
            A[n + k] = ratio * (mix * A[k] + g(rng));
        }
        DBuf<double> dA, sig;
        DBuf<int> err;
        const int zero = 0;
        err.upload(&zero, 1, 0);
        dA.upload(A.data(), A.size(), 0);
        sig.alloc(2);
        {
            CallMemory mem(err.p);
            onesided_jacobi_rows(0, dA.p, 2, n, n, nullptr, sig.p, err.p, 1);
        }
        dA.download(A.data(), A.size(), 0);
        if (cudaDeviceSynchronize() != cudaSuccess) { std::printf("failed\n"); return 1; }
        long double p = 0, q = 0, c = 0;
        for (int k = 0; k < n; ++k) {
            p += (long double)A[k] * A[k];
            q += (long double)A[n + k] * A[n + k];
            c += (long double)A[k] * A[n + k];
        }
        // the rotated entries round at the size of the larger row's part in them
        const double small = std::sqrt((double)std::min(p, q)), large = std::sqrt((double)std::max(p, q));
        worst = std::max(worst, std::fabs((double)c) / (small * large * 2.2e-16 * n + large * large * 2.2e-16 * 4));
    }
    std::printf("%.3g\n", worst);
    return 0;
}
