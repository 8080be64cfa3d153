// rsqrt_newton and rcp_newton against 1 / sqrt(x) and 1 / x: per function the largest relative error over 2^-53
// (against long double, for normal results), over every exponent and near its ends, and the count of special
// values whose result is another kind than CUDA's.
#include "../paper_2605_13987_gb300/csrc/coop.cuh"
#include "driver.cuh"

#include <cmath>
#include <limits>
#include <random>
#include <vector>

using namespace wt;

__global__ void apply(const double* x, int n, double* a, double* b, double* c, double* d) {
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    a[i] = rsqrt_newton(x[i]);
    b[i] = 1.0 / sqrt(x[i]);
    c[i] = rcp_newton(x[i]);
    d[i] = 1.0 / x[i];
}

int main() {
    std::mt19937_64 rng(11);
    std::uniform_real_distribution<double> u(1.0, 2.0);
    std::vector<double> x;
    for (int e = -1074; e <= 1023; ++e) {
        const double one = std::ldexp(1.0, e);
        for (double m : {1.0, 1.0 + 2.3e-16, 2.0 - 2.3e-16, 1.5, 4.0 / 3.0}) x.push_back(e < -1022 ? one : one * m);
        for (int k = 0; k < 100; ++k) x.push_back(e < -1022 ? one : one * u(rng));
    }
    const size_t n_pos = x.size();
    for (size_t k = 0; k < n_pos; k += 7) x.push_back(-x[k]);
    for (double s : {0.0, -0.0, (double)INFINITY, -(double)INFINITY, std::nan("")}) x.push_back(s);
    const int n = (int)x.size();
    DBuf<double> dx, r[4];
    dx.upload(x.data(), n, 0);
    std::vector<double> h[4];
    for (int k = 0; k < 4; ++k) { r[k].alloc(n); h[k].resize(n); }
    apply<<<(n + 255) / 256, 256>>>(dx.p, n, r[0].p, r[1].p, r[2].p, r[3].p);
    for (int k = 0; k < 4; ++k) r[k].download(h[k].data(), n, 0);
    if (cudaDeviceSynchronize() != cudaSuccess) { std::printf("failed\n"); return 1; }
    auto kind = [](double v) { return std::isnan(v) ? 3 : std::isinf(v) ? (v > 0 ? 1 : 2) : v == 0.0 ? 4 : 0; };
    double worst[2] = {0.0, 0.0};
    int kinds[2] = {0, 0};
    for (int i = 0; i < n; ++i)
        for (int f = 0; f < 2; ++f) {
            const double got = h[2 * f][i], ref = h[2 * f + 1][i];
            if (kind(got) != kind(ref)) { ++kinds[f]; continue; }
            if (kind(got) || std::fabs(ref) < std::numeric_limits<double>::min()) continue;
            const long double v = x[i], t = f ? 1.0L / v : 1.0L / sqrtl(v);
            worst[f] = std::max(worst[f], (double)(fabsl((got - t) / t) * 9007199254740992.0L));
        }
    std::printf("%.4f %d\n%.4f %d\n", worst[0], kinds[0], worst[1], kinds[1]);
    return 0;
}
