// The FP64 field from given tables: "n_cols nb" per line of standard input, on a 4 x 6 x 4 grid; prints the largest
// difference from long double sums over the sum of the terms' sizes.
#include "driver.cuh"

#include <cmath>
#include <random>
#include <vector>

namespace wt {
size_t t64_work(int, int, int, int);
void t64_fields(cudaStream_t, const double*, const double*, const double*, int, int, int, int, int, double*,
                unsigned char*, int*, double*);
}  // namespace wt
using namespace wt;

int main() {
    const int Nx = 4, Ny = 6, Nz = 4, nxy = Nx * Ny;
    int nc, nb;
    std::mt19937_64 rng(5);
    std::normal_distribution<double> g;
    while (std::scanf("%d %d", &nc, &nb) == 2) {
        std::vector<double> T((size_t)nc * 3 * Nz * nxy), Z((size_t)nb * nc * Nz), CS(2 * Nz * Nz), H((size_t)nb * 3 * nxy * Nz);
        for (double& x : T) x = g(rng);
        for (double& x : Z) x = g(rng);
        for (double& x : CS) x = g(rng);
        DBuf<double> dT, dZ, dCS, dR, dH;
        DBuf<unsigned char> ws;
        DBuf<int> err;
        const int zero = 0;
        err.upload(&zero, 1, 0);
        dT.upload(T.data(), T.size(), 0);
        dZ.upload(Z.data(), Z.size(), 0);
        dCS.upload(CS.data(), CS.size(), 0);
        dR.alloc((size_t)3 * Nz * nb * nxy);
        dH.alloc(H.size());
        ws.alloc(t64_work(nb, Nx, Ny, Nz));
        t64_fields(0, dT.p, dCS.p, dZ.p, nb, nc, Nx, Ny, Nz, dR.p, ws.p, err.p, dH.p);
        dH.download(H.data(), H.size(), 0);
        int e = 0;
        err.download(&e, 1, 0);
        if (cudaDeviceSynchronize() != cudaSuccess || e) { std::printf("failed\n"); return 1; }
        double worst = 0.0;
        for (int q = 0; q < 400; ++q) {
            const int t = rng() % nb, a = rng() % 3, xy = rng() % nxy, z = rng() % Nz;
            long double s = 0, size = 0;
            for (int k = 0; k < Nz; ++k) {
                long double r = 0;
                for (int c = 0; c < nc; ++c) {
                    const long double x = (long double)Z[((size_t)t * nc + c) * Nz + k] * T[(((size_t)c * 3 + a) * Nz + k) * nxy + xy];
                    r += x;
                    size += fabsl(x * CS[(a == 2 ? Nz * Nz : 0) + z * Nz + k]);
                }
                s += r * CS[(a == 2 ? Nz * Nz : 0) + z * Nz + k];
            }
            worst = std::max(worst, (double)(fabsl(H[((size_t)t * 3 + a) * nxy * Nz + (size_t)xy * Nz + z] - s) / size));
        }
        std::printf("%.3g\n", worst);
    }
    return 0;
}
