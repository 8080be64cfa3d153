// A call's pool gives back what nothing uses when another allocation needs it.  All but 1.5 GB of the device
// is held; a temporary of 1 GB is taken and given back, or a product's workspace is made, then a buffer of
// 1.2 GB is wanted: by itself, and as another temporary.  Prints "ok" per combination.
#include "driver.cuh"

#include <vector>

using namespace wt;

int main() {
    DBuf<int> err;
    const int zero = 0;
    err.upload(&zero, 1, 0);
    size_t fr = 0, tot = 0;
    WT_CUDA(cudaMemGetInfo(&fr, &tot));
    const size_t gb = (size_t)1 << 30, keep = 3 * gb / 2, big = gb + gb / 5;
    std::vector<void*> held;
    for (size_t want = fr - keep; want > 64u << 20;) {
        void* p = nullptr;
        const size_t n = std::min(want, 32 * gb);
        if (cudaMalloc(&p, n) != cudaSuccess) { cudaGetLastError(); break; }
        held.push_back(p);
        want -= n;
    }
    int rc = 0;
    for (int first = 0; first < 2; ++first)
        for (int then = 0; then < 2; ++then) {
            try {
                CallMemory mem(err.p);
                if (first == 0) {
                    TBuf<char> a;
                    a.alloc(gb);
                } else if (!mem.products(gb)) {
                    fail(WT_ERR_OOM, "workspace");
                }
                if (then == 0) {
                    DBuf<char> b;
                    b.alloc(big);
                } else {
                    TBuf<char> b;
                    b.alloc(big);
                }
                std::printf("ok\n");
            } catch (const Error& e) {
                std::printf("%d %d: %s\n", first, then, e.msg.c_str());
                rc = 0;
            }
        }
    for (void* p : held) cudaFree(p);
    return rc;
}
