// Shared-memory barrier, TMA, tensor-memory and tcgen05 helpers of the tensor-core kernels
// (k_expand_tc.cu, k_dgemm_tc.cu).  Every wait is bounded.
#pragma once

#include "wt_internal.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>

namespace wt {

// cuTensorMapEncodeTiled through the runtime's driver entry point (k_expand_tc.cu)
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder();

namespace tc {

constexpr unsigned long long TIMEOUT_NS = 2000000000ull;

__device__ __forceinline__ unsigned smem_u32(const void* p) {
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ unsigned long long globaltimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mbar_init(unsigned long long* b, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* b) {
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned long long* b, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(b)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: false on timeout (and the abort flag is raised).
// Every caller is a whole warp: the lanes vote, so that a warp either proceeds or unwinds as
// one (a lane that saw the phase complete while another saw the abort flag takes the abort),
// and no warp-collective instruction after the wait sees a divided warp.
__device__ __forceinline__ bool mbar_wait(unsigned long long* b, unsigned parity, volatile int* abort_flag,
                                          int* d_err) {
    bool ok = mbar_try(b, parity);
    if (!ok) {
        const unsigned long long t0 = globaltimer();
        while (true) {
            if (mbar_try(b, parity)) { ok = true; break; }
            if (*abort_flag) break;
            if (globaltimer() - t0 > TIMEOUT_NS) {
                *abort_flag = 1;
                atomicMax(d_err, (int)DERR_TIMEOUT);
                break;
            }
        }
    }
    return __all_sync(0xffffffffu, ok);
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* b, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
// 2D tiled TMA load into shared memory, completion signalled on an mbarrier
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* tm, int x, int y, unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_u32(dst)),
        "l"(tm), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}
// Drain wait used while unwinding: ignores the abort flag, still bounded in time.
__device__ __forceinline__ bool mbar_wait_drain(unsigned long long* b, unsigned parity, int* d_err) {
    const unsigned long long t0 = globaltimer();
    while (!mbar_try(b, parity)) {
        if (globaltimer() - t0 > TIMEOUT_NS) {
            atomicMax(d_err, (int)DERR_TIMEOUT);
            return false;
        }
    }
    return true;
}
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 B apart
__device__ __forceinline__ unsigned long long sdesc(unsigned addr) {
    return (unsigned long long)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | (64ull << 32) | (1ull << 46) |
           (2ull << 61);
}
__device__ __forceinline__ void mma_commit(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
// Issue a 32-column TMEM load without waiting (tcgen05.wait::ld before the values are read).
__device__ __forceinline__ void tmem_ld32_nowait(unsigned taddr, unsigned (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}

}  // namespace tc

}  // namespace wt
