// FP64 matrix products on the tensor cores, through residues (the Chinese-remainder form of
// Ozaki's error-free splitting; Ozaki, Uchino and Imamura, "Ozaki Scheme II", 2025).
//
//   C = alpha op(A) op(B) + beta C,   all FP64, row-major
//
// GB300's FP64 units give about 1.1 TFLOP/s, its bf16 tensor cores about 1 900.  Every row of
// op(A) and every column of op(B) is scaled by a power of two and rounded to integers a', b' with
// ||a'||, ||b'|| of 2^57 to 2^58, so that |sum a' b'| <= 2^116 < P / 2 with P the product of 15 pairwise
// coprime odd moduli p <= 255.  Per modulus the product of the centred residues (|r| <= 127, exact
// in bf16) is one bf16 product with FP32 accumulation: 1024 terms of at most 127^2 stay below
// 2^24, so every accumulator is exact; it is reduced mod p every 1024 terms.  The 15 residues of
// an output give sum a' b' exactly (as a fraction of P, 84 bits), and one conversion and one
// multiplication bring it back to FP64.  Nothing but the rounding to a', b' and the final
// conversion is inexact.  The error is one of the norms: half a unit per entry on either side, so at most
// sqrt(K) 2^-57 ||a|| ||b|| and about 0.4 x 2^-57 ||a|| ||b|| where the roundings are independent, whatever K.
// Against an FP64 sum, whose error follows sum |a_k b_k|: measured on rows whose entries range over
// e^-3 .. e^3, a tenth of it (0.3 to 1.8e-17 ||a|| ||b|| against 3.2e-17 to 2.2e-16 over K of 64 to 18 432);
// entries below 2^-5 of their row's norm keep fewer than 53 bits, those below 2^-59 none, so that a row with
// one dominant entry whose partner is zero or tiny comes out less exact than by FP64 sums.  On the setups, fields
// and point values of single cells and 3 x 3 matrices the errors against 64-bit references are those of
// the FP64 sums or below (modes 1 to 8 times smaller, the rest within the spread of repeated runs).
//
// What bounds it: at the fit's sizes the bf16 product (15 x 2 M N K flop: 2 304 x 2 304 x 4 608 in 501 us,
// 1 460 TFLOP/s of bf16, the tensor pipe active 62 % of the time); for a short K the residue planes of C
// (15 bytes written and read per output).  Against the FP64 kernel: 2 304 x 2 304 x 18 432 (lower half)
// 93.6 -> 2.0 ms, 18 432 x 2 304 x 2 304 158 -> 2.9 ms, 1 152^3 3.5 -> 0.14 ms, 256^3 80 -> 37 us.  Kernels:
//   scale     largest exponent and sum of squares of every row of op(A) / column of op(B);
//   residues  a' and its 15 residues as bf16 planes [modulus][row][K], K-major
//             (convert: both, for both operands, in one launch where K is short);
//   product   persistent CTAs over (modulus, 128 x 256 tile): TMA loads into four 128-byte
//             swizzled stages, tcgen05.mma kind::f16 into two 256-column accumulators in tensor
//             memory (a chunk of 1024 terms each), eight epilogue warps that reduce and sum the
//             chunks in registers while the next chunk runs; residues out as int8;
//   combine   the residues of every output back to FP64, alpha and beta.
#include "tc_common.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

namespace wt {

namespace tcg {

using namespace tc;

constexpr int NMOD = 15;
constexpr int kNormBits = 58;             // log2 of the largest ||a'||, ||b'||
constexpr int BM = 128, BN = 256, BK = 64, STAGES = 4;
constexpr int CHUNK = 1024;               // terms per accumulator: 1024 x 127^2 < 2^24
constexpr int EPI_WARPS = 8;
constexpr int kFusedK = 1024;             // longest K whose operands one launch converts
constexpr int kMostTerms = 65535 * 64 / CHUNK * CHUNK;    // per pass: 64 of them per block of the residues' grid
constexpr int A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2;

// pairwise coprime: 3 5 17, 11 23, 251, 13 19, 241, 239, 233, 229, 227, 223, 7 31, 211, 199, 197, 193
constexpr int kMod[NMOD] = {255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193};

constexpr int centred(int x, int p) {
    x %= p;
    return 2 * x > p ? x - p : x;
}
// 2^(12 j) mod p, centred
constexpr int pow12(int j, int p) {
    int x = 1;
    for (int i = 0; i < 12 * j; ++i) x = 2 * x % p;
    return centred(x, p);
}
// y = (P / p)^-1 mod p
constexpr int crt_inverse(int m) {
    const int p = kMod[m];
    int q = 1;
    for (int i = 0; i < NMOD; ++i)
        if (i != m) q = q * (kMod[i] % p) % p;
    for (int y = 1; y < p; ++y)
        if (q * y % p == 1) return y;
    return 0;
}
// limb l (28 bits, l = 2 the highest) of floor(2^84 y / p)
constexpr long long crt_limb(int m, int l) {
    const long long p = kMod[m];
    long long rem = crt_inverse(m), out = 0;
    for (int k = 2; k >= l; --k) {
        rem <<= 28;
        out = rem / p;
        rem %= p;
    }
    return out;
}
struct Tables {
    float coef[NMOD][5];
    float p[NMOD], inv[NMOD];
    int limb[NMOD][3];
};
constexpr Tables make_tables() {
    Tables t{};
    for (int m = 0; m < NMOD; ++m) {
        for (int j = 0; j < 5; ++j) t.coef[m][j] = (float)pow12(j, kMod[m]);
        t.p[m] = (float)kMod[m];
        t.inv[m] = 1.0f / (float)kMod[m];
        for (int l = 0; l < 3; ++l) t.limb[m][l] = (int)crt_limb(m, l);
    }
    return t;
}
__constant__ float c_p[NMOD] = {255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193};

// x mod p, centred, for integers |x| < 2^24 held in FP32 (1.5 x 2^23 rounds to the nearest integer)
__device__ __forceinline__ float mod_centred(float x, float p, float inv) {
    const float q = __fadd_rn(__fmaf_rn(x, inv, 12582912.0f), -12582912.0f);
    return __fmaf_rn(-q, p, x);
}

// ------------------------------------------------------------------ scale
// Element (r, k) of an operand: TRANS false X[r ld + k], true X[k ld + r].  Largest biased
// exponent per row, then the sum of squares relative to it (2^20 fixed point: the integer sums do
// not depend on the order).  Blocks of 32 rows x 256 k.
constexpr int SC_R = 32, SC_K = 256;

// Biased exponent of x; 1 (its unit's) for a subnormal x, 0 for zero.
__device__ __forceinline__ unsigned exponent_of(double x) {
    const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu, lo = (unsigned)__double2loint(x);
    const unsigned ex = hi >> 20;
    return ex ? ex : (unsigned)((hi | lo) != 0);
}
// |x| 2^-(em - 1023) from the top 24 bits of x, for an x of at most the exponent em
__device__ __forceinline__ float scaled_top(double x, unsigned em) {
    const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu, lo = (unsigned)__double2loint(x);
    const unsigned m = ((hi & 0xfffffu) << 3) | (lo >> 29);
    const int ex = (int)(hi >> 20), d = max(ex, 1) - (int)em;  // <= 0
    if (d < -60) return 0.f;
    if (ex == 0) return (float)m * __uint_as_float((unsigned)(104 + d) << 23);
    return __uint_as_float(((unsigned)(127 + d) << 23) | m);
}
template <bool TRANS, bool SUM>
__global__ void __launch_bounds__(256) scale_kernel(const double* __restrict__ X, int ld, int rows, int K,
                                                    unsigned* __restrict__ emax, unsigned long long* __restrict__ ss) {
    const int r0 = blockIdx.x * SC_R, k0 = blockIdx.y * SC_K;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k1 = min(K, k0 + SC_K);
    __shared__ unsigned sh_e[8][33];
    __shared__ float sh_s[8][33];
    auto add = [&](double x, unsigned em, unsigned& e, float& s) {
        if (!SUM) e = max(e, exponent_of(x));
        else {
            const float f = scaled_top(x, em);
            s = fmaf(f, f, s);
        }
    };
    if (TRANS) {                                               // lane = row, warps over k
        const int r = r0 + lane;
        unsigned e = 0;
        float s = 0.f;
        const unsigned em = (SUM && r < rows) ? emax[r] : 0;
        if (r < rows)
            for (int k = k0 + w; k < k1; k += 8) add(X[(size_t)k * ld + r], em, e, s);
        if (!SUM) sh_e[w][lane] = e; else sh_s[w][lane] = s;
        __syncthreads();
        if (w == 0 && r < rows) {
            if (!SUM) {
                for (int q = 1; q < 8; ++q) e = max(e, sh_e[q][lane]);
                atomicMax(&emax[r], e);
            } else {
                for (int q = 1; q < 8; ++q) s += sh_s[q][lane];
                atomicAdd(&ss[r], (unsigned long long)ceilf(s * 1048576.0f));
            }
        }
    } else {                                                   // warp = row, lanes over k
        for (int i = w; i < SC_R; i += 8) {
            const int r = r0 + i;
            if (r >= rows) break;
            unsigned e = 0;
            float s = 0.f;
            const unsigned em = SUM ? emax[r] : 0;
            for (int k = k0 + lane; k < k1; k += 32) add(X[(size_t)r * ld + k], em, e, s);
            for (int o = 16; o; o >>= 1) {
                if (!SUM) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
                else s += __shfl_xor_sync(0xffffffffu, s, o);
            }
            if (lane == 0) {
                if (!SUM) atomicMax(&emax[r], e);
                else atomicAdd(&ss[r], (unsigned long long)ceilf(s * 1048576.0f));
            }
        }
    }
}

// Power of two by which a row is scaled: 2^sh with ||a 2^sh|| <= 2^58 (a margin of 2^-9 covers the
// rounding of the sum and of a' itself).  kZeroRow: nothing in the row; kBadRow: an infinity or a NaN in it
// (its products are summed in FP64, see combine_kernel).
constexpr int kZeroRow = 1 << 20, kBadRow = 1 << 21;
__device__ __forceinline__ int row_shift(unsigned emax, unsigned long long ss) {
    if (emax == 0) return kZeroRow;
    if (emax == 0x7ff) return kBadRow;
    // norm^2 = ss 2^-20 2^(2 (emax - 1023)); ceil(log2) of ss + its rounding, halved and rounded up
    const unsigned long long n2 = ss + (ss >> 9) + 2;
    const int b = 64 - __clzll((long long)n2);                 // n2 < 2^b
    const int half = (b - 20 + 1 + 64) / 2 - 32;               // norm <= 2^half 2^(emax - 1023)
    return kNormBits - half - ((int)emax - 1023);
}

// --------------------------------------------------------------- residues
// The residues of two neighbouring entries of a row scaled by 2^sh: 12-bit limbs of a' in FP32,
// whose sums with the centred powers of 2^12 stay below 2^24 (exact), reduced mod p.
__device__ __forceinline__ void residues_of(const double (&x)[2], int sh, __nv_bfloat162* dst, size_t plane) {
    constexpr Tables kT = make_tables();
    float limb[2][5];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const unsigned hi = (unsigned)__double2hiint(x[j]);
        const int ex = (int)((hi >> 20) & 0x7ff);
        unsigned long long mant = ((unsigned long long)(hi & 0xfffffu) << 32) | (unsigned)__double2loint(x[j]);
        if (ex) mant |= 1ull << 52;
        const int s = max(ex, 1) - 1075 + sh;                  // a' = round(mant 2^s) <= 2^58
        if (sh >= kZeroRow / 2 || s < -54) mant = 0;
        else if (s >= 0) mant <<= s;
        else mant = (mant + (1ull << (-s - 1))) >> -s;
        const float sg = (hi >> 31) ? -1.f : 1.f;
#pragma unroll
        for (int l = 0; l < 5; ++l) limb[j][l] = sg * (float)(unsigned)((mant >> (12 * l)) & 0xfffu);
    }
#pragma unroll
    for (int m = 0; m < NMOD; ++m) {
        float v[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            float y = limb[j][0];
#pragma unroll
            for (int l = 1; l < 5; ++l) y = fmaf(limb[j][l], kT.coef[m][l], y);
            v[j] = mod_centred(y, kT.p[m], kT.inv[m]);
        }
        dst[m * plane] = __floats2bfloat162_rn(v[0], v[1]);
    }
}
// 32 rows x 64 k per block through shared memory; planes out[m][row][Kp].
template <bool TRANS>
__global__ void __launch_bounds__(256) residue_kernel(const double* __restrict__ X, int ld, int rows, int k_begin,
                                                      int k_end, int Kp, const unsigned* __restrict__ emax,
                                                      const unsigned long long* __restrict__ ss,
                                                      __nv_bfloat16* __restrict__ out) {
    __shared__ double tile[32][65];
    const int r0 = blockIdx.x * 32, k0 = blockIdx.y * 64;      // k0 relative to k_begin
    const int K = k_end - k_begin;
    for (int e = threadIdx.x; e < 32 * 64; e += 256) {
        int r, k;
        if (TRANS) { k = e >> 5; r = e & 31; } else { r = e >> 6; k = e & 63; }
        double x = 0.0;
        if (r0 + r < rows && k0 + k < K)
            x = TRANS ? X[(size_t)(k_begin + k0 + k) * ld + r0 + r] : X[(size_t)(r0 + r) * ld + k_begin + k0 + k];
        tile[r][k] = x;
    }
    __syncthreads();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = w; i < 32; i += 8) {
        const int r = r0 + i;
        if (r >= rows) break;
        const int k = k0 + 2 * lane;
        if (k < Kp) {
            const double x[2] = {tile[i][2 * lane], tile[i][2 * lane + 1]};
            residues_of(x, row_shift(emax[r], ss[r]),
                        reinterpret_cast<__nv_bfloat162*>(out + (size_t)r * Kp + k), (size_t)rows * Kp / 2);
        }
    }
}

// Scale and residues of both operands in one launch, for products whose K a block can go over
// itself: 32 rows per block, three passes (exponents, squares, residues; the later ones find the
// operand in L2).  The tall case leaves too few blocks, so it takes the three kernels above.
struct Operand {
    const double* X;
    int ld, rows, blocks;
    bool trans;
    unsigned* emax;
    unsigned long long* ss;
    __nv_bfloat16* out;
};
__global__ void __launch_bounds__(256) convert_kernel(Operand A, Operand B, int K, int Kp) {
    const bool first = (int)blockIdx.x < A.blocks;
    const Operand P = first ? A : B;
    const int r0 = (first ? blockIdx.x : blockIdx.x - A.blocks) * 32;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __shared__ double tile[32][65];
    __shared__ unsigned e_sh[32];
    __shared__ unsigned long long s_sh[32];
    if (threadIdx.x < 32) { e_sh[threadIdx.x] = 0; s_sh[threadIdx.x] = 0; }
    __syncthreads();
    auto at = [&](int r, int k) { return P.trans ? P.X[(size_t)k * P.ld + r0 + r] : P.X[(size_t)(r0 + r) * P.ld + k]; };
    auto square = [](double x, unsigned em) {
        const float f = scaled_top(x, em);
        return f * f;
    };
    if (P.trans) {
        if (r0 + lane < P.rows) {
            unsigned e = 0;
            for (int k = w; k < K; k += 8) e = max(e, exponent_of(at(lane, k)));
            atomicMax(&e_sh[lane], e);
        }
        __syncthreads();
        if (r0 + lane < P.rows) {
            float s = 0.f;
            for (int k = w; k < K; k += 8) s += square(at(lane, k), e_sh[lane]);
            atomicAdd(&s_sh[lane], (unsigned long long)ceilf(s * 1048576.0f));
        }
    } else {
        for (int i = w; i < 32 && r0 + i < P.rows; i += 8) {
            unsigned e = 0;
            for (int k = lane; k < K; k += 32) e = max(e, exponent_of(at(i, k)));
            e = __reduce_max_sync(0xffffffffu, e);
            float s = 0.f;
            for (int k = lane; k < K; k += 32) s += square(at(i, k), e);
            for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) { e_sh[i] = e; s_sh[i] = (unsigned long long)ceilf(s * 1048576.0f); }
        }
    }
    __syncthreads();
    if (threadIdx.x < 32 && r0 + (int)threadIdx.x < P.rows) {
        P.emax[r0 + threadIdx.x] = e_sh[threadIdx.x];
        P.ss[r0 + threadIdx.x] = s_sh[threadIdx.x];
    }
    const size_t plane = (size_t)P.rows * Kp / 2;
    for (int k0 = 0; k0 < K; k0 += 64) {
        __syncthreads();
        for (int e = threadIdx.x; e < 32 * 64; e += 256) {
            int r, k;
            if (P.trans) { k = e >> 5; r = e & 31; } else { r = e >> 6; k = e & 63; }
            tile[r][k] = (r0 + r < P.rows && k0 + k < K) ? at(r, k0 + k) : 0.0;
        }
        __syncthreads();
        const int k = k0 + 2 * lane;
        if (k < Kp)
            for (int i = w; i < 32 && r0 + i < P.rows; i += 8) {
                const double x[2] = {tile[i][2 * lane], tile[i][2 * lane + 1]};
                residues_of(x, row_shift(e_sh[i], s_sh[i]),
                            reinterpret_cast<__nv_bfloat162*>(P.out + (size_t)(r0 + i) * Kp + k), plane);
            }
    }
}

// ---------------------------------------------------------------- product
struct Smem {
    unsigned long long full[STAGES], empty[STAGES], acc_full[2], acc_empty[2], drain;
    unsigned tmem_base;
    int abort_flag;
};

__device__ __forceinline__ void mma_bf16(unsigned tmem_d, unsigned long long a, unsigned long long b, unsigned idesc,
                                         unsigned accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}
// 3D tiled TMA load (k, row, modulus)
__device__ __forceinline__ void tma_load_3d(unsigned dst, const CUtensorMap* tm, int x, int y, int z,
                                            unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::
            "r"(dst),
        "l"(tm), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// Unit u -> modulus, tile.  Tiles of one modulus run together (their planes share L2), in bands of
// eight tile rows so that concurrent CTAs reuse both operands.
struct Units {
    int tm, tn, per_mod, n;
    int lower;                       // only tiles that touch the lower triangle
};
__device__ __forceinline__ bool unit_tile(const Units& U, int u, int& mod, int& m0, int& n0) {
    mod = u / U.per_mod;
    const int t = u % U.per_mod;
    constexpr int BAND = 8;
    const int band = t / (BAND * U.tn), in = t % (BAND * U.tn);
    const int rows = min(BAND, U.tm - band * BAND);
    m0 = (band * BAND + in % rows) * BM;
    n0 = (in / rows) * BN;
    return !U.lower || n0 <= m0 + BM - 1;
}

__global__ void __launch_bounds__(64 + 32 * EPI_WARPS, 1)
    product_kernel(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb, Units U, int M,
                   int N, int K, signed char* __restrict__ T, int Tp, int add, int* __restrict__ d_err) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    Smem* S = reinterpret_cast<Smem*>(base + (size_t)STAGES * (A_BYTES + B_BYTES));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < STAGES; ++i) {
            mbar_init(&S->full[i], 1);
            mbar_init(&S->empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&S->acc_full[i], 1);
            mbar_init(&S->acc_empty[i], 32 * EPI_WARPS);
        }
        mbar_init(&S->drain, 1);
        S->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S->tmem_base)), "n"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = S->tmem_base;
    volatile int* abort_flag = &S->abort_flag;
    const int kblocks = (K + BK - 1) / BK;
    constexpr int KB_CHUNK = CHUNK / BK;

    if (warp == 0) {
        // ---------------- producer: one TMA box of A (128 rows) and one of B (256 rows) per stage
        int i = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < U.n && ok; u += gridDim.x) {
            int mod, m0, n0;
            if (!unit_tile(U, u, mod, m0, n0)) continue;
            for (int kb = 0; kb < kblocks; ++kb, ++i) {
                const int st = i % STAGES;
                if (!mbar_wait(&S->empty[st], ((i / STAGES) & 1) ^ 1, abort_flag, d_err)) { ok = false; break; }
                if (lane == 0) {
                    const unsigned sa = smem_u32(base + (size_t)st * (A_BYTES + B_BYTES));
                    mbar_expect_tx(&S->full[st], A_BYTES + B_BYTES);
                    tma_load_3d(sa, &ma, kb * BK, m0, mod, &S->full[st]);
                    tma_load_3d(sa + A_BYTES, &mb, kb * BK, n0, mod, &S->full[st]);
                }
                __syncwarp();
            }
        }
        // after an abort: the loads still in flight land before the CTA exits (the barriers of the
        // last STAGES loads; a phase that completed earlier passes at once)
        if (!ok)
            for (int k = max(0, i - STAGES); k < i; ++k) mbar_wait_drain(&S->full[k % STAGES], (k / STAGES) & 1, d_err);
    } else if (warp == 1) {
        // ---------------- MMA issuer
        constexpr unsigned idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(BN >> 3) << 17) |
                                   ((unsigned)(BM >> 4) << 24);
        int i = 0, g = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < U.n && ok; u += gridDim.x) {
            int mod, m0, n0;
            if (!unit_tile(U, u, mod, m0, n0)) continue;
            for (int kb = 0; kb < kblocks && ok; ++kb, ++i) {
                const int in = kb % KB_CHUNK, b = g & 1;
                if (in == 0) {
                    if (!mbar_wait(&S->acc_empty[b], ((g >> 1) & 1) ^ 1, abort_flag, d_err)) { ok = false; break; }
                    tc_fence_after();
                }
                const int st = i % STAGES;
                if (!mbar_wait(&S->full[st], (i / STAGES) & 1, abort_flag, d_err)) { ok = false; break; }
                tc_fence_after();
                if (lane == 0) {
                    const unsigned sa = smem_u32(base + (size_t)st * (A_BYTES + B_BYTES)), sb = sa + A_BYTES;
#pragma unroll
                    for (int ks = 0; ks < BK / 16; ++ks)
                        mma_bf16(tmem + (unsigned)(b * BN), sdesc(sa + 32 * ks), sdesc(sb + 32 * ks), idesc,
                                 in > 0 || ks > 0);
                    mma_commit(&S->empty[st]);
                    if (in == KB_CHUNK - 1 || kb == kblocks - 1) mma_commit(&S->acc_full[b]);
                }
                __syncwarp();
                if (in == KB_CHUNK - 1 || kb == kblocks - 1) ++g;
            }
        }
        if (lane == 0) {
            mma_commit(&S->drain);
            mbar_wait_drain(&S->drain, 0, d_err);
        }
        __syncwarp();
    } else {
        // ---------------- epilogue: warps 2-9, TMEM lane quadrant warp & 3, 128 columns each
        const int q = warp & 3, half = (warp - 2) >> 2;
        const int n_chunks = (kblocks + KB_CHUNK - 1) / KB_CHUNK;
        int g = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < U.n && ok; u += gridDim.x) {
            int mod, m0, n0;
            if (!unit_tile(U, u, mod, m0, n0)) continue;
            const float p = c_p[mod], inv = __frcp_rn(p);
            float sum[128];
#pragma unroll
            for (int e = 0; e < 128; ++e) sum[e] = 0.f;
            for (int ch = 0; ch < n_chunks; ++ch, ++g) {
                const int b = g & 1;
                if (!mbar_wait(&S->acc_full[b], (g >> 1) & 1, abort_flag, d_err)) { ok = false; break; }
                tc_fence_after();
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    unsigned r[32];
                    tmem_ld32_nowait(tmem + ((unsigned)(q * 32) << 16) + (unsigned)(b * BN + half * 128 + j * 32), r);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int e = 0; e < 32; ++e) sum[32 * j + e] += mod_centred(__uint_as_float(r[e]), p, inv);
                }
                tc_fence_before();
                mbar_arrive(&S->acc_empty[b]);
            }
            if (!ok) break;
            const int m = m0 + q * 32 + lane, n = n0 + half * 128;
            if (m < M) {
                signed char* dst = T + ((size_t)mod * M + m) * Tp + n;
#pragma unroll
                for (int v = 0; v < 8; ++v) {
                    if (n + 16 * v >= Tp) break;
                    if (add) {                                  // the residues of the terms before this launch's
                        const int4 o = *reinterpret_cast<const int4*>(dst + 16 * v);
                        const int w[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
                        for (int e = 0; e < 16; ++e) sum[16 * v + e] += (float)(signed char)(w[e >> 2] >> (8 * (e & 3)));
                    }
                    int w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        unsigned x = 0;
#pragma unroll
                        for (int f = 0; f < 4; ++f)
                            x |= ((unsigned)(int)mod_centred(sum[16 * v + 4 * e + f], p, inv) & 0xffu) << (8 * f);
                        w[e] = (int)x;
                    }
                    *reinterpret_cast<int4*>(dst + 16 * v) = make_int4(w[0], w[1], w[2], w[3]);
                }
            }
        }
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(512));
    }
}

// ---------------------------------------------------------------- combine
// sum a' b' = P x frac(sum_m r_m y_m / p_m), the fraction to 84 bits in three 28-bit limbs, taken
// as signed; its top 64 bits to FP64 (2^-63 P is 2^-61 of ||a'|| ||b'||).  scale = alpha P 2^-64.
// Four outputs per thread.  The row blocks are the grid's first dimension: the rows of a field of many time
// samples (samples x lateral points) pass the 65 535 blocks of the others.
//
// An output whose row of op(A) or column of op(B) holds an infinity or a NaN is the FP64 sum itself.
struct Factors {
    const double *A, *B;
    int lda, ldb, K;
    bool ta, tb;
};
__global__ void __launch_bounds__(256) combine_kernel(const signed char* __restrict__ T, int Tp, int M, int N,
                                                      const unsigned* __restrict__ ea,
                                                      const unsigned long long* __restrict__ sa,
                                                      const unsigned* __restrict__ eb,
                                                      const unsigned long long* __restrict__ sb, double scale,
                                                      double beta, double* __restrict__ C, int ldc, int lower,
                                                      int mblk, size_t mstride, Factors F, double alpha) {
    const int n = 4 * (blockIdx.y * 64 + (threadIdx.x & 63)), m = blockIdx.x * 4 + (threadIdx.x >> 6);
    if (m >= M || n >= N || (lower && n > m)) return;
    constexpr Tables kT = make_tables();
    long long acc[4][3];
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int l = 0; l < 3; ++l) acc[e][l] = 0;
    const signed char* src = T + (size_t)m * Tp + n;
    int w[NMOD];
#pragma unroll
    for (int k = 0; k < NMOD; ++k) w[k] = *reinterpret_cast<const int*>(src + (size_t)k * M * Tp);
#pragma unroll
    for (int k = 0; k < NMOD; ++k)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int r = (int)(signed char)(w[k] >> (8 * e));
#pragma unroll
            for (int l = 0; l < 3; ++l) acc[e][l] += (long long)r * kT.limb[k][l];
        }
    const int sm = row_shift(ea[m], sa[m]);
    auto out = [&](int e) {
        return C + (mblk ? (size_t)(m / mblk) * mstride + (size_t)(m % mblk) * ldc : (size_t)m * ldc) + n + e;
    };
    int bad = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if (n + e >= N || (lower && n + e > m)) break;
        long long a1 = acc[e][1] + (acc[e][0] >> 28);
        long long a2 = acc[e][2] + (a1 >> 28);
        const unsigned lo = (unsigned)acc[e][0] & 0xfffffffu, mid = (unsigned)a1 & 0xfffffffu;
        const long long top = (long long)(((unsigned long long)a2 << 36) | ((unsigned long long)mid << 8) | (lo >> 20));
        const int sn = row_shift(eb[n + e], sb[n + e]);
        double v;
        if (sm >= kBadRow || sn >= kBadRow) {
            bad |= 1 << e;
            continue;
        }
        if (sm >= kZeroRow || sn >= kZeroRow) v = 0.0;
        else {
            const int h = -(sm + sn);
            if (abs(h) < 900)                    // scale 2^h by its exponent bits (scale is +-2^53.4)
                v = (double)top * __hiloint2double(__double2hiint(scale) + (h << 20), __double2loint(scale));
            else
                v = scalbn((double)top * scale, h);
        }
        double* c = out(e);
        *c = beta == 0.0 ? v : fma(beta, *c, v);
    }
    for (int e = 0; bad >> e; ++e) {
        if (!(bad >> e & 1)) continue;
        const double *a = F.A + (F.ta ? (size_t)m : (size_t)m * F.lda), *b = F.B + (F.tb ? (size_t)(n + e) * F.ldb : (size_t)(n + e));
        const size_t da = F.ta ? F.lda : 1, db = F.tb ? 1 : F.ldb;
        double v = 0.0;
        for (int k = 0; k < F.K; ++k, a += da, b += db) v = fma(*a, *b, v);
        double* c = out(e);
        *c = beta == 0.0 ? alpha * v : fma(beta, *c, alpha * v);
    }
}

static void encode_planes(CUtensorMap* m, const __nv_bfloat16* X, int rows, int K, int Kp, int box_rows) {
    cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)NMOD};
    cuuint64_t strides[2] = {(cuuint64_t)Kp * 2, (cuuint64_t)rows * Kp * 2};
    cuuint32_t box[3] = {BK, (cuuint32_t)box_rows, 1};
    cuuint32_t es[3] = {1, 1, 1};
    CUresult r = tensor_map_encoder()(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<__nv_bfloat16*>(X), dims,
                                      strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) fail(WT_ERR_CUDA, "tensor map for the residue planes: error " + std::to_string((int)r));
}

static void scales(cudaStream_t s, const double* X, int ld, bool trans, int rows, int K, unsigned* e,
                   unsigned long long* ss) {
    dim3 g((rows + SC_R - 1) / SC_R, (K + SC_K - 1) / SC_K);
    if (trans) {
        scale_kernel<true, false><<<g, 256, 0, s>>>(X, ld, rows, K, e, ss);
        scale_kernel<true, true><<<g, 256, 0, s>>>(X, ld, rows, K, e, ss);
    } else {
        scale_kernel<false, false><<<g, 256, 0, s>>>(X, ld, rows, K, e, ss);
        scale_kernel<false, true><<<g, 256, 0, s>>>(X, ld, rows, K, e, ss);
    }
    WT_LAUNCH("residue scales");
}

static void residues(cudaStream_t s, const double* X, int ld, bool trans, int rows, int kb, int ke, int Kp,
                     const unsigned* e, const unsigned long long* ss, __nv_bfloat16* out) {
    dim3 g((rows + 31) / 32, (ke - kb + 63) / 64);
    if (trans) residue_kernel<true><<<g, 256, 0, s>>>(X, ld, rows, kb, ke, Kp, e, ss, out);
    else residue_kernel<false><<<g, 256, 0, s>>>(X, ld, rows, kb, ke, Kp, e, ss, out);
    WT_LAUNCH("residues");
}

}  // namespace tcg

static thread_local CallMemory* t_memory = nullptr;
CallMemory::CallMemory(int* err) : d_err(err), outer(t_memory) { t_memory = this; }
CallMemory::~CallMemory() {
    t_memory = outer;
    if (ws) cudaFree(ws);
    for (void* c : chunks) cudaFree(c);
}
CallMemory* CallMemory::current() { return t_memory; }
bool CallMemory::trim() {
    bool any = false;
    for (CallMemory* m = this; m; m = m->outer) {
        if (m->ws) {
            cudaFree(m->ws);                     // waits for the products that still use it
            m->ws = nullptr;
            m->ws_cap = 0;
            any = true;
        }
        for (size_t k = 0; k < m->chunks.size(); ++k) {
            bool used = !m->chunks[k];
            for (const Piece& q : m->pieces) used = used || (q.chunk == (int)k && q.used);
            if (used) continue;
            cudaFree(m->chunks[k]);
            m->chunks[k] = nullptr;
            m->pieces.erase(std::remove_if(m->pieces.begin(), m->pieces.end(), [&](const Piece& q) { return q.chunk == (int)k; }),
                            m->pieces.end());
            any = true;
        }
    }
    return any;
}
// cudaMalloc, once more after trim(); NULL when the memory is not to be had.
static void* malloc_or_trim(CallMemory* m, size_t bytes) {
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) == cudaSuccess) return p;
    cudaGetLastError();
    if (m->trim() && cudaMalloc(&p, bytes) == cudaSuccess) return p;
    cudaGetLastError();
    return nullptr;
}
unsigned char* CallMemory::products(size_t bytes) {
    if (bytes <= ws_cap) return ws;
    if (fault_enabled("alloc")) return nullptr;
    if (ws) cudaFree(ws);                        // waits for the products that still use it
    ws = nullptr;
    ws_cap = 0;
    ws = static_cast<unsigned char*>(malloc_or_trim(this, bytes));
    if (ws) ws_cap = bytes;
    return ws;
}
// Best fit among the free pieces, else a chunk of its own size (at least 16 MB, shared by small ones).
void* CallMemory::take(size_t bytes) {
    const size_t need = (bytes + 511) & ~(size_t)511;
    int best = -1;
    for (size_t k = 0; k < pieces.size(); ++k)
        if (!pieces[k].used && pieces[k].size >= need && (best < 0 || pieces[k].size < pieces[best].size)) best = (int)k;
    if (best < 0) {
        size_t size = std::max(need, (size_t)16 << 20);
        void* c = nullptr;
        if (cudaMalloc(&c, size) != cudaSuccess) {           // then no more than is needed
            cudaGetLastError();
            size = need;
            c = malloc_or_trim(this, size);
            if (!c) return nullptr;
        }
        chunks.push_back(c);
        pieces.push_back({static_cast<unsigned char*>(c), size, (int)chunks.size() - 1, false});
        best = (int)pieces.size() - 1;
    }
    Piece& q = pieces[best];
    const Piece rest{q.p + need, q.size - need, q.chunk, false};
    q.used = true;
    q.size = need;
    void* p = q.p;
    if (rest.size) pieces.insert(pieces.begin() + best + 1, rest);
    return p;
}
void CallMemory::give(void* p) {
    for (size_t k = 0; k < pieces.size(); ++k) {
        if (pieces[k].p != p) continue;
        pieces[k].used = false;
        if (k + 1 < pieces.size() && !pieces[k + 1].used && pieces[k + 1].chunk == pieces[k].chunk) {
            pieces[k].size += pieces[k + 1].size;
            pieces.erase(pieces.begin() + k + 1);
        }
        if (k > 0 && !pieces[k - 1].used && pieces[k - 1].chunk == pieces[k].chunk) {
            pieces[k - 1].size += pieces[k].size;
            pieces.erase(pieces.begin() + k);
        }
        return;
    }
}

static size_t product_smem() {
    return 1024 + (size_t)tcg::STAGES * (tcg::A_BYTES + tcg::B_BYTES) + sizeof(tcg::Smem);
}
// Shared-memory limit of the product kernel on the current device; returns its SMs.
static int product_setup() {
    int dev = 0, n_sm = 0;
    WT_CUDA(cudaGetDevice(&dev));
    WT_CUDA(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev));
    allow_dyn_smem(tcg::product_kernel, product_smem());
    return n_sm;
}

// Workspace layout of one product: scales, residue planes of op(A) and op(B), residues of C.
struct Layout {
    bool same;
    int kc, Kp, Tp;
    size_t b_e, b_s, b_a, b_b, total;
};
static Layout layout(int M, int N, int K, bool same) {
    using namespace tcg;
    Layout L{};
    L.same = same;
    // terms per pass: residue planes of at most about 6 GB
    const size_t per_k = (size_t)(same ? M : M + N) * NMOD * 2;
    L.kc = K;
    if (per_k * (size_t)K > ((size_t)6 << 30))
        L.kc = (int)std::max<size_t>(CHUNK, (((size_t)6 << 30) / per_k) / CHUNK * CHUNK);
    L.kc = std::min(L.kc, kMostTerms);
    L.Kp = (std::min(K, L.kc) + 7) & ~7;
    L.Tp = (N + 15) & ~15;
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    L.b_e = up((size_t)(M + N) * 4);
    L.b_s = up((size_t)(M + N) * 8);
    L.b_a = up((size_t)NMOD * M * L.Kp * 2);
    L.b_b = same ? 0 : up((size_t)NMOD * N * L.Kp * 2);
    L.total = L.b_e + L.b_s + L.b_a + L.b_b + up((size_t)NMOD * M * L.Tp);
    return L;
}

// The product in workspace p.  mblk > 0: row m of C lies at (m / mblk) mstride + (m % mblk) ldc.
static void product(cudaStream_t s, bool ta, bool tb, int M, int N, int K, double alpha, const double* A, int lda,
                    const double* B, int ldb, double beta, double* C, int ldc, bool lower_only, int mblk, size_t mstride,
                    const Layout& L, unsigned char* p, int n_sm, int* d_err) {
    using namespace tcg;
    const bool same = L.same;
    const int kc = L.kc, Kp = L.Kp, Tp = L.Tp;
    unsigned* ea = reinterpret_cast<unsigned*>(p);
    unsigned* eb = same ? ea : ea + M;
    unsigned long long* sa = reinterpret_cast<unsigned long long*>(p + L.b_e);
    unsigned long long* sb = same ? sa : sa + M;
    __nv_bfloat16* ra = reinterpret_cast<__nv_bfloat16*>(p + L.b_e + L.b_s);
    __nv_bfloat16* rb = same ? ra : reinterpret_cast<__nv_bfloat16*>(p + L.b_e + L.b_s + L.b_a);
    signed char* T = reinterpret_cast<signed char*>(p + L.b_e + L.b_s + L.b_a + L.b_b);
    // op(A) rows: k contiguous unless transposed; op(B) columns: k contiguous when transposed.  One
    // conversion launch up to K = kFusedK (2304 x 2304 x 256: 3 launches, 21 us against 9 and 47 us of
    // host time); beyond, 32 rows per block leave SMs idle.
    const bool fused = K <= kFusedK && kc >= K;
    if (fused) {
        Operand oa{A, lda, M, (M + 31) / 32, ta, ea, sa, ra}, ob{B, ldb, N, (N + 31) / 32, !tb, eb, sb, rb};
        convert_kernel<<<oa.blocks + (same ? 0 : ob.blocks), 256, 0, s>>>(oa, ob, K, Kp);
        WT_LAUNCH("residues");
    } else {
        WT_CUDA(cudaMemsetAsync(p, 0, L.b_e + L.b_s, s));
        scales(s, A, lda, ta, M, K, ea, sa);
        if (!same) scales(s, B, ldb, !tb, N, K, eb, sb);
    }
    Units U{};
    U.tm = (M + BM - 1) / BM;
    U.tn = (N + BN - 1) / BN;
    U.per_mod = U.tm * U.tn;
    U.n = U.per_mod * NMOD;
    U.lower = lower_only ? 1 : 0;
    const size_t sh = product_smem();
    for (int k0 = 0; k0 < K; k0 += kc) {
        const int k1 = std::min(K, k0 + kc);
        if (!fused) {
            residues(s, A, lda, ta, M, k0, k1, Kp, ea, sa, ra);
            if (!same) residues(s, B, ldb, !tb, N, k0, k1, Kp, eb, sb, rb);
        }
        CUtensorMap ma, mb;
        encode_planes(&ma, ra, M, k1 - k0, Kp, BM);
        encode_planes(&mb, rb, N, k1 - k0, Kp, BN);
        product_kernel<<<std::min(n_sm, U.n), 64 + 32 * EPI_WARPS, sh, s>>>(ma, mb, U, M, N, k1 - k0, T, Tp, k0 > 0,
                                                                          d_err);
        WT_LAUNCH("residue product");
    }
    unsigned __int128 P = 1;
    for (int m = 0; m < NMOD; ++m) P *= (unsigned)kMod[m];     // 117.4 bits, exact
    combine_kernel<<<dim3((M + 3) / 4, (N + 255) / 256), 256, 0, s>>>(
        T, Tp, M, N, ea, sa, eb, sb, std::ldexp((double)P, -64) * alpha, beta, C, ldc, lower_only ? 1 : 0, mblk, mstride,
        Factors{A, B, lda, ldb, K, ta, tb}, alpha);
    WT_LAUNCH("residue combine");
    // WT_FAULT=product_timeout: as if a wait of the product had run out (WT_FAULT_AT=n: of the call's n-th product)
    if (fault_enabled("product_timeout")) {
        const char* at = std::getenv("WT_FAULT_AT");
        CallMemory* mem = CallMemory::current();
        if (!at || (mem && ++mem->n_products == std::atoi(at))) {
            const int v = DERR_TIMEOUT;
            WT_CUDA(cudaMemcpyAsync(d_err, &v, sizeof(int), cudaMemcpyHostToDevice, s));
        }
    }
}

// True when the product was launched; false: the caller's FP64 kernel takes it.
bool dgemm_tc(cudaStream_t s, bool ta, bool tb, int M, int N, int K, double alpha, const double* A, int lda,
              const double* B, int ldb, double beta, double* C, int ldc, bool lower_only) {
    CallMemory* mem = t_memory;
    if (!mem || !mem->d_err || std::fabs(alpha) != 1.0 || K > 65535 * tcg::SC_K || N > 65535 * 256) return false;
    // op(A) rows and op(B) columns that are the same vectors are converted once
    const Layout L = layout(M, N, K, A == B && lda == ldb && ta != tb && M == N);
    unsigned char* p = mem->products(L.total);
    if (!p) return false;
    if (!mem->n_sm) mem->n_sm = product_setup();              // once per call of the library
    product(s, ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, lower_only, 0, 0, L, p, mem->n_sm, mem->d_err);
    return true;
}

// C[m / mblk][m % mblk][n] = sum_k A[k][m] B[n][k] for M = blocks x mblk rows, row block b of C at
// b mstride: the z series of many lines.  Workspace from the caller (dgemm_tc_rows_bytes).
size_t dgemm_tc_rows_bytes(int M, int N, int K) { return layout(M, N, K, false).total; }
void dgemm_tc_rows(cudaStream_t s, int M, int N, int K, const double* A, int lda, const double* B, int ldb, double* C,
                   int ldc, int mblk, size_t mstride, unsigned char* ws, int* d_err) {
    product(s, true, true, M, N, K, 1.0, A, lda, B, ldb, 0.0, C, ldc, false, mblk, mstride, layout(M, N, K, false), ws,
            product_setup(), d_err);
}

}  // namespace wt
