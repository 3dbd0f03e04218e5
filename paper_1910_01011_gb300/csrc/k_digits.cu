// k_digits.cu -- complex128 matrix x block of vectors on the tensor cores,
// each run of 256 columns to ~2^-51 of the largest term it can have, sums
// exact or in FP64 (the FP64 residual of the refinement, r = b - A_hat u with
// the assembled complex128 A_hat).
//
// GB300 runs FP64 at 1/64 of its FP32 rate, and carrying the products in FP32
// pairs takes ~25 packed FP32 instructions per entry and vector.  Here both
// operands are fixed-point numbers cut into digits, and the digits' products
// and sums are exact (the error-free splitting of Ozaki, Ogita, Oishi and
// Rump, "Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication and its applications", 2012):
//
//  * K is cut into units of 256 columns.  In each, A' = 2^-row A 2^-col with
//    powers of two per column and per row and unit (columns first, so that psi
//    and phi columns, a factor |k| apart, share their bits where a unit holds
//    both), each real part below 1/4 as Q 2^-56, |Q| < 2^54, and
//    Q = sum_i d_i 128^(7 - i) with eight digits d_i in [-64, 63].  A digit is a
//    byte (d + 64): 16 bytes per complex entry, as complex128 itself.
//  * vectors likewise, x_j 2^col_j with a power of two per vector and unit (one
//    for the whole vector and one per row lost 2^-40 of sum |a| |x| on 20,484
//    unknowns: the phi columns hold W, whose diagonal is 2^10 and more above
//    everything in the psi columns), as BF16 digits (integers up to 256 are
//    exact in BF16).
//  * Y' = sum_{i + j <= 7} 2^(-7 (i + j + 2)) A_i X_j on tcgen05 (kind::f16,
//    BF16 in, FP32 out): the products are integers of at most 2^12, a sum of
//    K = 256 of both real parts and up to eight (i, j) stays below 2^24, so
//    every FP32 accumulator holds its integer exactly whatever the order or
//    rounding mode of the unit.  Dropped are the seven products with i + j = 8,
//    at most 2^12 2^-70 each, and smaller ones: 2^-55, or 2^-51 of the largest a
//    term can be (1/4 x 1/4).
//  * at the end of a unit the eight accumulators of an output are added in a
//    64-bit integer (exact; only sums of nearly the largest size lose the lowest
//    8 of 70 bits), which goes into the FP64 sum of the CTA's run with the unit's
//    power of two; pieces of K are added in FP64.
//
// The 36 digit products of a step need no 36 instructions: X's digits lie side
// by side as rows of B, X_0 first, and A_i times the first 8 - i of them, into
// accumulators starting at the i-th, adds every product to the accumulator of
// its weight.  Real and imaginary parts of A are two A operands with
// B = [Xr | Xi] and [-Xi | Xr] on the same accumulators.
//
// What binds it is reading A once (16 N^2 bytes): A's bytes are stored in the
// order in which a CTA reads them (stages of 128 rows x 32 of K x 16 digit
// planes, 64 KB, in two bulk copies, real and imaginary digits), four warps turn
// them into BF16 pairs (a byte permute and one subtraction per two digits) and
// put them into tensor memory as the A operand, so shared memory holds them only
// once, as bytes.  Every CTA takes an equal run of stages across row tiles, and
// pieces of a tile are added in FP64.  The copies of A and the set-up of a CTA do
// not wait for the vectors' digits, and where the accumulators take half of their
// columns (up to eight vectors) a second set takes the next unit while the first
// is read.  With whole units per CTA (15 for some, 14 for others), one set of
// accumulators, 64 KB copies and two more launches, one vector took 223 us on
// N = 8,200 and 36 us on N = 324 (FP32 pairs 193 and 28 us), now 193 and 20 us.
//
// N = 10,776, 16 vectors: a call takes 410 us (4.5 TB/s of A; the instructions of
// half a stage take 1,306 cycles, its bytes 1,490 at the copy rate) against 4,550
// us in FP32 pairs; N = 10,608, one vector 306 us (5.9 TB/s) against 403 us.
// Error of the product with a smooth vector on 20,484 unknowns, against
// 128-bit sums of the entries: 3e-14, and 2^-47.7 of a row's sum |a| |x| at most
// (FP32 pairs 2.4e-13 and 2^-43.7; one power of two per vector and row 6.7e-13 and
// 2^-40.1).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstdint>
#include <string>
#include <vector>

#include "ctx.h"
#include "internal.h"
#include "launch.cuh"

namespace gbem {

constexpr int DG = 8;                      // digits of a real number
constexpr int DG_M = 128;                  // rows of A per tile
constexpr int DG_K = 32;                   // K per stage (bytes per digit row)
constexpr int DG_STEPS = 8;                // stages per unit
constexpr int DG_UNIT = DG_K * DG_STEPS;   // K of a unit: 256
constexpr int DG_CTAS = 152;
constexpr int DG_PLANE = DG_M * DG_K;      // bytes of one digit plane of a stage
constexpr int DG_ABYTES = 2 * DG * DG_PLANE;
constexpr int DG_WARPS = 10;               // 0 copies, 1 MMA, 2-5 digits to BF16, 6-9 accumulators
constexpr int DG_NONE = INT_MIN / 4;       // exponent of a zero row, column or vector
constexpr int DG_BAD = INT_MAX / 4;        // of one with an infinity or a NaN

// NC columns of B per digit: NC / 2 right-hand sides, real and imaginary parts
template <int NC>
struct DgCfg {
    static constexpr int HN = NC / 2;
    static constexpr int BROWS = DG * NC;              // B rows: digit j, column n at j NC + n
    static constexpr int BBYTES = 2 * BROWS * DG_K * 2;  // [Xr | Xi] and [-Xi | Xr] of a stage
    static constexpr int ACC = 256 / (DG * NC);        // sets of accumulators in 256 columns of tensor memory
    static constexpr int RING = NC == 16 ? 5 : 4;      // half stages (the real or the imaginary digits of A) in flight
    struct Smem {
        alignas(1024) uint8_t a[RING][DG_ABYTES / 2];
        alignas(1024) uint8_t b[RING][BBYTES / 2];
        double sum[NC][DG_M];                          // of the CTA's units of a tile
        uint64_t full[RING], empty[RING];              // copies landed; bytes converted (4 warps) and B used (MMA)
        uint64_t tfull[2], tempty[2];                  // A operand of a half stage in tensor memory
        uint64_t dfull[ACC], dempty[ACC];              // accumulators of a unit
        uint32_t tmem;
        int vmax[HN];
    };
    static_assert(sizeof(Smem) + 1024 <= 227 * 1024, "digits smem");
};

// ----------------------------------------------------------------- digits

// e with |v| < 2^e of a double, from its bits; DG_NONE for zero (and subnormals), DG_BAD for infinities and NaN
__device__ __forceinline__ int dg_exp(double v) {
    const int b = (__double2hiint(v) >> 20) & 0x7ff;
    return b == 0 ? DG_NONE : b == 0x7ff ? DG_BAD : b - 1022;
}
__device__ __forceinline__ int dg_exp2(double2 v) { return max(dg_exp(v.x), dg_exp(v.y)); }

// Q + bias of v 2^(56 - e), |v| < 2^(e - 2), rounded to nearest, in integers
// (no FP64): its base-128 digits are d + 64, the bias 64 sum_t 128^t.
__device__ __forceinline__ unsigned long long dg_biased(double v, int e) {
    constexpr unsigned long long bias = 0x0081020408102040ull;
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    const int be = (int)(bits >> 52) & 0x7ff;
    if (be == 0) return bias;  // zero (and subnormals)
    const unsigned long long m = (bits & 0xfffffffffffffull) | 0x10000000000000ull;  // v = m 2^(be - 1075)
    const int sh = be - 1075 + 56 - e;
    const unsigned long long q = sh >= 0 ? m << sh : sh < -54 ? 0 : (m + (1ull << (-sh - 1))) >> -sh;
    return (bits >> 63) ? bias - q : bias + q;
}

// col[j] = largest exponent of column j of A (n rows, leading dimension ld); CTA: 128 columns, a range of rows
__global__ void dg_colexp_kernel(const double2* __restrict__ A, int64_t n, int64_t ld, int64_t rows_per, int* col) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const int64_t r1 = min(n, ((int64_t)blockIdx.y + 1) * rows_per);
    int e = DG_NONE;
#pragma unroll 4
    for (int64_t i = (int64_t)blockIdx.y * rows_per; i < r1; i++) e = max(e, dg_exp2(A[i * ld + j]));
    atomicMax(&col[j], e);
}

__device__ __forceinline__ int warp_max(int e) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    return e;
}

// One row per CTA: its exponents (rowe [unit][mpad], rowm the largest), then its digits into the row tile's blocks
// (out: the first tile of the launch).
__global__ void __launch_bounds__(256) dg_digits_kernel(const double2* __restrict__ A, int64_t n, int64_t ld, int64_t row0,
                                                        int64_t nkb, const int* __restrict__ col, int* __restrict__ rowm,
                                                        int* rowe, int64_t mpad, uint8_t* __restrict__ out) {
    __shared__ int sh[8];
    const int64_t i = row0 + blockIdx.x;
    const int r = blockIdx.x % DG_M, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double2* a = A + i * ld;
    int top = DG_NONE;
    for (int64_t u = warp; u * DG_UNIT < ld; u += 8) {
        int e = DG_NONE;
        if (i < n)
            for (int64_t j = u * DG_UNIT + lane; j < min(n, (u + 1) * DG_UNIT); j += 32) {
                const int v = dg_exp2(a[j]), c = col[j];
                if (v != DG_NONE) e = max(e, v == DG_BAD || c == DG_BAD ? DG_BAD : v - c);
            }
        e = warp_max(e);
        if (lane == 0) rowe[u * mpad + i] = e;
        top = max(top, e);
    }
    if (lane == 0) sh[warp] = top;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; w++) top = max(top, sh[w]);
        rowm[i] = top;
    }
    // a thread takes four neighbouring entries: 4-byte stores per digit plane
    uint8_t* tile = out + (int64_t)(blockIdx.x / DG_M) * nkb * DG_ABYTES;
    for (int64_t q = threadIdx.x; q < nkb * (DG_K / 4); q += blockDim.x) {
        const int64_t kb = q / (DG_K / 4);
        const int k = (int)(q % (DG_K / 4)) * 4;
        const int e = rowe[kb / DG_STEPS * mpad + i];
        unsigned long long u[2][4];
#pragma unroll
        for (int t = 0; t < 4; t++) {
            const int64_t j = kb * DG_K + k + t;
            double2 v = make_double2(0, 0);
            int s = 0;
            if (i < n && j < n && e != DG_BAD && e != DG_NONE) {
                v = a[j];
                s = col[j] + e + 2;
            }
            u[0][t] = dg_biased(v.x, s);
            u[1][t] = dg_biased(v.y, s);
        }
        // 32-byte rows, 16-byte halves swapped in every other group of four rows (bank conflicts)
        uint8_t* dst = tile + kb * DG_ABYTES + r * DG_K + ((k / 16) ^ ((r >> 2) & 1)) * 16 + k % 16;
#pragma unroll
        for (int p = 0; p < 2; p++)
#pragma unroll
            for (int d = 0; d < DG; d++) {
                uint32_t w = 0;
#pragma unroll
                for (int t = 0; t < 4; t++) w |= ((uint32_t)(u[p][t] >> (7 * (DG - 1 - d))) & 127u) << (8 * t);
                *reinterpret_cast<uint32_t*>(dst + (p * DG + d) * DG_PLANE) = w;
            }
    }
}

// Digits of R <= hn vectors as the B operand: blocks of one stage, [part][digit HN*2 + column][32 K], 64-byte rows
// in the 64-byte swizzle; vectors above R and K above n are zero.  ve[r][u] = largest exponent of x_r 2^col in unit u.
// Grid (units, hn), a thread an entry.
__global__ void __launch_bounds__(DG_UNIT) dg_vector_kernel(const double2* __restrict__ x, int64_t n, int64_t kpad, int R, int hn,
                                                            const int* __restrict__ col, int* __restrict__ ve,
                                                            uint8_t* __restrict__ out) {
    __shared__ int sh[DG_UNIT / 32];
    dependents_may_start();
    const int64_t j = (int64_t)blockIdx.x * DG_UNIT + threadIdx.x;
    const int r = blockIdx.y;
    double2 v = make_double2(0, 0);
    int c = DG_NONE, e = DG_NONE;
    if (r < R && j < n) {
        v = x[(int64_t)r * n + j];
        c = col[j];
        const int t = dg_exp2(v);
        if (t != DG_NONE) e = t == DG_BAD || c == DG_BAD ? DG_BAD : c == DG_NONE ? DG_NONE : t + c;
    }
    e = warp_max(e);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = e;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < DG_UNIT / 32; w++) e = max(e, sh[w]);
    if (r < R && threadIdx.x == 0) ve[(int64_t)r * gridDim.x + blockIdx.x] = e;
    if (j >= kpad) return;
    int s = 0;
    if (e == DG_NONE || e == DG_BAD || c == DG_NONE) v = make_double2(0, 0);
    else s = e + 2 - c;
    const unsigned long long u[2] = {dg_biased(v.x, s), dg_biased(v.y, s)};
    const int brows = DG * 2 * hn, k = (int)(j % DG_K);
    uint8_t* blk = out + j / DG_K * (int64_t)(2 * brows * DG_K * 2);
#pragma unroll
    for (int d = 0; d < DG; d++) {
        const float re = (float)((int)((u[0] >> (7 * (DG - 1 - d))) & 127u) - 64);
        const float im = (float)((int)((u[1] >> (7 * (DG - 1 - d))) & 127u) - 64);
        const float val[2][2] = {{re, im}, {-im, re}};
#pragma unroll
        for (int p = 0; p < 2; p++)
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int row = p * brows + d * 2 * hn + h * hn + r;
                *reinterpret_cast<__nv_bfloat16*>(blk + (int64_t)row * 64 + (((k / 8) ^ ((row >> 1) & 3)) * 16) + (k % 8) * 2) =
                    __float2bfloat16_rn(val[p][h]);
            }
    }
}

// ----------------------------------------------------------------- the product

__device__ __forceinline__ uint32_t d_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void d_init(uint64_t* b, uint32_t n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(d_u32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void d_arrive(uint64_t* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(d_u32(b)) : "memory");
}
__device__ __forceinline__ bool d_try(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 100000;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(d_u32(b)), "r"(parity)
        : "memory");
    return ok;
}
// Bounded wait (about a second); on timeout raises the error flag and returns false, as does every later wait.
__device__ __forceinline__ bool d_wait(uint64_t* b, uint32_t parity, int* err) {
    if (d_try(b, parity)) return true;
    if (*(volatile int*)err) return false;
    const long long t0 = clock64();
    while (!d_try(b, parity))
        if (clock64() - t0 > (1ll << 31)) {
            atomicExch(err, 2);
            return false;
        }
    return true;
}
__device__ __forceinline__ void d_bulk(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(d_u32(dst)),
        "l"(src), "r"(bytes), "r"(d_u32(bar))
        : "memory");
}
// B operand: K-major, 64-byte rows in the 64-byte swizzle, 8-row groups 512 bytes apart
__device__ __forceinline__ uint64_t d_desc(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | (uint64_t)1 << 16 | (uint64_t)(512 >> 4) << 32 | (uint64_t)1 << 46 |
           (uint64_t)4 << 61;
}
// D (128 x N) += A (tensor memory, 128 x 16) B (N x 16)
__device__ __forceinline__ void d_mma(uint32_t d, uint32_t a, uint64_t b, uint32_t n, uint32_t accumulate) {
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((uint32_t)(DG_M >> 4) << 24);
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(d),
        "r"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void d_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(d_u32(bar)) : "memory");
}
__device__ __forceinline__ void d_st8(uint32_t t, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(t), "r"(r[0]), "r"(r[1]),
                 "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
__device__ __forceinline__ void d_ld8(uint32_t t, float (&v)[8]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(t));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = __uint_as_float(r[i]);
}
#define DG_FENCE_BEFORE asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory")
#define DG_FENCE_AFTER asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory")

struct DgArgs {
    const uint8_t* A;     // [row tile][K block][plane][row][32]
    const uint8_t* B;     // [K block][part][row][32 bf16]
    int nkb, stages, pieces, m, R;  // K blocks; stages (row tiles x K blocks)
    int64_t mpad;
    const int *rowm, *rowe, *ve;
    double2* part;        // [row tile][piece][HN][128]
    double2* Y;           // [R][m]
    int* err;
};

__host__ __device__ inline int dg_first_stage(int stages, int ctas, int b) { return (int)((int64_t)stages * b / ctas); }
// the first of the CTAs that hold stages of `tile`
__host__ __device__ inline int dg_first_cta(int stages, int ctas, int nkb, int tile) {
    const int g = tile * nkb;
    int b = (int)((int64_t)g * ctas / stages);
    while (b + 1 < ctas && dg_first_stage(stages, ctas, b + 1) <= g) b++;
    while (b > 0 && dg_first_stage(stages, ctas, b) > g) b--;
    return b;
}
// The part of a unit that starts at stage g of a run up to g1: its row tile, unit and K blocks.
struct DgSpan {
    int tile, unit, kb0, kb1;
    __device__ __forceinline__ DgSpan(int g, int g1, int nkb) {
        tile = g / nkb;
        kb0 = g - tile * nkb;
        unit = kb0 / DG_STEPS;
        kb1 = min(min(nkb, (unit + 1) * DG_STEPS), kb0 + g1 - g);
    }
};

template <int NC>
__global__ void __launch_bounds__(DG_WARPS * 32, 1) digits_gemm_kernel(const DgArgs a) {
    typedef DgCfg<NC> C;
    extern __shared__ uint8_t smem_raw[];
    typename C::Smem& sm =
        *reinterpret_cast<typename C::Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g0 = dg_first_stage(a.stages, gridDim.x, blockIdx.x), g1 = dg_first_stage(a.stages, gridDim.x, blockIdx.x + 1);
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::RING; s++) {
            d_init(&sm.full[s], 1);
            d_init(&sm.empty[s], 5);
        }
        for (int b = 0; b < 2; b++) {
            d_init(&sm.tfull[b], 4);
            d_init(&sm.tempty[b], 1);
        }
        for (int d = 0; d < C::ACC; d++) {
            d_init(&sm.dfull[d], 1);
            d_init(&sm.dempty[d], 4);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(d_u32(&sm.tmem)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    DG_FENCE_BEFORE;
    __syncthreads();
    DG_FENCE_AFTER;
    const uint32_t tmem = sm.tmem;      // accumulators: sets of 8 NC columns
    const uint32_t ta = tmem + 256;     // two A operands: [K = 16 step][plane] x 8 columns

    if (warp == 0) {
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 1;
            bool ok = true;
            for (int g = g0; g < g1 && ok;) {
                const DgSpan w(g, g1, a.nkb);
                for (int h = 2 * w.kb0; h < 2 * w.kb1; h++) {
                    if (!(ok = d_wait(&sm.empty[s], ph, a.err))) break;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(d_u32(&sm.full[s])),
                                 "r"((DG_ABYTES + C::BBYTES) / 2)
                                 : "memory");
                    d_bulk(sm.a[s], a.A + ((int64_t)w.tile * a.nkb * 2 + h) * (DG_ABYTES / 2), DG_ABYTES / 2, &sm.full[s]);
                    if (g == g0 && h == 2 * w.kb0) inputs_ready();  // (A was there before the vectors)
                    d_bulk(sm.b[s], a.B + (int64_t)h * (C::BBYTES / 2), C::BBYTES / 2, &sm.full[s]);
                    if (++s == C::RING) {
                        s = 0;
                        ph ^= 1;
                    }
                }
                g += w.kb1 - w.kb0;
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int s = 0, b = 0;
            uint32_t ph = 0, tph = 0;
            bool ok = true;
            int d = 0;
            uint32_t dph = 1;
            for (int g = g0; g < g1 && ok;) {
                const DgSpan w(g, g1, a.nkb);
                if (!(ok = d_wait(&sm.dempty[d], dph, a.err))) break;  // (at once the first time)
                DG_FENCE_AFTER;
                const uint32_t acc = tmem + d * DG * NC;
                for (int h = 2 * w.kb0; h < 2 * w.kb1; h++) {
                    if (!(ok = d_wait(&sm.full[s], ph, a.err) && d_wait(&sm.tfull[b], tph, a.err))) break;
                    DG_FENCE_AFTER;
                    const uint32_t bs = d_u32(sm.b[s]);
#pragma unroll
                    for (int kk = 0; kk < 2; kk++)
#pragma unroll
                        for (int i = 0; i < DG; i++)
                            d_mma(acc + i * NC, ta + b * 128 + (kk * DG + i) * 8, d_desc(bs + kk * 32), NC * (DG - i),
                                  h > 2 * w.kb0 || kk > 0 || i > 0);
                    d_commit(&sm.tempty[b]);
                    d_commit(&sm.empty[s]);
                    b ^= 1;
                    if (b == 0) tph ^= 1;
                    if (++s == C::RING) {
                        s = 0;
                        ph ^= 1;
                    }
                }
                if (ok) d_commit(&sm.dfull[d]);
                if (++d == C::ACC) {
                    d = 0;
                    dph ^= 1;
                }
                g += w.kb1 - w.kb0;
            }
        }
    } else if (warp < 6) {
        // bytes d + 64 -> BF16 128 + (d + 64) by a byte permute, minus 192
        const int q = warp & 3, row = q * 32 + lane, sw = ((row >> 2) & 1) * 16;
        const uint32_t lt = ta + ((uint32_t)(q * 32) << 16);
        const __nv_bfloat162 off = __floats2bfloat162_rn(192.f, 192.f);
        int s = 0, b = 0;
        uint32_t ph = 0, tph = 1;
        for (int h = 2 * g0; h < 2 * g1; h++) {
            d_wait(&sm.full[s], ph, a.err);
            const uint8_t* src = sm.a[s] + row * DG_K;
            d_wait(&sm.tempty[b], tph, a.err);
            DG_FENCE_AFTER;
#pragma unroll 2
            for (int p = 0; p < DG; p++)
#pragma unroll
                for (int kk = 0; kk < 2; kk++) {
                    const uint4 v = *reinterpret_cast<const uint4*>(src + p * DG_PLANE + ((kk * 16) ^ sw));
                    const uint32_t in[4] = {v.x, v.y, v.z, v.w};
                    uint32_t r[8];
#pragma unroll
                    for (int w = 0; w < 4; w++)
#pragma unroll
                        for (int hb = 0; hb < 2; hb++) {
                            const uint32_t t = __byte_perm(in[w], 0x43434343u, hb ? 0x4342 : 0x4140);
                            const __nv_bfloat162 d = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&t), off);
                            r[2 * w + hb] = *reinterpret_cast<const uint32_t*>(&d);
                        }
                    d_st8(lt + b * 128 + (kk * DG + p) * 8, r);
                }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            DG_FENCE_BEFORE;
            __syncwarp();
            if (lane == 0) {
                d_arrive(&sm.tfull[b]);
                d_arrive(&sm.empty[s]);
            }
            b ^= 1;
            if (b == 0) tph ^= 1;
            if (++s == C::RING) {
                s = 0;
                ph ^= 1;
            }
        }
    } else {
        const int q = warp & 3, r = q * 32 + lane;
        const uint32_t ld = tmem + ((uint32_t)(q * 32) << 16);
        // the largest exponent of each vector: eight lanes a vector
        inputs_ready();
        dependents_may_start();
        const int nch = (a.nkb + DG_STEPS - 1) / DG_STEPS;
        for (int j = (warp - 6) * 4 + lane / 8; j < a.R; j += 16) {
            int e = DG_NONE;
            for (int u = lane % 8; u < nch; u += 8) e = max(e, a.ve[(int64_t)j * nch + u]);
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffu << (lane & 24), e, o));
            if (lane % 8 == 0) sm.vmax[j] = e;
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");  // (these four warps)
        bool fresh = true;  // no unit of the tile in `sum` yet
        int d = 0;
        uint32_t dph = 0;
        for (int g = g0; g < g1;) {
            const DgSpan w(g, g1, a.nkb);
            const int64_t row = (int64_t)w.tile * DG_M + r;
            const int er = max(a.rowe[w.unit * a.mpad + row] - a.rowm[row], -2000);  // -2000: nothing in this unit
            d_wait(&sm.dfull[d], dph, a.err);
            DG_FENCE_AFTER;
            // sums in 2^-49 of the first accumulator, exact, or from 2^62 on (bit set in `large`) rounded to 2^-41
            long long y[NC];
            uint32_t large = 0;
#pragma unroll
            for (int j0 = 0; j0 < NC; j0 += 8) {
                long long t[2][8];
#pragma unroll
                for (int h = 0; h < 2; h++)
#pragma unroll
                    for (int s = 0; s < 4; s++) {
                        float v[8];
                        d_ld8(ld + (d * DG + 4 * h + s) * NC + j0, v);
#pragma unroll
                        for (int j = 0; j < 8; j++) t[h][j] = (s ? t[h][j] * 128 : 0) + __float2int_rn(v[j]);
                    }
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    const bool l = t[0][j] >= (1ll << 34) || t[0][j] <= -(1ll << 34);
                    y[j0 + j] = l ? t[0][j] * (1 << 20) + ((t[1][j] + 128) >> 8) : t[0][j] * (1 << 28) + t[1][j];
                    large |= (uint32_t)l << (j0 + j);
                }
            }
            DG_FENCE_BEFORE;
            __syncwarp();
            if (lane == 0) d_arrive(&sm.dempty[d]);
            if (++d == C::ACC) {
                d = 0;
                dph ^= 1;
            }
            g += w.kb1 - w.kb0;
            const bool end = g == g1 || w.kb1 == a.nkb;
            const int piece = blockIdx.x - dg_first_cta(a.stages, gridDim.x, a.nkb, w.tile);
            double2* out = a.part + (int64_t)(w.tile * a.pieces + piece) * C::HN * DG_M + r;
#pragma unroll
            for (int j = 0; j < C::HN; j++) {
                if (j >= a.R) break;
                const int e = er + max(a.ve[(int64_t)j * nch + w.unit] - sm.vmax[j], -2000);
                const double fx = e < -1000 ? 0.0 : __hiloint2double((1023 + e + (large >> j & 1) * 8) << 20, 0);
                const double fy = e < -1000 ? 0.0 : __hiloint2double((1023 + e + (large >> (C::HN + j) & 1) * 8) << 20, 0);
                double2 s = fresh ? make_double2(0, 0) : make_double2(sm.sum[j][r], sm.sum[C::HN + j][r]);
                s.x = fma((double)y[j], fx, s.x);
                s.y = fma((double)y[C::HN + j], fy, s.y);
                if (end) {
                    out[j * DG_M] = s;
                } else {
                    sm.sum[j][r] = s.x;
                    sm.sum[C::HN + j][r] = s.y;
                }
            }
            fresh = end;
        }
    }
    __syncwarp();
    DG_FENCE_BEFORE;
    __syncthreads();
    if (warp == 2) {
        DG_FENCE_AFTER;
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// Y = the pieces of every row added in CTA order, times the powers of two.  Grid (blocks of rows, vectors).
struct DgFinish {
    DgArgs a;
    int ctas, hn;
};
constexpr int DG_FT = 128;
__global__ void __launch_bounds__(DG_FT) dg_finish_kernel(DgFinish f) {
    const DgArgs& a = f.a;
    const int row = blockIdx.x * DG_FT + threadIdx.x, r = blockIdx.y, lane = threadIdx.x & 31;
    const int nch = (a.nkb + DG_STEPS - 1) / DG_STEPS;
    const int tile = min(row, a.m - 1) / DG_M, first = dg_first_cta(a.stages, f.ctas, a.nkb, tile);
    inputs_ready();
    int ev = DG_NONE;
    for (int u = lane; u < nch; u += 32) ev = max(ev, a.ve[(int64_t)r * nch + u]);
    ev = warp_max(ev);
    if (row >= a.m) return;
    double x = 0, y = 0;
    for (int p = 0; p < a.pieces; p++) {
        if (first + p >= f.ctas || dg_first_stage(a.stages, f.ctas, first + p) >= (tile + 1) * a.nkb) break;
        const double2 v = a.part[((int64_t)(tile * a.pieces + p) * f.hn + r) * DG_M + row % DG_M];
        x += v.x;
        y += v.y;
    }
    const int er = a.rowm[row];
    if (er == DG_BAD || ev == DG_BAD) x = y = __longlong_as_double(0x7ff8000000000000ll);
    else if (er == DG_NONE || ev == DG_NONE) x = y = 0;
    else {
        const int e = er + ev + 4 - 14 - 49;  // both operands below 2^-2 of their scale, first digits 2^-7 each
        x = ldexp(x, e);
        y = ldexp(y, e);
    }
    a.Y[(int64_t)r * a.m + row] = make_double2(x, y);
}

// ----------------------------------------------------------------- host side

int64_t digits_kpad(int64_t n) { return (n + DG_K - 1) / DG_K * DG_K; }
int64_t digits_mpad(int64_t n) { return (n + DG_M - 1) / DG_M * DG_M; }
// bytes of a matrix (as complex128 with leading dimension kpad, then as digits in the same place)
size_t digits_bytes(int64_t n) { return (size_t)digits_mpad(n) * digits_kpad(n) * 16; }
static int64_t dg_units(int64_t n) { return (n + DG_UNIT - 1) / DG_UNIT; }
// ... and of its exponents: columns [kpad], rows [mpad], rows of each unit [units][mpad]
size_t digits_exp_bytes(int64_t n) { return (size_t)(digits_kpad(n) + digits_mpad(n) * (1 + dg_units(n))) * sizeof(int); }

constexpr int DG_TILES = 2;  // row tiles converted at a time
static int dg_hn(int64_t R) { return R <= 8 ? 8 : 16; }
// CTAs of a product: every one a run of equal length, at least two stages for
// up to eight vectors and four for more, whose pieces are dearer (N = 1,284, 16
// vectors: 48 us with runs of three stages, 38 us with four, 39 us with eight).
static int dg_ctas(int stages, int hn) { return std::max(1, std::min(DG_CTAS, stages / (hn == 8 ? 2 : 4))); }
static int dg_pieces(int stages, int nkb, int hn) {
    const int q = stages / dg_ctas(stages, hn);  // a CTA holds q or q + 1 stages
    return (nkb + q - 1) / q + 1;
}
// scratch of a product of R vectors (B operand, exponents, pieces), and of the conversion
size_t digits_work_bytes(int64_t n, int64_t R) {
    const int hn = dg_hn(R);
    const int nkb = (int)(digits_kpad(n) / DG_K), tiles = (int)(digits_mpad(n) / DG_M), stages = tiles * nkb;
    return (size_t)nkb * 2 * DG * 2 * hn * DG_K * 2 + (size_t)tiles * dg_pieces(stages, nkb, hn) * hn * DG_M * 16 +
           16 * (size_t)dg_units(n) * sizeof(int);
}
size_t digits_convert_bytes(int64_t n) { return (size_t)DG_TILES * DG_M * digits_kpad(n) * 16; }

#define DCK(expr)                                                                                        \
    do {                                                                                                 \
        cudaError_t e_ = (expr);                                                                         \
        if (e_ != cudaSuccess) return ctx->fail(BEM_ERR_CUDA, std::string("digits: ") + cudaGetErrorString(e_)); \
    } while (0)

// Complex128 matrix A (n x n in a buffer of digits_bytes, leading dimension
// digits_kpad) -> digits in place; exps: device, digits_exp_bytes.
int digits_prepare(bem_ctx* ctx, double2* A, int64_t n, int* exps) {
    const int64_t kpad = digits_kpad(n), mpad = digits_mpad(n), nkb = kpad / DG_K;
    int rc;
    uint8_t* tmp = (uint8_t*)ctx->dalloc(digits_convert_bytes(n), &rc);
    if (rc) return rc;
    int* col = exps;
    int* row = exps + kpad;
    std::vector<int> none((size_t)kpad, DG_NONE);
    DCK(cudaMemcpyAsync(col, none.data(), kpad * sizeof(int), cudaMemcpyHostToDevice, ctx->stream));
    DCK(cudaStreamSynchronize(ctx->stream));
    const int64_t rows_per = 256;
    dg_colexp_kernel<<<dim3((unsigned)((n + 127) / 128), (unsigned)((n + rows_per - 1) / rows_per)), 128, 0, ctx->stream>>>(
        A, n, kpad, rows_per, col);
    DCK(cudaGetLastError());
    ctx->launches += 1;
    for (int64_t r0 = 0; r0 < mpad; r0 += DG_TILES * DG_M) {
        const int64_t rows = std::min<int64_t>(DG_TILES * DG_M, mpad - r0);
        dg_digits_kernel<<<(unsigned)rows, 256, 0, ctx->stream>>>(A, n, kpad, r0, nkb, col, row, row + mpad, mpad, tmp);
        DCK(cudaGetLastError());
        DCK(cudaMemcpyAsync(A + r0 * kpad, tmp, (size_t)rows * kpad * 16, cudaMemcpyDeviceToDevice, ctx->stream));
        ctx->launches += 1;
    }
    DCK(cudaStreamSynchronize(ctx->stream));
    ctx->dfree(tmp);
    return BEM_OK;
}

template <int NC>
static cudaError_t launch_digits(const DgArgs& a, unsigned ctas, cudaStream_t s) {
    constexpr size_t smem = sizeof(typename DgCfg<NC>::Smem) + 1024;
    static const cudaError_t attr_e =
        cudaFuncSetAttribute(digits_gemm_kernel<NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (attr_e != cudaSuccess) return attr_e;
    return launch_after(digits_gemm_kernel<NC>, dim3(ctas), DG_WARPS * 32, smem, s, a);
}

// Y [R][n] = A X [R][n] with A as digits (digits_prepare); work: digits_work_bytes(n, min(R, 16)).
int digits_gemm(bem_ctx* ctx, const void* A, const int* exps, int64_t n, const double2* X, int64_t R, double2* Y, void* work) {
    const int64_t kpad = digits_kpad(n), mpad = digits_mpad(n);
    const int hn = dg_hn(R);
    DgArgs a{};
    a.A = (const uint8_t*)A;
    a.nkb = (int)(kpad / DG_K);
    const int tiles = (int)(mpad / DG_M);
    a.stages = tiles * a.nkb;
    const int ctas = dg_ctas(a.stages, hn);
    a.pieces = dg_pieces(a.stages, a.nkb, hn);
    a.m = (int)n;
    a.mpad = mpad;
    a.rowm = exps + kpad;
    a.rowe = a.rowm + mpad;
    a.err = ctx->dev.err;
    uint8_t* b = (uint8_t*)work;
    const size_t bb = (size_t)a.nkb * 2 * DG * 2 * hn * DG_K * 2;
    a.B = b;
    a.part = (double2*)(b + bb);
    int* ve = (int*)(a.part + (size_t)tiles * a.pieces * hn * DG_M);
    a.ve = ve;
    for (int64_t r0 = 0; r0 < R; r0 += hn) {
        const int nr = (int)std::min<int64_t>(hn, R - r0);
        a.R = nr;
        a.Y = Y + r0 * n;
        dg_vector_kernel<<<dim3((unsigned)dg_units(n), (unsigned)hn), DG_UNIT, 0, ctx->stream>>>(X + r0 * n, n, kpad, nr, hn,
                                                                                               exps, ve, b);
        DCK(cudaGetLastError());
        DCK(hn == 8 ? launch_digits<16>(a, (unsigned)ctas, ctx->stream) : launch_digits<32>(a, (unsigned)ctas, ctx->stream));
        const DgFinish f{a, ctas, hn};
        DCK(launch_after(dg_finish_kernel, dim3((unsigned)((n + DG_FT - 1) / DG_FT), (unsigned)nr), DG_FT, 0, ctx->stream, f));
        ctx->launches += 3;
    }
    return BEM_OK;
}

}  // namespace gbem
