// k_gemm.cu -- complex64 matrix x block of vectors on the 5th-generation
// tensor cores (tcgen05), split BF16 with FP32 accumulation.
//
// Y = A X with A (m x k) and X (k x n) complex.  Each real plane P of A and
// of X is split into three BF16 numbers, P ~ P0 + P1 + P2 with
// P0 = bf16(P), P1 = bf16(P - P0), P2 = bf16(P - P0 - P1), and the product
// keeps the six terms Pi Qj with i + j <= 2 (everything down to ~2^-24 of
// the product, FP32 level).  A two-term split (three products, ~2^-17 per
// term) is not enough for the oscillatory high-frequency operators: its
// per-term error is amplified by the cancellation in A x (measured 1.2e-4
// on the 0.5 MHz rib scene against 2e-6 for the FP32 matrix-free path).
//
// The complex product is two real GEMMs sharing the B operand
// B = [X_re | X_im] (k x 2n):  C1 = A_re B,  C2 = A_im B, then
//   Y_re = C1[:, :n] - C2[:, n:],   Y_im = C1[:, n:] + C2[:, :n].
// A unit of work is a 128-row tile of A times a GN-column tile of B over 256
// of K; C1 and C2 are two 128 x GN FP32 accumulators in tensor memory,
// double-buffered.  GN = 32 (up to 16 right-hand sides, real and imaginary
// parts) or 128 (64 right-hand sides).  Operands stream in by TMA (64-byte
// swizzle, K-major, 32 of K per stage) through a ring of 216 KB; one thread
// issues the MMAs and commits each stage back to the producer.
//
// Up to 64 right-hand sides the product is bound by reading the 12 N^2 bytes
// of A once, so every SM has to stream all the time: each of 152 CTAs takes
// an equal, contiguous range of units (tile-major), crossing tile borders, and
// the pieces of a tile that several CTAs share are summed in CTA order by
// gemm_finish_kernel.  One CTA per tile left SMs idle (165 tiles on 152 SMs
// are two waves, 65 tiles use 65 SMs): N = 21,016, 16 right-hand sides took
// 1,364 us against 774 us (12 N^2 bytes at 6.85 TB/s), N = 8,200
// 258 us against 132 us.  With more right-hand sides the
// tensor cores bind it, and one CTA per tile over all of K (column tiles
// fastest) lets the column tiles of a row share A through L2.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <string>

#include "ctx.h"
#include "internal.h"

namespace gbem {

constexpr int GM = 128;                       // rows of A per CTA
constexpr int GK = 32;                        // k per stage (64 bytes of bf16, 64-byte swizzle)
constexpr int NSPLIT = 3;                     // BF16 terms per real number
constexpr int TILE_BYTES = GM * GK * 2;       // 8 KB per A operand tile
constexpr int A_TILES = 2 * NSPLIT;           // A re (3 terms), A im (3 terms)
constexpr int GEMM_THREADS = 192;             // warp 0 TMA, warp 1 MMA, warps 2-5 accumulate / epilogue
constexpr int KCH_STAGES = 8;                 // stages per accumulation chunk (K = 256)
constexpr int GEMM_CTAS = 152;                // CTAs of a split product: one per SM

template <int GN>
struct GemmCfg {
    static constexpr int HN = GN / 2;                 // right-hand sides per column tile
    static constexpr int BT_BYTES = GN * GK * 2;      // bytes per B operand tile
    static constexpr int STAGE_BYTES = A_TILES * TILE_BYTES + NSPLIT * BT_BYTES;
    static constexpr int STAGES = 216 * 1024 / STAGE_BYTES;
    static constexpr uint32_t TMEM_COLS = 4 * GN;     // two buffers of C1 | C2
    // instruction descriptor, kind::f16: BF16 A and B, FP32 D, both K-major, M = 128, N = GN
    static constexpr uint32_t IDESC =
        (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(GN >> 3) << 17) | ((uint32_t)(GM >> 4) << 24);
    struct Smem {
        alignas(1024) uint8_t stage[STAGES][STAGE_BYTES];
        uint64_t full[STAGES];
        uint64_t empty[STAGES];
        uint64_t accf[2];   // chunk accumulated in TMEM buffer b (MMA commit)
        uint64_t acce[2];   // TMEM buffer b drained (4 epilogue warps)
        uint32_t tmem_base;
    };
    static_assert(STAGE_BYTES % 1024 == 0 && sizeof(Smem) + 1024 <= 227 * 1024, "gemm smem");
};

__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void g_mbar_init(uint64_t* b, uint32_t n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s_u32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void g_mbar_expect_tx(uint64_t* b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s_u32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint32_t g_mbar_try(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(s_u32(b)), "r"(parity)
        : "memory");
    return ok;
}
// Bounded wait (about a second); on timeout raise the error flag and return false.
__device__ __forceinline__ bool g_mbar_wait(uint64_t* b, uint32_t parity, int* err) {
    if (g_mbar_try(b, parity)) return true;
    if (*(volatile int*)err) return false;  // an earlier wait already gave up: do not wait again
    const long long t0 = clock64();
    while (!g_mbar_try(b, parity)) {
        if (clock64() - t0 > (1ll << 31)) {
            atomicExch(err, 2);
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ void tma_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
            "r"(s_u32(dst)),
        "l"(map), "r"(x), "r"(y), "r"(s_u32(bar))
        : "memory");
}

// Shared-memory matrix descriptor: K-major operand, 64-byte swizzle, rows of
// 64 bytes, 8-row groups 512 bytes apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);           // start address
    d |= (uint64_t)1 << 16;                          // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(512 >> 4) << 32;                 // stride byte offset: 8 rows x 64 B
    d |= (uint64_t)1 << 46;                          // descriptor version
    d |= (uint64_t)4 << 61;                          // 64-byte swizzle
    return d;
}

__device__ __forceinline__ void mma_bf16(uint32_t idesc, uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(s_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = __uint_as_float(r[i]);
}

// The tensor cores accumulate FP32 with truncation, so a long K sum drifts
// by ~K x 2^-24 relative.  The MMAs therefore accumulate only KCH_STAGES*GK
// of K in tensor memory (two buffers, double-buffered); four epilogue warps
// drain each chunk into round-to-nearest FP32 registers.
//
// Unit u = tile * nch + chunk, tile = row tile * n_ct + column tile; CTA b
// takes units [units b / CTAs, units (b + 1) / CTAs).  part != null: each
// CTA's sum over its units of a tile goes to part[tile][piece][rhs][128]
// (piece: the CTA's place among those of the tile); else (whole tiles per CTA)
// straight to Y or Y64.
struct GemmArgs {
    int64_t mpad, nbpad;
    int kblocks, m, n_rhs, n_ct, nch, pieces, units;
    float2* Y;
    double2* Y64;
    float2* part;
    int* err;
};

__host__ __device__ inline int gemm_first_unit(int units, int ctas, int b) { return (int)((int64_t)units * b / ctas); }
// the first of the CTAs that hold units of `tile`
__host__ __device__ inline int gemm_first_cta(int units, int ctas, int nch, int tile) {
    const int u = tile * nch;
    int b = (int)((int64_t)u * ctas / units);
    while (b + 1 < ctas && gemm_first_unit(units, ctas, b + 1) <= u) b++;
    while (b > 0 && gemm_first_unit(units, ctas, b) > u) b--;
    return b;
}

template <int GN>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
    gemm_bf16x3_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmArgs a) {
    typedef GemmCfg<GN> C;
    constexpr int GSTAGES = C::STAGES, HN = C::HN;
    extern __shared__ uint8_t smem_raw[];
    typename C::Smem& sm =
        *reinterpret_cast<typename C::Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int u0 = gemm_first_unit(a.units, gridDim.x, blockIdx.x), u1 = gemm_first_unit(a.units, gridDim.x, blockIdx.x + 1);
    int* const err = a.err;

    if (threadIdx.x == 0) {
        for (int s = 0; s < GSTAGES; s++) {
            g_mbar_init(&sm.full[s], 1);
            g_mbar_init(&sm.empty[s], 1);
        }
        for (int b = 0; b < 2; b++) {
            g_mbar_init(&sm.accf[b], 1);
            g_mbar_init(&sm.acce[b], 4);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_u32(&sm.tmem_base)),
                     "r"(C::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = sm.tmem_base;

    if (warp == 0) {
        if (lane == 0) {
            // producer: the stages of all units one after another
            int s = 0;
            uint32_t ph = 1;  // parity of the ring's previous round (the first wait on a fresh barrier passes)
            bool ok = true;
            for (int u = u0; u < u1 && ok; u++) {
                const int tile = u / a.nch;
                const int c = u - tile * a.nch;
                const int m0 = tile / a.n_ct * GM, b0 = tile % a.n_ct * GN;
                const int ke = min(a.kblocks, (c + 1) * KCH_STAGES);
                for (int kb = c * KCH_STAGES; kb < ke; kb++) {
                    if (!(ok = g_mbar_wait(&sm.empty[s], ph, err))) break;
                    uint8_t* st = sm.stage[s];
                    g_mbar_expect_tx(&sm.full[s], C::STAGE_BYTES);
                    const int kx = kb * GK;
                    for (int pl = 0; pl < A_TILES; pl++)
                        tma_2d(st + pl * TILE_BYTES, &tmA, kx, (int)(pl * a.mpad + m0), &sm.full[s]);
                    for (int pl = 0; pl < NSPLIT; pl++)
                        tma_2d(st + A_TILES * TILE_BYTES + pl * C::BT_BYTES, &tmB, kx, (int)(pl * a.nbpad + b0), &sm.full[s]);
                    if (++s == GSTAGES) {
                        s = 0;
                        ph ^= 1;
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // MMA issuer: per unit, buffer b: C1 (cols 2 GN b ...) = A_re B,
            // C2 (cols 2 GN b + GN ...) = A_im B, each as the six products A_i B_j, i + j <= 2
            bool ok = true;
            int s = 0;
            uint32_t ph = 0;
            for (int u = u0; u < u1 && ok; u++) {
                const int c = u % a.nch, cc = u - u0, buf = cc & 1;
                const uint32_t acc_base = tmem + (uint32_t)(buf * 2 * GN);
                if (cc >= 2) {
                    ok = g_mbar_wait(&sm.acce[buf], (uint32_t)(((cc >> 1) - 1) & 1), err);
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                }
                const int kb0 = c * KCH_STAGES, ke = min(a.kblocks, kb0 + KCH_STAGES);
                for (int kb = kb0; kb < ke && ok; kb++) {
                    if (!(ok = g_mbar_wait(&sm.full[s], ph, err))) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t base = s_u32(sm.stage[s]);
#pragma unroll
                    for (int kk = 0; kk < GK / 16; kk++) {
                        const uint32_t off = kk * 32;
                        uint64_t ar[NSPLIT], ai[NSPLIT], bd[NSPLIT];
#pragma unroll
                        for (int t = 0; t < NSPLIT; t++) {
                            ar[t] = smem_desc(base + t * TILE_BYTES + off);
                            ai[t] = smem_desc(base + (NSPLIT + t) * TILE_BYTES + off);
                            bd[t] = smem_desc(base + A_TILES * TILE_BYTES + t * C::BT_BYTES + off);
                        }
                        const uint32_t acc = (kb > kb0 || kk > 0) ? 1u : 0u;
#pragma unroll
                        for (int h = 0; h < 2; h++) {
                            const uint64_t* A = h ? ai : ar;
                            const uint32_t d = acc_base + h * GN;
                            mma_bf16(C::IDESC, d, A[0], bd[0], acc);
                            mma_bf16(C::IDESC, d, A[0], bd[1], 1u);
                            mma_bf16(C::IDESC, d, A[1], bd[0], 1u);
                            mma_bf16(C::IDESC, d, A[0], bd[2], 1u);
                            mma_bf16(C::IDESC, d, A[1], bd[1], 1u);
                            mma_bf16(C::IDESC, d, A[2], bd[0], 1u);
                        }
                    }
                    mma_commit(&sm.empty[s]);
                    if (++s == GSTAGES) {
                        s = 0;
                        ph ^= 1;
                    }
                }
                if (ok) mma_commit(&sm.accf[buf]);
            }
            // a unit cut short by a timeout still signals its buffer
            if (!ok) {
                mma_commit(&sm.accf[0]);
                mma_commit(&sm.accf[1]);
            }
        }
    } else {
        // accumulate each unit (round-to-nearest FP32); at the end of a tile or of the CTA's range write the sums
        const int q = warp & 3;  // TMEM lane quarter this warp may access
        float yr[HN], yi[HN];
#pragma unroll
        for (int j = 0; j < HN; j++) yr[j] = yi[j] = 0.f;
        for (int u = u0; u < u1; u++) {
            const int tile = u / a.nch;
            const int cc = u - u0, buf = cc & 1;
            g_mbar_wait(&sm.accf[buf], (uint32_t)((cc >> 1) & 1), err);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t lb = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * 2 * GN);
#pragma unroll
            for (int jc = 0; jc < HN; jc += 8) {
                float ta[8], tb[8];
                tmem_ld8(lb + jc, ta);                // A_re X_re
                tmem_ld8(lb + GN + HN + jc, tb);      // A_im X_im
#pragma unroll
                for (int j = 0; j < 8; j++) yr[jc + j] += ta[j] - tb[j];
                tmem_ld8(lb + HN + jc, ta);           // A_re X_im
                tmem_ld8(lb + GN + jc, tb);           // A_im X_re
#pragma unroll
                for (int j = 0; j < 8; j++) yi[jc + j] += ta[j] + tb[j];
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(s_u32(&sm.acce[buf])) : "memory");
            if (u + 1 < u1 && (u + 1) % a.nch != 0) continue;
            const int ct = tile % a.n_ct, r = q * 32 + lane, row = tile / a.n_ct * GM + r;
            if (a.part) {
                const int piece = blockIdx.x - gemm_first_cta(a.units, gridDim.x, a.nch, tile);
                float2* out = a.part + (int64_t)(tile * a.pieces + piece) * HN * GM + r;
#pragma unroll
                for (int j = 0; j < HN; j++)
                    if (ct * HN + j < a.n_rhs) out[j * GM] = make_float2(yr[j], yi[j]);
            } else if (row < a.m) {
#pragma unroll
                for (int j = 0; j < HN; j++) {
                    const int rhs = ct * HN + j;
                    if (rhs >= a.n_rhs) continue;
                    if (a.Y64) a.Y64[(int64_t)rhs * a.m + row] = make_double2(yr[j], yi[j]);
                    else a.Y[(int64_t)rhs * a.m + row] = make_float2(yr[j], yi[j]);
                }
            }
#pragma unroll
            for (int j = 0; j < HN; j++) yr[j] = yi[j] = 0.f;
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 2) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM_COLS) : "memory");
    }
}

// Y = the pieces of every tile summed in CTA order (one column tile: n_rhs <= HN).
__global__ void gemm_finish_kernel(GemmArgs a, int ctas, int hn) {
    const int row = blockIdx.x * blockDim.x + threadIdx.x, rhs = blockIdx.y;
    if (row >= a.m) return;
    const int tile = row / GM;
    const int first = gemm_first_cta(a.units, ctas, a.nch, tile);
    float2 y = make_float2(0.f, 0.f);
    for (int p = 0; p < a.pieces; p++) {
        if (first + p >= ctas || gemm_first_unit(a.units, ctas, first + p) >= (tile + 1) * a.nch) break;
        const float2 v = a.part[((int64_t)(tile * a.pieces + p) * hn + rhs) * GM + row % GM];
        y.x += v.x;
        y.y += v.y;
    }
    if (a.Y64) a.Y64[(int64_t)rhs * a.m + row] = make_double2(y.x, y.y);
    else a.Y[(int64_t)rhs * a.m + row] = y;
}

// x -> three BF16 terms, x ~ t0 + t1 + t2
__device__ __forceinline__ void split3(float x, __nv_bfloat16& t0, __nv_bfloat16& t1, __nv_bfloat16& t2) {
    t0 = __float2bfloat16_rn(x);
    const float r1 = x - __bfloat162float(t0);
    t1 = __float2bfloat16_rn(r1);
    t2 = __float2bfloat16_rn(r1 - __bfloat162float(t1));
}

// A (m x k, complex64 row-major) -> bf16 planes [re0, re1, re2, im0, im1, im2][mpad][kpad], zero padded
__global__ void split_a_kernel(const float2* A, int64_t m, int64_t k, int64_t mpad, int64_t kpad, __nv_bfloat16* P) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= mpad * kpad) return;
    const int64_t r = idx / kpad, c = idx % kpad;
    float2 v = make_float2(0.f, 0.f);
    if (r < m && c < k) v = A[r * k + c];
    const int64_t plane = mpad * kpad;
    split3(v.x, P[0 * plane + idx], P[1 * plane + idx], P[2 * plane + idx]);
    split3(v.y, P[3 * plane + idx], P[4 * plane + idx], P[5 * plane + idx]);
}

// X (n_rhs x k, complex64 or complex128 rounded to it, rhs-major) -> bf16 planes [t0, t1, t2][nbpad][kpad];
// B row of rhs j, part p (0 re, 1 im) = (j / hn) * 2 hn + p * hn + j % hn.
template <class T>
__global__ void split_x_kernel(const T* X, int64_t n_rhs, int64_t k, int64_t nbpad, int64_t kpad, int hn,
                               __nv_bfloat16* P) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= nbpad * kpad) return;
    const int64_t brow = idx / kpad, c = idx % kpad;
    const int64_t blk = brow / (2 * hn), within = brow % (2 * hn), part = within / hn, j = blk * hn + within % hn;
    float x = 0.f;
    if (j < n_rhs && c < k) {
        const T v = X[j * k + c];
        x = (float)(part ? v.y : v.x);
    }
    split3(x, P[idx], P[nbpad * kpad + idx], P[2 * nbpad * kpad + idx]);
}

// Resolved once (thread-safe static initialisation; contexts on several
// threads share it).
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return (PFN_cuTensorMapEncodeTiled_v12000)p;
        return (PFN_cuTensorMapEncodeTiled_v12000) nullptr;
    }();
    return fn;
}

static bool make_map(CUtensorMap* map, void* base, int64_t rows, int64_t kpad, int box_rows) {
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)kpad, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)kpad * 2};
    cuuint32_t box[2] = {GK, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// Right-hand sides per column tile and bytes of scratch (X planes, then the
// pieces of a split product) for n_rhs right-hand sides.
static int gemm_hn(int64_t n_rhs) { return n_rhs <= 16 ? 16 : 64; }
static int gemm_pieces(int64_t units, int64_t ctas, int nch) {
    const int q = (int)(units / ctas);  // a CTA holds q or q + 1 units
    return (nch + q - 1) / q + 1;
}
size_t gemm_work_bytes(int64_t mpad, int64_t kpad, int64_t n_rhs) {
    const int hn = gemm_hn(n_rhs);
    const int64_t nbpad = (n_rhs + hn - 1) / hn * 2 * hn;
    size_t b = (size_t)NSPLIT * nbpad * kpad * 2;
    if (n_rhs <= hn) {
        const int nch = (int)((kpad / GK + KCH_STAGES - 1) / KCH_STAGES);
        const int64_t units = mpad / GM * nch, ctas = std::min<int64_t>(GEMM_CTAS, units);
        b = (b + 15) / 16 * 16 + (size_t)(mpad / GM) * gemm_pieces(units, ctas, nch) * hn * GM * sizeof(float2);
    }
    return b;
}

template <int GN>
static cudaError_t launch_gemm(const CUtensorMap& ta, const CUtensorMap& tb, const GemmArgs& a, unsigned ctas, cudaStream_t s) {
    constexpr size_t smem = sizeof(typename GemmCfg<GN>::Smem) + 1024;
    static const cudaError_t attr_e =
        cudaFuncSetAttribute(gemm_bf16x3_kernel<GN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (attr_e != cudaSuccess) return attr_e;
    gemm_bf16x3_kernel<GN><<<ctas, GEMM_THREADS, smem, s>>>(ta, tb, a);
    return cudaGetLastError();
}

// Planes of A are kept by the caller (they are the assembled operator); X
// is split per call into work (gemm_work_bytes).  X is complex64 (X) or
// complex128 (X64), and Y (n_rhs x m) = A X likewise.
int gemm_bf16x3(bem_ctx* ctx, const __nv_bfloat16* Aplanes, int64_t m, int64_t k, int64_t mpad, int64_t kpad,
                const float2* X, const double2* X64, int64_t n_rhs, float2* Y, double2* Y64, void* work) {
    const int hn = gemm_hn(n_rhs);
    const int64_t nbpad = (n_rhs + hn - 1) / hn * 2 * hn;
    __nv_bfloat16* xplanes = (__nv_bfloat16*)work;
    CUtensorMap ta, tb;
    if (!make_map(&ta, (void*)Aplanes, A_TILES * mpad, kpad, GM) || !make_map(&tb, (void*)xplanes, NSPLIT * nbpad, kpad, 2 * hn))
        return ctx->fail(BEM_ERR_CUDA, "cuTensorMapEncodeTiled failed");
    const int64_t nx = nbpad * kpad;
    const unsigned nbx = (unsigned)((nx + 255) / 256);
    if (X64) split_x_kernel<<<nbx, 256, 0, ctx->stream>>>(X64, n_rhs, k, nbpad, kpad, hn, xplanes);
    else split_x_kernel<<<nbx, 256, 0, ctx->stream>>>(X, n_rhs, k, nbpad, kpad, hn, xplanes);
    GemmArgs a{};
    a.mpad = mpad; a.nbpad = nbpad; a.kblocks = (int)(kpad / GK); a.m = (int)m; a.n_rhs = (int)n_rhs;
    a.n_ct = (int)(nbpad / (2 * hn));
    a.nch = (a.kblocks + KCH_STAGES - 1) / KCH_STAGES;
    a.units = (int)(mpad / GM * a.n_ct * a.nch);
    a.Y = Y; a.Y64 = Y64; a.err = ctx->dev.err;
    const bool split = a.n_ct == 1;
    int64_t ctas = mpad / GM * a.n_ct;  // whole tiles
    if (split) {
        ctas = std::min<int64_t>(GEMM_CTAS, a.units);
        a.pieces = gemm_pieces(a.units, ctas, a.nch);
        a.part = (float2*)((char*)work + ((size_t)NSPLIT * nx * 2 + 15) / 16 * 16);
    }
    cudaError_t e = hn == 16 ? launch_gemm<32>(ta, tb, a, (unsigned)ctas, ctx->stream)
                             : launch_gemm<128>(ta, tb, a, (unsigned)ctas, ctx->stream);
    ctx->launches += 2;
    if (e == cudaSuccess && split) {
        gemm_finish_kernel<<<dim3((unsigned)((m + 255) / 256), (unsigned)n_rhs), 256, 0, ctx->stream>>>(a, (int)ctas, hn);
        ctx->launches++;
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return ctx->fail(BEM_ERR_CUDA, std::string("gemm launch: ") + cudaGetErrorString(e));
    return BEM_OK;
}

int gemm_a_planes() { return A_TILES; }
int gemm_k_align() { return GK; }

int split_a(bem_ctx* ctx, const float2* A, int64_t m, int64_t k, int64_t mpad, int64_t kpad, __nv_bfloat16* P) {
    const int64_t n = mpad * kpad;
    split_a_kernel<<<(unsigned)((n + 255) / 256), 256, 0, ctx->stream>>>(A, m, k, mpad, kpad, P);
    ctx->launches++;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return ctx->fail(BEM_ERR_CUDA, std::string("split_a: ") + cudaGetErrorString(e));
    return BEM_OK;
}

}  // namespace gbem

using namespace gbem;

// Test/utility entry: Y = A X for device complex64 arrays (see bem.h).
extern "C" int bem_zgemm_bf16x3(bem_ctx* ctx, int64_t m, int64_t k, int64_t n_rhs, const void* A, const void* X,
                                void* Y) {
    if (!ctx) return BEM_ERR_INVALID_ARG;
    if (m < 1 || k < 1 || n_rhs < 1 || !A || !X || !Y) return ctx->fail(BEM_ERR_INVALID_ARG, "bad gemm arguments");
    if (cudaSetDevice(ctx->device) != cudaSuccess) return ctx->fail(BEM_ERR_CUDA, "cudaSetDevice");
    if (!ctx->dev.err) {
        int rc;
        ctx->dev.err = (int*)ctx->dalloc(sizeof(int), &rc);
        if (rc) return rc;
        cudaMemsetAsync(ctx->dev.err, 0, sizeof(int), ctx->stream);
    }
    const int64_t mpad = (m + GM - 1) / GM * GM, kpad = (k + GK - 1) / GK * GK;
    int rc;
    __nv_bfloat16* ap = (__nv_bfloat16*)ctx->dalloc((size_t)A_TILES * mpad * kpad * 2, &rc);
    if (rc) return rc;
    void* work = ctx->dalloc(gemm_work_bytes(mpad, kpad, n_rhs), &rc);
    if (rc) { ctx->dfree(ap); return rc; }
    rc = split_a(ctx, (const float2*)A, m, k, mpad, kpad, ap);
    if (!rc) rc = gemm_bf16x3(ctx, ap, m, k, mpad, kpad, (const float2*)X, nullptr, n_rhs, (float2*)Y, nullptr, work);
    cudaStreamSynchronize(ctx->stream);
    ctx->dfree(ap);
    ctx->dfree(work);
    if (!rc) rc = ctx->check_device_error();
    return rc;
}
