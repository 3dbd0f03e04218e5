// k_farmm.cu -- FP32 far field of several right-hand sides on the tensor cores.
//
// For a target point x and the 192 points y of a source tile the potentials of
// one right-hand side (k_apply.cu) are products of two complex numbers per
// pair, G(x, y) and F(x, y), with densities of the source alone:
//   PV = sum G d1,   PWm = n_x . sum G (n_y d2),   PWc = sum G c,
//   PK' = (n_x . X) sum F d1 - n_x . sum F (g d1),
//   PK  = sum F (h d2) - X . sum F (n_y d2),        X = x - c_source,
// with g the point's offset from its tile's centre, h = n_y . g, d1, d2 the
// weighted psi, phi and c the weighted curl: 7 complex densities for G and 8
// for F.  The one-vector formulation spends 20 of its ~42 packed FP32
// instructions per pair and wavenumber on these sums, and 16 for every
// further right-hand side; here they are a tcgen05 contraction, and the FP32
// and MUFU pipes only evaluate G and F.
//
//  * Precision: every FP32 value is split into two FP16 numbers of 11 bits:
//    densities rounded to the first and the rest rounded to the second (2^-23
//    of the value at most), G and F truncated, which takes fewer instructions,
//    and the rest rounded (2^-22).  Products with FP16 operands are exact in
//    FP32.  Three of the four products are kept, hi hi in one accumulator, the
//    two cross terms in another; the fourth is at most 2^-21 of a term, and of
//    either sign because the densities' second numbers are.  Powers of two bring G and F (by the distance of the tiles)
//    and the densities (by the vector's largest) to 2^8 at most, so that
//    nothing leaves FP16's range and small values keep 2^-33 of the largest.
//    The tensor cores truncate when they accumulate, so an accumulator takes
//    the 24 instructions of one source tile only and is then added to FP32
//    registers, round to nearest.  The normals of a tile are taken in a frame
//    with its mean normal, in which X . n_y does not cancel on flat surfaces.
//  * Tiles that come close (centres nearer than FARMM_SEP times the sum of
//    their radii), where 1/r spans too much, stay with far32m_kernel.
//  * Structure: a CTA holds 128 target points, one wavenumber slot, four
//    right-hand sides, and walks a list of source tiles.  Sixteen warps
//    evaluate G and -F, two source points per packed instruction, and write
//    them to tensor memory as the A operand, 8 points (K = 16: real and
//    imaginary parts) per step, eight buffers; two threads issue
//    A_hi x [B_hi | B_lo] (N = 128) and A_lo x B_hi (N = 64) for G and F; four
//    warps drain the accumulators after every tile.  B (the densities, laid out
//    by farmm_pack_kernel) and the source geometry come by bulk copies through
//    a ring of eight stages of 16 points.
//  * What binds it: issue slots and MUFU of the evaluating warps and the
//    hand-over of operands, about evenly (without the evaluation a step of
//    eight points still takes 400 of its 550 cycles; the tensor pipe itself needs
//    242).  Kidney scene of 12,184 triangles, 16 right-hand sides: far field
//    139.6 ms with far32m_kernel for all pairs of tiles, now 58 + 9 ms (close
//    pairs); relative error against 64 bits on 121-178 tiles 0.9-1.3e-6 (5.4e-6
//    at k r of several hundred; 1.0-1.4e-6 with densities truncated too), before
//    1.5-2.4e-6 (1.3e-5).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "ctx.h"
#include "internal.h"
#include "pair_math.h"

namespace gbem {

constexpr int MM_M = 128;                 // target points per CTA
constexpr int MM_RB = 4;                  // right-hand sides per CTA
constexpr int MM_N = 16 * MM_RB;          // columns of an operand (14 or 16 real sums per right-hand side)
constexpr int MM_SP = 16;                 // source points per stage (two K = 16 steps)
constexpr int MM_TS = TP / MM_SP;         // stages per tile
constexpr int MM_STEPS = TP / 8;          // steps per tile
constexpr int MM_BBYTES = 2 * 2 * MM_N * MM_SP * 2 * 2;  // G and F: hi and lo rows of 32 halves (64 bytes)
constexpr int MM_GBYTES = MM_SP * 16;
constexpr int MM_RING = 8;                // stages
constexpr int MM_ABUF = 8;                // A operands in tensor memory, 32 columns each
constexpr int MM_WG = 4;                  // evaluating warpgroups
constexpr int MM_WARPS = 4 * MM_WG + 7;   // + 4 draining, 1 copying, 2 issuing (G and F)
constexpr int MM_LIST = 256;              // source tiles of a work item, at most
static_assert(MM_STEPS % MM_ABUF == 0 && MM_RING == MM_ABUF, "two rounds of A operands per ring of stages");
static_assert(MM_BBYTES == 16384 && TP % MM_SP == 0 && MM_STEPS % MM_WG == 0 && TP % 32 == 0, "farmm layout");

struct MmSmem {
    alignas(1024) uint8_t b[MM_RING][MM_BBYTES];
    alignas(16) float4 geo[MM_RING][MM_SP];   // pairs: (x_a, x_b, y_a, y_b), (z_a, z_b, |g|^2_a, |g|^2_b)
    float4 tab[MM_LIST][2][2];                // per source tile and target tile: (2D, R_c^2), (R_c, phase, scale, F scale)
    int src[MM_LIST];
    int use[MM_LIST];                         // bit t: target tile t of the block takes this source tile
    int n;
    uint64_t full[MM_RING], empty[MM_RING];   // empty: 8 evaluating warps (geometry) and both MMA warps (B)
    uint64_t tfull[MM_ABUF], tempty[MM_ABUF / 2];  // (A operands are given back two at a time)
    uint64_t dfull[2], dempty[2];             // accumulators of G and of F
    uint32_t tmem;
};
static_assert(sizeof(MmSmem) + 1024 <= 227 * 1024, "farmm smem");

__device__ __forceinline__ uint32_t m_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void m_init(uint64_t* b, uint32_t n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(m_u32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void m_arrive(uint64_t* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(m_u32(b)) : "memory");
}
__device__ __forceinline__ bool m_try(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 100000;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(m_u32(b)), "r"(parity)
        : "memory");
    return ok;
}
// Bounded wait (about a second); on timeout raises the error flag and returns false, as does every later wait.
__device__ __forceinline__ bool m_wait(uint64_t* b, uint32_t parity, int* err) {
    if (m_try(b, parity)) return true;
    if (*(volatile int*)err) return false;
    const long long t0 = clock64();
    while (!m_try(b, parity))
        if (clock64() - t0 > (1ll << 31)) {
            atomicExch(err, 1);
            return false;
        }
    return true;
}
__device__ __forceinline__ void m_bulk(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(m_u32(dst)),
        "l"(src), "r"(bytes), "r"(m_u32(bar))
        : "memory");
}
// B operand: K-major, 64-byte rows in the 64-byte swizzle, 8-row groups 512 bytes apart
__device__ __forceinline__ uint64_t m_desc(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | (uint64_t)1 << 16 | (uint64_t)(512 >> 4) << 32 | (uint64_t)1 << 46 |
           (uint64_t)4 << 61;
}
// D (128 x N, FP32) += A (tensor memory, 128 x 16 FP16) B (N x 16 FP16)
__device__ __forceinline__ void m_mma(uint32_t d, uint32_t a, uint64_t b, uint32_t n, uint32_t accumulate) {
    const uint32_t idesc = (1u << 4) | ((n >> 3) << 17) | ((uint32_t)(MM_M >> 4) << 24);
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(d),
        "r"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void m_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(m_u32(bar)) : "memory");
}
__device__ __forceinline__ void m_st2(uint32_t t, uint32_t a, uint32_t b) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(t), "r"(a), "r"(b));
}
// eight accumulators plus the eight of their cross terms, MM_N columns on
__device__ __forceinline__ void m_ld_sum8(uint32_t t, float (&v)[8]) {
    uint32_t r[8], c[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(t));
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(c[0]), "=r"(c[1]), "=r"(c[2]), "=r"(c[3]), "=r"(c[4]), "=r"(c[5]), "=r"(c[6]), "=r"(c[7])
                 : "r"(t + MM_N));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = __uint_as_float(r[i]) + __uint_as_float(c[i]);
}
#define MM_FENCE_BEFORE asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory")
#define MM_FENCE_AFTER asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory")

// x as hi + lo in FP16, both lanes: hi truncated to 11 bits (exact in FP16), lo rounded
__device__ __forceinline__ void m_split(f2 x, uint32_t& hi, uint32_t& lo) {
    const f2 h = make_float2(__uint_as_float(__float_as_uint(x.x) & 0xffffe000u),
                             __uint_as_float(__float_as_uint(x.y) & 0xffffe000u));
    const f2 l = add2(x, neg2(h));
    const __half2 a = __floats2half2_rn(h.x, h.y), b = __floats2half2_rn(l.x, l.y);
    hi = *reinterpret_cast<const uint32_t*>(&a);
    lo = *reinterpret_cast<const uint32_t*>(&b);
}

__device__ __forceinline__ float mm_reduce_phase(double t) {
    const double two_pi_hi = 6.283185307179586, two_pi_lo = 2.4492935982947064e-16;
    const double n = rint(t * 0.15915494309189535);
    double r = fma(-n, two_pi_hi, t);
    r = fma(-n, two_pi_lo, r);
    return (float)r;
}
// 2^e, e in [-126, 127]
__device__ __forceinline__ float mm_pow2(int e) { return __int_as_float((max(-126, min(127, e)) + 127) << 23); }
// e of the largest power of two with 2^e v <= 2^8 (0 for zero and non-finite v), within +-120
__device__ __forceinline__ int mm_scale_exp(float v) {
    const int b = (int)((__float_as_uint(v) >> 23) & 0xff);
    return b == 0 || b == 0xff ? 0 : max(-120, min(120, 7 - (b - 127)));
}

struct FarMmArgs {
    const float4* pg;       // target points (dx, dy, dz, w)
    const float4* tg;       // triangles (n, h)
    const double4* tc;      // tile centres and radii
    const int* tdom;
    const int2* dom_tiles;
    const double2* kdom;
    double2 k0;
    const float* frame;     // [n_tiles][9] rows: two tangents and the mean normal of a tile
    const uint32_t* near;   // [n_tiles][near_words] bit s of row t: the pair (t, s) is close
    int near_words;
    const float4* geo;      // [n_pts] source geometry (MmSmem::geo)
    const int* perm;        // [n_slots] the slot of partial that each slot of these tiles is
    const uint8_t* B;       // [groups][n_tiles][MM_TS][MM_BBYTES]
    const float* unscale;   // [R][3] 1 / scale of d1, d2 and the curls of a vector
    float rho;              // power of two at or above every tile's radius
    int n_tiles, chunk_tiles, R;
    int64_t n_pts, rstride;
    float* partial;         // [R][n_chunks][2][NCOMP][n_pts]
    int* err;
    const int4* work;       // (block, chunk, slot, group)
};

// G and -F of a warp's 32 targets against the eight points of one step, into the A operand at ta.
template <bool LOSSY>
__device__ __forceinline__ void mm_eval(const float4* geo, uint32_t ta, f2 m2x, f2 m2y, f2 m2z, f2 cb, f2 Rc2, f2 Rc, f2 th,
                                        f2 S, f2 SF, f2 kr, f2 nkr, f2 ki, f2 nkil2) {
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const float4 GA = geo[2 * j], GB = geo[2 * j + 1];
        const f2 s = fma2(lo2(GA), m2x, fma2(hi2(GA), m2y, fma2(lo2(GB), m2z, add2(hi2(GB), cb))));
        const f2 r2 = add2(s, Rc2);
        const f2 rinv = make_float2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
        const f2 r = mul2(r2, rinv);
        const f2 den = add2(r, Rc);  // r + R_c
        const f2 rho = mul2(s, make_float2(rcp_approx(den.x), rcp_approx(den.y)));
        const f2 arg = fma2(kr, rho, th);
        f2 sn, cs;
        sincos_approx(arg.x, &sn.x, &cs.x);
        sincos_approx(arg.y, &sn.y, &cs.y);
        f2 a = mul2(rinv, S);
        if constexpr (LOSSY) {
            const f2 e = mul2(nkil2, r);
            a = mul2(make_float2(ex2_approx(e.x), ex2_approx(e.y)), a);
        }
        const f2 Gr = mul2(a, cs), Gi = mul2(a, sn);
        const f2 rs = mul2(rinv, SF);
        const f2 B = mul2(kr, rs), nB = mul2(nkr, rs);
        const f2 P = LOSSY ? fma2(ki, rs, mul2(rs, rinv)) : mul2(rs, rinv);
        const f2 nFr = fma2(P, Gr, mul2(B, Gi));
        const f2 nFi = fma2(P, Gi, mul2(nB, Gr));
        uint32_t h0, l0, h1, l1;
        m_split(Gr, h0, l0);
        m_split(Gi, h1, l1);
        m_st2(ta + 2 * j, h0, h1);
        m_st2(ta + 8 + 2 * j, l0, l1);
        m_split(nFr, h0, l0);
        m_split(nFi, h1, l1);
        m_st2(ta + 16 + 2 * j, h0, h1);
        m_st2(ta + 24 + 2 * j, l0, l1);
    }
}

__global__ void __launch_bounds__(MM_WARPS * 32, 1) farmm_kernel(const FarMmArgs A) {
    extern __shared__ uint8_t smem_raw[];
    MmSmem& sm = *reinterpret_cast<MmSmem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int4 w = A.work[blockIdx.x];
    const int64_t p0 = (int64_t)w.x * MM_M;
    const int slot = w.z, grp = w.w;
    const int t0 = (int)(p0 / TP), t1 = min(A.n_tiles - 1, (int)((p0 + MM_M - 1) / TP));  // the block's target tiles
    const int sb = w.y * A.chunk_tiles, se = min(sb + A.chunk_tiles, A.n_tiles);

    // source tiles that either target tile takes: not close, for slot 1 of the target's domain
    if (warp == 0) {
        int n = 0;
        for (int s0 = sb; s0 < se; s0 += 32) {
            const int s = s0 + lane;
            int u = 0;
            if (s < se)
                for (int t = 0; t < 2; t++) {
                    const int tt = t ? t1 : t0;
                    if (t && t1 == t0) continue;
                    const int2 dr = A.dom_tiles[A.tdom[tt]];
                    const bool close = (A.near[(int64_t)tt * A.near_words + (s >> 5)] >> (s & 31)) & 1;
                    if (!close && (!slot || (s >= dr.x && s < dr.y))) u |= 1 << t;
                }
            const uint32_t m = __ballot_sync(0xffffffffu, u != 0);
            if (u) {
                const int at = n + __popc(m & ((1u << lane) - 1));
                sm.src[at] = s;
                sm.use[at] = u;
            }
            n += __popc(m);
        }
        if (lane == 0) sm.n = n;
    }
    if (tid == 32) {
        for (int s = 0; s < MM_RING; s++) {
            m_init(&sm.full[s], 1);
            m_init(&sm.empty[s], 10);
        }
        for (int b = 0; b < MM_ABUF; b++) m_init(&sm.tfull[b], 4);
        for (int b = 0; b < MM_ABUF / 2; b++) m_init(&sm.tempty[b], 2);
        for (int f = 0; f < 2; f++) {
            m_init(&sm.dfull[f], 1);
            m_init(&sm.dempty[f], 4);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(m_u32(&sm.tmem)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    MM_FENCE_BEFORE;
    __syncthreads();
    MM_FENCE_AFTER;
    const int n = sm.n;
    const uint32_t tmem = sm.tmem;     // G hi hi | G cross | F hi hi | F cross, MM_N columns each
    const uint32_t ta = tmem + 256;    // A operands: G hi, G lo, F hi, F lo of 8 columns each

    // per (source tile, target tile): 2D, R_c^2, R_c, the FP64-reduced phase and the powers of two
    for (int i = tid; i < 2 * n; i += MM_WARPS * 32) {
        const int e = i >> 1, t = i & 1, tt = t ? t1 : t0;
        const double4 ct = A.tc[tt], cs = A.tc[sm.src[e]];
        const double2 kk = slot ? A.kdom[A.tdom[tt]] : A.k0;
        const double Dx = ct.x - cs.x, Dy = ct.y - cs.y, Dz = ct.z - cs.z;
        const double R = sqrt(Dx * Dx + Dy * Dy + Dz * Dz);
        // |G| <= 1 / rmin, |F| <= |G| (|k| + 1 / rmin) / rmin
        const float rmin = fmaxf((float)(R - ct.w - cs.w), (float)R * 0.05f), ir = 1.f / rmin;
        const float kabs = fabsf((float)kk.x) + fabsf((float)kk.y);
        const int eg = mm_scale_exp(ir), ef = mm_scale_exp(ir * ir * (kabs + ir));
        sm.tab[e][t][0] = make_float4((float)(2 * Dx), (float)(2 * Dy), (float)(2 * Dz), (float)(R * R));
        sm.tab[e][t][1] = make_float4((float)R, mm_reduce_phase(kk.x * R), mm_pow2(eg), mm_pow2(ef - eg));
    }
    __syncthreads();

    if (warp < 4 * MM_WG) {
        // ---- evaluate: warpgroup g takes the steps g, g + MM_WG, ... (eight points each)
        const int g = warp >> 2, q = warp & 3;
        const int64_t p = p0 + q * 32 + lane;
        const bool live = p0 + q * 32 < A.n_pts;  // (a warp's points lie in one tile)
        const int tt = live ? (int)((p0 + q * 32) / TP) : t0, t = tt == t0 ? 0 : 1;
        const float4 x = live ? A.pg[p] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float dd = x.x * x.x + x.y * x.y + x.z * x.z;
        const double2 kk = slot ? A.kdom[A.tdom[tt]] : A.k0;
        const f2 kr = bc2((float)kk.x), nkr = bc2((float)-kk.x), ki = bc2((float)kk.y);
        const f2 nkil2 = bc2((float)(-kk.y * 1.4426950408889634));
        const bool lossy = kk.y != 0.0;
        const uint32_t lt = ta + ((uint32_t)(q * 32) << 16);
        // a step is handed over after a first look for the next one's buffers: its stores complete meanwhile
        int pb = -1, psr = 0;
        auto hand_over = [&] {
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            MM_FENCE_BEFORE;
            __syncwarp();
            if (lane == 0) {
                m_arrive(&sm.tfull[pb]);
                m_arrive(&sm.empty[psr]);
            }
        };
        for (int i = 0; i < n; i++) {
            const float4 c0 = sm.tab[i][t][0], c1 = sm.tab[i][t][1];
            const bool use = live && ((sm.use[i] >> t) & 1);
            const f2 m2x = bc2(-fmaf(2.f, x.x, c0.x)), m2y = bc2(-fmaf(2.f, x.y, c0.y)), m2z = bc2(-fmaf(2.f, x.z, c0.z));
            const f2 cb = bc2(fmaf(c0.x, x.x, fmaf(c0.y, x.y, fmaf(c0.z, x.z, dd))));
            for (int m = 0; m < MM_STEPS / MM_WG; m++) {
                const int st = i * MM_STEPS + m * MM_WG + g;  // step of the CTA
                const int stage = st >> 1, sr = stage % MM_RING, b = st % MM_ABUF;
                const uint32_t pf = (uint32_t)((stage / MM_RING) & 1), pt = (uint32_t)(((st / MM_ABUF) & 1) ^ 1);
                const bool ready = __all_sync(0xffffffffu, m_try(&sm.full[sr], pf) && m_try(&sm.tempty[b >> 1], pt));
                if (pb >= 0) hand_over();
                if (!ready) {
                    m_wait(&sm.full[sr], pf, A.err);
                    m_wait(&sm.tempty[b >> 1], pt, A.err);
                }
                MM_FENCE_AFTER;
                pb = b;
                psr = sr;
                const uint32_t ab = lt + b * 32;
                const float4* geo = sm.geo[sr] + (st & 1) * 8;
                if (!use) {
#pragma unroll
                    for (int c = 0; c < 32; c += 2) m_st2(ab + c, 0u, 0u);
                } else if (lossy) {
                    mm_eval<true>(geo, ab, m2x, m2y, m2z, cb, bc2(c0.w), bc2(c1.x), bc2(c1.y), bc2(c1.z), bc2(c1.w), kr, nkr,
                                  ki, nkil2);
                } else {
                    mm_eval<false>(geo, ab, m2x, m2y, m2z, cb, bc2(c0.w), bc2(c1.x), bc2(c1.y), bc2(c1.z), bc2(c1.w), kr, nkr,
                                   ki, nkil2);
                }
            }
        }
        if (pb >= 0) hand_over();
    } else if (warp < 4 * MM_WG + 4) {
        // ---- drain: FP32 sums of this thread's target
        const int q = warp & 3;
        const int64_t p = p0 + q * 32 + lane;
        const bool live = p0 + q * 32 < A.n_pts;
        const int tt = live ? (int)((p0 + q * 32) / TP) : t0, t = tt == t0 ? 0 : 1;
        const float4 x = live ? A.pg[p] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 nx = live ? A.tg[p / QP] : make_float4(0.f, 0.f, 0.f, 0.f);
        const uint32_t ld = tmem + ((uint32_t)(q * 32) << 16);
        float acc[MM_RB][NCOMP];
#pragma unroll
        for (int v = 0; v < MM_RB; v++)
#pragma unroll
            for (int c = 0; c < NCOMP; c++) acc[v][c] = 0.f;
        for (int i = 0; i < n; i++) {
            const float4 c0 = sm.tab[i][t][0], c1 = sm.tab[i][t][1];
            const float* fr = A.frame + (int64_t)sm.src[i] * 9;
            const float X[3] = {fmaf(0.5f, c0.x, x.x), fmaf(0.5f, c0.y, x.y), fmaf(0.5f, c0.z, x.z)};  // x - c_source
            const float nX = nx.x * X[0] + nx.y * X[1] + nx.z * X[2];
            float fX[3];  // in the tile's frame
#pragma unroll
            for (int c = 0; c < 3; c++) fX[c] = __ldg(fr + 3 * c) * X[0] + __ldg(fr + 3 * c + 1) * X[1] + __ldg(fr + 3 * c + 2) * X[2];
            const float ug = 1.f / c1.z, uf = -1.f / (c1.z * c1.w);  // powers of two; A holds -F
            m_wait(&sm.dfull[0], (uint32_t)(i & 1), A.err);
            MM_FENCE_AFTER;
#pragma unroll
            for (int v = 0; v < MM_RB; v++) {
                float a[8];
                m_ld_sum8(ld + 16 * v, a);  // d1, n_y d2
                acc[v][0] = fmaf(ug, a[0], acc[v][0]);
                acc[v][1] = fmaf(ug, a[1], acc[v][1]);
                acc[v][6] = fmaf(ug, fmaf(nx.x, a[2], fmaf(nx.y, a[4], nx.z * a[6])), acc[v][6]);
                acc[v][7] = fmaf(ug, fmaf(nx.x, a[3], fmaf(nx.y, a[5], nx.z * a[7])), acc[v][7]);
                m_ld_sum8(ld + 16 * v + 8, a);  // c
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    acc[v][8 + c] = fmaf(ug, a[2 * c], acc[v][8 + c]);
                    acc[v][11 + c] = fmaf(ug, a[2 * c + 1], acc[v][11 + c]);
                }
            }
            MM_FENCE_BEFORE;
            __syncwarp();
            if (lane == 0) m_arrive(&sm.dempty[0]);
            m_wait(&sm.dfull[1], (uint32_t)(i & 1), A.err);
            MM_FENCE_AFTER;
#pragma unroll
            for (int v = 0; v < MM_RB; v++) {
                float a[8];
                m_ld_sum8(ld + 2 * MM_N + 16 * v, a);  // d1, g d1 / rho
#pragma unroll
                for (int c = 0; c < 2; c++)
                    acc[v][4 + c] = fmaf(uf, fmaf(nX, a[c], -A.rho * fmaf(nx.x, a[2 + c], fmaf(nx.y, a[4 + c], nx.z * a[6 + c]))),
                                         acc[v][4 + c]);
                m_ld_sum8(ld + 2 * MM_N + 16 * v + 8, a);  // h d2 / rho, n_y d2 in the frame
#pragma unroll
                for (int c = 0; c < 2; c++)
                    acc[v][2 + c] = fmaf(uf, fmaf(A.rho, a[c], -fmaf(fX[0], a[2 + c], fmaf(fX[1], a[4 + c], fX[2] * a[6 + c]))),
                                         acc[v][2 + c]);
            }
            MM_FENCE_BEFORE;
            __syncwarp();
            if (lane == 0) m_arrive(&sm.dempty[1]);
        }
        if (live) {
#pragma unroll
            for (int v = 0; v < MM_RB; v++) {
                const int r = grp * MM_RB + v;
                if (r >= A.R) break;
                const float u1 = A.unscale[3 * r], u2 = A.unscale[3 * r + 1], u3 = A.unscale[3 * r + 2];
                float* out = A.partial + (int64_t)r * A.rstride + ((int64_t)w.y * 2 + slot) * NCOMP * A.n_pts +
                             (int64_t)A.perm[p / QP] * QP + p % QP;
#pragma unroll
                for (int c = 0; c < NCOMP; c++) {
                    const float u = c < 2 || c == 4 || c == 5 ? u1 : c < 8 ? u2 : u3;
                    out[(int64_t)c * A.n_pts] = acc[v][c] * u;
                }
            }
        }
    } else if (warp == 4 * MM_WG + 4) {
        // ---- copies
        if (lane == 0) {
            bool ok = true;
            for (int i = 0; i < n && ok; i++) {
                const int s = sm.src[i];
                const uint8_t* B = A.B + ((int64_t)grp * A.n_tiles + s) * MM_TS * MM_BBYTES;
                for (int c = 0; c < MM_TS; c++) {
                    const int stage = i * MM_TS + c, sr = stage % MM_RING;
                    if (!(ok = m_wait(&sm.empty[sr], (uint32_t)(((stage / MM_RING) & 1) ^ 1), A.err))) break;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(m_u32(&sm.full[sr])),
                                 "r"(MM_BBYTES + MM_GBYTES)
                                 : "memory");
                    m_bulk(sm.b[sr], B + (int64_t)c * MM_BBYTES, MM_BBYTES, &sm.full[sr]);
                    m_bulk(sm.geo[sr], A.geo + (int64_t)s * TP + c * MM_SP, MM_GBYTES, &sm.full[sr]);
                }
            }
        }
    } else if (lane == 0) {
        // ---- MMA: one warp for G, one for F (a single thread takes 60 to 150 cycles to issue an instruction that
        // runs for 56 to 65, among the evaluating warps).  A full A operand says that its stage of B has landed.
        const int f = warp - (4 * MM_WG + 5);
        const uint32_t d0 = tmem + f * 2 * MM_N, a0 = ta + f * 16;
        const uint64_t bd = m_desc(m_u32(sm.b[0]) + f * (MM_BBYTES / 2));
        bool ok = true;
        uint32_t round = 0;  // of the eight A operands
        for (int i = 0; i < n && ok; i++) {
            if (i > 0) {
                if (!(ok = m_wait(&sm.dempty[f], (uint32_t)((i - 1) & 1), A.err))) break;
                MM_FENCE_AFTER;
            }
            for (int k = 0; k < MM_STEPS && ok; k += MM_ABUF, round++) {
                const int s0 = (int)(round & 1) * (MM_ABUF / 2);  // stage in the ring
                const uint64_t br = bd + (uint64_t)s0 * (MM_BBYTES / 16);
#pragma unroll
                for (int b = 0; b < MM_ABUF; b++) {
                    if (!(ok = m_wait(&sm.tfull[b], round & 1, A.err))) break;
                    MM_FENCE_AFTER;
                    const uint64_t d = br + (b >> 1) * (MM_BBYTES / 16) + (b & 1) * 2;
                    m_mma(d0, a0 + b * 32, d, 2 * MM_N, b > 0 || k > 0);
                    m_mma(d0 + MM_N, a0 + b * 32 + 8, d, MM_N, 1u);
                    if (b & 1) {
                        m_commit(&sm.tempty[b >> 1]);
                        m_commit(&sm.empty[s0 + (b >> 1)]);
                    }
                }
            }
            if (ok) m_commit(&sm.dfull[f]);
        }
    }
    __syncwarp();
    MM_FENCE_BEFORE;
    __syncthreads();
    if (warp == 2) {
        MM_FENCE_AFTER;
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// ----------------------------------------------------------------- the densities as B operands

// largest |d1|, |d2| (components) and |w c| of each vector, as the bits of non-negative floats; grid (blocks, vectors)
__global__ void farmm_max_kernel(const float4* __restrict__ pd, const float4* __restrict__ tcurl, const float4* __restrict__ pg,
                                 int64_t n_pts, int64_t n_slots, uint32_t* __restrict__ out) {
    const int r = blockIdx.y;
    const float4* d = pd + r * n_pts;
    const float4* tc = tcurl + r * 2 * n_slots;
    float m1 = 0.f, m2 = 0.f, m3 = 0.f;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_pts; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 v = d[i];  // pair-interleaved: d1 in the even entries, d2 in the odd ones
        const float m = fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
        if (i & 1) m2 = fmaxf(m2, m);
        else m1 = fmaxf(m1, m);
        const int64_t s = i / QP;
        const float4 a = tc[2 * s], b = tc[2 * s + 1];
        const float c = fmaxf(fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fabsf(a.z)), fmaxf(fmaxf(fabsf(b.x), fabsf(b.y)), fabsf(b.z)));
        m3 = fmaxf(m3, c * pg[i].w);
    }
    for (int o = 16; o > 0; o >>= 1) {
        m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, o));
        m2 = fmaxf(m2, __shfl_xor_sync(0xffffffffu, m2, o));
        m3 = fmaxf(m3, __shfl_xor_sync(0xffffffffu, m3, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&out[3 * r], __float_as_uint(m1));
        atomicMax(&out[3 * r + 1], __float_as_uint(m2));
        atomicMax(&out[3 * r + 2], __float_as_uint(m3));
    }
}

// One CTA per (stage of 16 points, group): thread (point, right-hand side) writes its 30 complex entries, hi and lo,
// as K rows (Gr) and (Gi) of its columns into shared memory in the operand's layout; then the 16 KB go out.
__global__ void __launch_bounds__(64) farmm_pack_kernel(const float4* __restrict__ pd, const float4* __restrict__ tcurl,
                                                        const float4* __restrict__ pg, const float4* __restrict__ tg,
                                                        const float* __restrict__ frame, const uint32_t* __restrict__ mx,
                                                        int64_t n_pts, int64_t n_slots, int R, float rho,
                                                        uint8_t* __restrict__ out, float* __restrict__ unscale) {
    __shared__ __align__(16) uint8_t sb[MM_BBYTES];
    const int64_t stage = blockIdx.x;
    const int grp = blockIdx.y, k = threadIdx.x & 15, v = threadIdx.x >> 4, r = grp * MM_RB + v;
    const int64_t p = stage * MM_SP + k, s = p / QP;
    float col[2][16][2];  // [G, F][column pair][re, im]: 8 complex densities each
#pragma unroll
    for (int f = 0; f < 2; f++)
#pragma unroll
        for (int c = 0; c < 8; c++) col[f][c][0] = col[f][c][1] = 0.f;
    if (r < R) {
        const int e1 = mm_scale_exp(__uint_as_float(mx[3 * r])), e2 = mm_scale_exp(__uint_as_float(mx[3 * r + 1])),
                  e3 = mm_scale_exp(__uint_as_float(mx[3 * r + 2]));
        const float T1 = mm_pow2(e1), T2 = mm_pow2(e2), T3 = mm_pow2(e3);
        if (stage == 0 && k == 0) {
            unscale[3 * r] = mm_pow2(-e1);
            unscale[3 * r + 1] = mm_pow2(-e2);
            unscale[3 * r + 2] = mm_pow2(-e3);
        }
        const float4 D = pair_point(pd + (int64_t)r * n_pts + s * QP, (int)(p - s * QP));
        const float4 g = pg[p], t = tg[s];
        const float4 cr = tcurl[(int64_t)r * 2 * n_slots + 2 * s], ci = tcurl[(int64_t)r * 2 * n_slots + 2 * s + 1];
        const float* fr = frame + (stage / MM_TS) * 9;
        const float d1[2] = {D.x * T1, D.y * T1}, d2[2] = {D.z * T2, D.w * T2};
        const float ir = 1.f / rho, h = t.w * ir, w = g.w * T3;
        const float gg[3] = {g.x * ir, g.y * ir, g.z * ir}, n[3] = {t.x, t.y, t.z};
        const float c[3][2] = {{cr.x * w, ci.x * w}, {cr.y * w, ci.y * w}, {cr.z * w, ci.z * w}};
#pragma unroll
        for (int z = 0; z < 2; z++) {
            col[0][0][z] = d1[z];
            col[1][0][z] = d1[z];
            col[1][4][z] = h * d2[z];
#pragma unroll
            for (int a = 0; a < 3; a++) {
                const float na = fr[3 * a] * n[0] + fr[3 * a + 1] * n[1] + fr[3 * a + 2] * n[2];
                col[0][1 + a][z] = n[a] * d2[z];
                col[0][4 + a][z] = c[a][z];
                col[1][1 + a][z] = gg[a] * d1[z];
                col[1][5 + a][z] = na * d2[z];
            }
        }
    }
    // K of this point within its step of eight: (Gr, Gr, Gi, Gi) per pair of points
    const int kk = k >> 3, pt = k & 7, kre = kk * 16 + (pt >> 1) * 4 + (pt & 1), kim = kre + 2;
    auto put = [&](int row, int kx, __half x) {
        *reinterpret_cast<__half*>(sb + row * 64 + (((kx >> 3) ^ ((row >> 1) & 3)) << 4) + (kx & 7) * 2) = x;
    };
#pragma unroll
    for (int f = 0; f < 2; f++)
#pragma unroll
        for (int c = 0; c < 8; c++)
#pragma unroll
            for (int z = 0; z < 2; z++) {  // output part: re = Gr d.re - Gi d.im, im = Gr d.im + Gi d.re
                const float a = col[f][c][z], b = z ? col[f][c][0] : -col[f][c][1];
                const __half ah = __float2half_rn(a), bh = __float2half_rn(b);
                const int row = f * 2 * MM_N + v * 16 + 2 * c + z;
                put(row, kre, ah);
                put(row, kim, bh);
                put(row + MM_N, kre, __float2half_rn(a - __half2float(ah)));
                put(row + MM_N, kim, __float2half_rn(b - __half2float(bh)));
            }
    __syncthreads();
    uint4* dst = reinterpret_cast<uint4*>(out + ((int64_t)grp * gridDim.x + stage) * MM_BBYTES);
    for (int i = threadIdx.x; i < MM_BBYTES / 16; i += 64) dst[i] = reinterpret_cast<const uint4*>(sb)[i];
}

// ----------------------------------------------------------------- host side

size_t farmm_bytes(int n_tiles, int64_t R) {
    const int64_t groups = (R + MM_RB - 1) / MM_RB;
    return (size_t)groups * n_tiles * MM_TS * MM_BBYTES + (size_t)R * 6 * sizeof(float) + 64;
}

// Source chunks: long enough to amortise a work item's start, within 2 GiB of
// partials where MM_LIST allows.
void farmm_chunking(int n_tiles, int64_t n_pts, int64_t R, int* n_chunks, int* chunk_tiles) {
    const size_t per_chunk = (size_t)R * 2 * NCOMP * n_pts * sizeof(float);
    const int nc_mem = (int)std::max<size_t>(1, ((size_t)2 << 30) / std::max<size_t>(1, per_chunk));
    int nc = std::min((n_tiles + FARMM_CHUNK - 1) / FARMM_CHUNK, nc_mem);
    nc = std::max(nc, (n_tiles + MM_LIST - 1) / MM_LIST);
    const int ct = (n_tiles + nc - 1) / nc;
    *chunk_tiles = ct;
    *n_chunks = (n_tiles + ct - 1) / ct;
}

cudaError_t launch_farmm(const FarMmPlan& P, cudaStream_t s) {
    constexpr size_t smem = sizeof(MmSmem) + 1024;
    static const cudaError_t attr_e = cudaFuncSetAttribute(farmm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (attr_e != cudaSuccess) return attr_e;
    const int groups = (P.R + MM_RB - 1) / MM_RB;
    uint8_t* B = (uint8_t*)P.buf;
    uint32_t* mx = (uint32_t*)(B + (size_t)groups * P.n_tiles * MM_TS * MM_BBYTES);
    float* un = (float*)(mx + 3 * P.R);
    cudaError_t e = cudaMemsetAsync(mx, 0, 3 * P.R * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    farmm_max_kernel<<<dim3((unsigned)std::min<int64_t>(152, (P.n_pts + 255) / 256), (unsigned)P.R), 256, 0, s>>>(
        P.pd, P.tcurl, P.pg, P.n_pts, P.n_slots, mx);
    farmm_pack_kernel<<<dim3((unsigned)(P.n_tiles * MM_TS), (unsigned)groups), 64, 0, s>>>(
        P.pd, P.tcurl, P.pg, P.tg, P.frame, mx, P.n_pts, P.n_slots, P.R, P.rho, B, un);
    FarMmArgs a{};
    a.pg = P.pg; a.tg = P.tg; a.tc = P.tc; a.tdom = P.tdom; a.dom_tiles = P.dom_tiles; a.kdom = P.kdom; a.k0 = P.k0;
    a.frame = P.frame; a.near = P.near; a.near_words = P.near_words; a.geo = P.geo; a.perm = P.perm; a.B = B; a.unscale = un; a.rho = P.rho;
    a.n_tiles = P.n_tiles; a.chunk_tiles = P.chunk_tiles; a.R = P.R; a.n_pts = P.n_pts; a.rstride = P.rstride;
    a.partial = P.partial; a.err = P.err; a.work = P.work;
    if (P.n_work > 0) farmm_kernel<<<(unsigned)P.n_work, MM_WARPS * 32, smem, s>>>(a);
    return cudaGetLastError();
}

int farmm_blocks(int64_t n_pts) { return (int)((n_pts + MM_M - 1) / MM_M); }
int farmm_groups(int64_t R) { return (int)((R + MM_RB - 1) / MM_RB); }

}  // namespace gbem
