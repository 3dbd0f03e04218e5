// k_apply.cu -- matrix-free application of the Galerkin boundary operators.
//
// Paper App. A (eqs. SLP, DLP, ADJDLP, HYP, green_func) and Sec. 2.3 (eq.
// Galerkin_disc_lhs): with G = exp(ikr)/(4 pi r), F = G (ik - 1/r)/r and P1
// trial data phi (Dirichlet) and psi (Neumann), the potentials at a target
// quadrature point x are
//   P_V   = sum_y G       w_y psi(y)                       (single layer)
//   P_K   = sum_y F (y-x).n_y w_y phi(y)                   (double layer)
//   P_K'  = sum_y F (x-y).n_x w_y psi(y)                   (adjoint double layer)
//   P_Wc  = sum_y G w_y curl phi(y),  P_Wm = sum_y G (n_x.n_y) w_y phi(y)
// (the hypersingular operator in its integration-by-parts form), and the
// Galerkin rows follow by testing with the P1 functions at the target
// points.  Per trial triangle t the plane offset (y-x).n_t and n_x.n_t are
// constant, and curl phi is constant, so three per-triangle sums
// S1 = sum F sigma_D, S2 = sum G w, S3 = sum G sigma_D carry K and W.
//
// The FP32 kernel keeps kr accurate for large k|x-y| by reconstructing the
// distance from the tile-pair centre distance R_c (FP64) and a local
// offset: with D = c_target - c_source and delta = dx - dy (tile-local),
//   s = delta.(2D + delta) = r^2 - R_c^2,   r - R_c = s / (r + R_c),
//   phase = (Re k R_c mod 2 pi, FP64) + Re k (r - R_c).
#include <cstdio>
#include <type_traits>

#include "internal.h"
#include "launch.cuh"
#include "pair_math.h"

namespace gbem {

// ----------------------------------------------------------------- helpers

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ uint32_t mbar_try_wait(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(b)), "r"(parity)
        : "memory");
    return ok;
}

// Bulk (TMA) copy global -> shared completing on an mbarrier.  Both
// addresses 16-byte aligned, size a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// Bounded wait: gives up after ~2^31 cycles (about a second), raises the
// device error flag and lets the caller continue on whatever the buffer
// holds, so that every thread still reaches every __syncthreads.
__device__ __forceinline__ void mbar_wait_bounded(uint64_t* b, uint32_t parity, int* err) {
    if (mbar_try_wait(b, parity)) return;
    long long t0 = clock64();
    while (!mbar_try_wait(b, parity)) {
        if (clock64() - t0 > (1ll << 31)) {
            atomicExch(err, 1);
            return;
        }
    }
}

// x - 2 pi round(x / 2 pi) in FP64 (2 pi split in two doubles), as float.
__device__ __forceinline__ float reduce_phase(double t) {
    const double two_pi_hi = 6.283185307179586, two_pi_lo = 2.4492935982947064e-16;
    double n = rint(t * 0.15915494309189535);
    double r = fma(-n, two_pi_hi, t);
    r = fma(-n, two_pi_lo, r);
    return (float)r;
}


// ----------------------------------------------------------------- gather (trial densities)

// One thread per (triangle, rule point): each point takes ~16 FP64
// operations, which GB300 issues at 1/64 of its FP32 rate, so the kernel is
// bound by how many SMs share them (one thread per triangle: 10 us at any
// size up to a few thousand triangles; now 6-7 us, cold caches).  Thread q of a triangle
// also forms one of the six real curl components.
constexpr int GATHER_THREADS = 96;  // 16 triangles
static_assert(GATHER_THREADS % QP == 0 && QP == 6, "six threads per triangle, one curl component each");

__global__ void __launch_bounds__(GATHER_THREADS) gather_kernel(GatherArgs a) {
    dependents_may_start();  // (launched behind everything before it)
    const int64_t i = a.s_begin * QP + (int64_t)blockIdx.x * GATHER_THREADS + threadIdx.x;
    const int64_t s = i / QP;
    const int q = (int)(i - s * QP);
    const bool live = s < a.s_end;
    const int4 v = live ? a.slot_v[s] : make_int4(-1, -1, -1, 0);
    const bool real = v.x >= 0;
    double2 xs[3], xf[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const int vid = k == 0 ? v.x : k == 1 ? v.y : v.z;
        xs[k] = real ? a.x[a.v_dof1[vid]] : make_double2(0, 0);
        xf[k] = real ? a.x[a.v_dof2[vid]] : make_double2(0, 0);
    }
    const double w = real ? a.pt_w[i] : 0.0;
    double sr = 0, si = 0, dr = 0, di = 0;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const double l = a.lam[q][k];
        sr += l * xs[k].x;
        si += l * xs[k].y;
        dr += l * xf[k].x;
        di += l * xf[k].y;
    }
    sr *= w;
    si *= w;
    dr *= w;
    di *= w;
    // curl component c, real (q < 3) or imaginary part
    const int c = q < 3 ? q : q - 3;
    double cu = 0;
    if (real)
#pragma unroll
        for (int k = 0; k < 3; k++) cu += (q < 3 ? xf[k].x : xf[k].y) * a.slot_curl[s * 9 + 3 * k + c];
    if (a.pd32) {
        // pair-interleaved: the even point of a pair writes (x_a, x_b, y_a, y_b), the odd one (z_a, z_b, w_a, w_b)
        const float4 p = make_float4((float)sr, (float)si, (float)dr, (float)di);
        const bool odd = q & 1;
        const float ox = __shfl_xor_sync(0xffffffffu, odd ? p.x : p.z, 1);
        const float oy = __shfl_xor_sync(0xffffffffu, odd ? p.y : p.w, 1);
        if (live) a.pd32[i] = odd ? make_float4(ox, p.z, oy, p.w) : make_float4(p.x, ox, p.y, oy);
    }
    if (!live) return;
    if (a.pd64) a.pd64[i] = make_double4(sr, si, dr, di);
    if (a.tcurl32) {
        float* t = reinterpret_cast<float*>(a.tcurl32 + 2 * s + (q >= 3));
        t[c] = (float)cu;
        if (c == 0) t[3] = 0.f;
    }
    if (a.tcurl64) {
        double* t = reinterpret_cast<double*>(a.tcurl64 + 2 * s + (q >= 3));
        t[c] = cu;
        if (c == 0) t[3] = 0.0;
    }
}

// ----------------------------------------------------------------- FP32 far field
//
// One CTA = one target tile (TP threads, one target point each) against a
// contiguous range of source tiles.  Source tiles stream through an
// NSTAGE-deep ring of shared-memory stages filled by bulk (TMA) copies that
// complete on per-stage mbarriers.  There is no CTA-wide barrier in the
// loop: each warp counts itself out of a stage when it has finished the
// tile in it, and the last warp to leave a stage refills it with the tile
// NSTAGE ahead, so warps drift freely within the ring.

constexpr int NSTAGE = 4;
constexpr int NWARP = TP / 32;

struct __align__(16) Stage {
    float4 pg[TP];      // source points (dx, dy, dz, w), pair-interleaved
    float4 pd[TP];      // densities, pair-interleaved
    float4 tg[TT];      // triangles (n, h)
    float4 tc[2 * TT];  // curl densities
};
constexpr uint32_t STAGE_BYTES = sizeof(Stage);
static_assert(STAGE_BYTES == 7680, "stage layout");

struct FarSmem {
    Stage st[NSTAGE];
    float4 tab[2 * CHUNK_MAX];
    uint64_t full[NSTAGE];
    int cnt[NSTAGE];
};

struct Acc {
    float v[NCOMP];  // PV(2) PK(2) PKp(2) PWm(2) PWc(6)
};

// Source points are processed two at a time, side by side in the two lanes
// of a float2, so that one packed FP32 instruction (FFMA2 / FADD2 / FMUL2)
// advances both.  The points of a triangle are stored pair-interleaved:
// pair j (points 2j and 2j+1) is the float4 (x_a, x_b, y_a, y_b) followed by
// (z_a, z_b, w_a, w_b), for the source geometry (offsets from the tile
// centre and weight) and for the gathered densities (the two complex
// densities in place of x, y and z, w).  The packed helpers are in
// pair_math.h.

// One wavenumber slot, both lanes.
struct PairK {
    f2 kr, th, ki, nkil2;  // Re k, reduced FP64 phase of the tile pair, Im k, -Im k log2(e)
};

// Sums over the points of one tile (V, K') and of one triangle (the rest),
// per lane; they are folded into the chunk's accumulators at the end of
// their tile or triangle.  The K' and K sums are kept with the sign of -F,
// the form in which the gradient factor comes out without a sign flip.
struct PairTile {
    f2 Vr, Vi, nKpr, nKpi;
};
struct PairTri {
    f2 nS1r, nS1i, S2r, S2i, S3r, S3i;
};

// Contribution of two source points at one wavenumber.  With
// (ik - 1/r)/r = A + iB, B = Re k / r, P = -A = Im k / r + 1/r^2, the
// gradient factor is F = G (A + iB), so -Re F = P Gr + B Gi and
// -Im F = P Gi - B Gr.  LOSSY: Im k != 0 (exp(-Im k r) evaluated);
// otherwise the amplitude is 1/r and P = 1/r^2.
template <bool LOSSY>
__device__ __forceinline__ void pair_slot(const PairK& k, f2 rho, f2 r, f2 rinv, f2 rinv2, f2 ndot, f2 w, f2 d1r,
                                          f2 d1i, f2 nd1i, f2 d2r, f2 d2i, f2 nd2i, PairTile& T, PairTri& S) {
    const f2 arg = fma2(k.kr, rho, k.th);
    f2 sn, cs;
    sincos_approx(arg.x, &sn.x, &cs.x);
    sincos_approx(arg.y, &sn.y, &cs.y);
    f2 a = rinv;
    if constexpr (LOSSY) {
        const f2 e = mul2(k.nkil2, r);
        a = mul2(make_float2(ex2_approx(e.x), ex2_approx(e.y)), rinv);
    }
    const f2 Gr = mul2(a, cs), Gi = mul2(a, sn);
    const f2 B = mul2(k.kr, rinv);
    const f2 P = LOSSY ? fma2(k.ki, rinv, rinv2) : rinv2;
    const f2 nFr = fma2(P, Gr, mul2(B, Gi));
    const f2 nFi = fma2(P, Gi, neg2(mul2(B, Gr)));
    T.Vr = fma2(Gr, d1r, fma2(Gi, nd1i, T.Vr));
    T.Vi = fma2(Gr, d1i, fma2(Gi, d1r, T.Vi));
    const f2 nFnr = mul2(ndot, nFr), nFni = mul2(ndot, nFi);
    T.nKpr = fma2(nFnr, d1r, fma2(nFni, nd1i, T.nKpr));
    T.nKpi = fma2(nFnr, d1i, fma2(nFni, d1r, T.nKpi));
    S.nS1r = fma2(nFr, d2r, fma2(nFi, nd2i, S.nS1r));
    S.nS1i = fma2(nFr, d2i, fma2(nFi, d2r, S.nS1i));
    S.S2r = fma2(Gr, w, S.S2r);
    S.S2i = fma2(Gi, w, S.S2i);
    S.S3r = fma2(Gr, d2r, fma2(Gi, nd2i, S.S3r));
    S.S3i = fma2(Gr, d2i, fma2(Gi, d2r, S.S3i));
}

// Per-triangle terms: K through (y-x).n_t, W through curl phi and n_x.n_t.
__device__ __forceinline__ void slot_triangle(float fK, float nn, const float4& cre, const float4& cim,
                                              const PairTri& P, Acc& t) {
    const float nS1r = P.nS1r.x + P.nS1r.y, nS1i = P.nS1i.x + P.nS1i.y;
    const float S2r = P.S2r.x + P.S2r.y, S2i = P.S2i.x + P.S2i.y;
    const float S3r = P.S3r.x + P.S3r.y, S3i = P.S3i.x + P.S3i.y;
    t.v[2] = fmaf(-fK, nS1r, t.v[2]);
    t.v[3] = fmaf(-fK, nS1i, t.v[3]);
    t.v[6] = fmaf(nn, S3r, t.v[6]);
    t.v[7] = fmaf(nn, S3i, t.v[7]);
    t.v[8] = fmaf(S2r, cre.x, fmaf(-S2i, cim.x, t.v[8]));
    t.v[9] = fmaf(S2r, cre.y, fmaf(-S2i, cim.y, t.v[9]));
    t.v[10] = fmaf(S2r, cre.z, fmaf(-S2i, cim.z, t.v[10]));
    t.v[11] = fmaf(S2r, cim.x, fmaf(S2i, cre.x, t.v[11]));
    t.v[12] = fmaf(S2r, cim.y, fmaf(S2i, cre.y, t.v[12]));
    t.v[13] = fmaf(S2r, cim.z, fmaf(S2i, cre.z, t.v[13]));
}

// The target point of a thread: offset d from its tile centre, normal n,
// with -n and |d|^2, n.d kept for the per-tile constants.
struct PairTgt {
    float dx, dy, dz, nx, ny, nz, dd, nd;
    f2 nnx, nny, nnz;
};

// One target point against one source tile.  With D = c_target - c_source
// (c0 carries 2D and R_c^2 = |D|^2, c1 R_c and the reduced phases), a source
// point offset g from its centre gives x - y = d - g + D and
//   s = r^2 - R_c^2 = |g|^2 - 2 g.(d + D) + |d|^2 + 2 D.d,
// a sum whose terms are as small as s itself times R_c / tile size, so that
// the phase offset r - R_c = s / (r + R_c) keeps FP32 accuracy;
// n_x.(x - y) = (n.d + n.D) - n.g.
template <bool TWO, bool L0, bool L1>
__device__ __forceinline__ void tile_body(const Stage& st, int ntri, int skip_tl, const PairTgt& X, float4 c0, float4 c1,
                                          PairK k0, PairK k1, Acc& a0, Acc& a1) {
    const float D2x = c0.x, D2y = c0.y, D2z = c0.z;
    const f2 m2x = bc2(-fmaf(2.f, X.dx, D2x)), m2y = bc2(-fmaf(2.f, X.dy, D2y)), m2z = bc2(-fmaf(2.f, X.dz, D2z));
    const f2 cb = bc2(fmaf(D2x, X.dx, fmaf(D2y, X.dy, fmaf(D2z, X.dz, X.dd))));
    const f2 cn = bc2(fmaf(0.5f, X.nx * D2x + X.ny * D2y + X.nz * D2z, X.nd));
    const f2 Rc2 = bc2(c0.w), Rc = bc2(c1.x);
    k0.th = bc2(c1.y);
    if constexpr (TWO) k1.th = bc2(c1.z);
    const float Xx = fmaf(0.5f, D2x, X.dx), Xy = fmaf(0.5f, D2y, X.dy), Xz = fmaf(0.5f, D2z, X.dz);  // x - c_source
    const f2 z2 = make_float2(0.f, 0.f);
    PairTile T0{z2, z2, z2, z2}, T1{z2, z2, z2, z2};
    for (int tl = 0; tl < ntri; tl++) {
        if (tl == skip_tl) continue;  // identical triangle: near-field correction only
        PairTri S0{z2, z2, z2, z2, z2, z2}, S1{z2, z2, z2, z2, z2, z2};
#pragma unroll
        for (int j = 0; j < QP / 2; j++) {
            const float4 GA = st.pg[tl * QP + 2 * j], GB = st.pg[tl * QP + 2 * j + 1];
            const float4 DA = st.pd[tl * QP + 2 * j], DB = st.pd[tl * QP + 2 * j + 1];
            const f2 gx = lo2(GA), gy = hi2(GA), gz = lo2(GB), w = hi2(GB);
            const f2 d1r = lo2(DA), d1i = hi2(DA), d2r = lo2(DB), d2i = hi2(DB);
            const f2 s = fma2(gx, add2(gx, m2x), fma2(gy, add2(gy, m2y), fma2(gz, add2(gz, m2z), cb)));
            const f2 r2 = add2(s, Rc2);
            const f2 rinv = make_float2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
            const f2 rinv2 = mul2(rinv, rinv);
            const f2 den = fma2(r2, rinv, Rc);  // r + R_c
            const f2 rho = mul2(s, make_float2(rcp_approx(den.x), rcp_approx(den.y)));
            const f2 ndot = fma2(X.nnx, gx, fma2(X.nny, gy, fma2(X.nnz, gz, cn)));
            const f2 r = (L0 || L1) ? mul2(r2, rinv) : z2;
            const f2 nd1i = neg2(d1i), nd2i = neg2(d2i);
            pair_slot<L0>(k0, rho, r, rinv, rinv2, ndot, w, d1r, d1i, nd1i, d2r, d2i, nd2i, T0, S0);
            if constexpr (TWO) pair_slot<L1>(k1, rho, r, rinv, rinv2, ndot, w, d1r, d1i, nd1i, d2r, d2i, nd2i, T1, S1);
        }
        const float4 tg = st.tg[tl];
        const float4 cre = st.tc[2 * tl], cim = st.tc[2 * tl + 1];
        const float fK = tg.w - (tg.x * Xx + tg.y * Xy + tg.z * Xz);  // n_t.(y - x)
        const float nn = X.nx * tg.x + X.ny * tg.y + X.nz * tg.z;      // n_x.n_t
        slot_triangle(fK, nn, cre, cim, S0, a0);
        if constexpr (TWO) slot_triangle(fK, nn, cre, cim, S1, a1);
    }
    a0.v[0] += T0.Vr.x + T0.Vr.y;
    a0.v[1] += T0.Vi.x + T0.Vi.y;
    a0.v[4] -= T0.nKpr.x + T0.nKpr.y;
    a0.v[5] -= T0.nKpi.x + T0.nKpi.y;
    if constexpr (TWO) {
        a1.v[0] += T1.Vr.x + T1.Vr.y;
        a1.v[1] += T1.Vi.x + T1.Vi.y;
        a1.v[4] -= T1.nKpr.x + T1.nKpr.y;
        a1.v[5] -= T1.nKpi.x + T1.nKpi.y;
    }
}

// One work item: target tile tx (offset from A.tgt_begin) against source chunk cy.
__device__ __forceinline__ void far32_item(const FarArgs32& A, int tx, int cy) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    FarSmem& sm = *reinterpret_cast<FarSmem*>(smem_raw);

    const int tid = threadIdx.x, lane = tid & 31;
    const int tt = A.tgt_begin + tx;
    const int sb = A.src_begin + cy * A.chunk_tiles;
    const int se = min(sb + A.chunk_tiles, A.src_end);
    const int nsrc = max(0, se - sb);

    const int64_t p = (int64_t)tt * TP + tid;
    const float4 g = A.pg[p];
    const int mt = tid / QP;
    const float4 ng = A.tg[(int64_t)tt * TT + mt];
    const double4 ct = A.tc[tt];
    const int mydom = A.tdom[tt];
    const int2 dr = A.dom_tiles[mydom];
    const double2 kj = A.kdom[mydom];
    const PairK k0{bc2((float)A.k0.x), bc2(0.f), bc2((float)A.k0.y),
                   bc2((float)(-A.k0.y * 1.4426950408889634))};
    const PairK k1{bc2((float)kj.x), bc2(0.f), bc2((float)kj.y),
                   bc2((float)(-kj.y * 1.4426950408889634))};
    const bool lossy0 = A.k0.y != 0.0, lossy1 = kj.y != 0.0;
    const PairTgt X{g.x, g.y, g.z, ng.x, ng.y, ng.z, g.x * g.x + g.y * g.y + g.z * g.z,
                    ng.x * g.x + ng.y * g.y + ng.z * g.z, bc2(-ng.x), bc2(-ng.y), bc2(-ng.z)};

    // tile-pair table: 2D, R_c^2, R_c and the FP64-reduced phases
    for (int i = tid; i < nsrc; i += TP) {
        const int s = sb + i;
        const double4 cs = A.tc[s];
        const double Dx = ct.x - cs.x, Dy = ct.y - cs.y, Dz = ct.z - cs.z;
        const double R = sqrt(Dx * Dx + Dy * Dy + Dz * Dz);
        const bool own = A.slot1 && s >= dr.x && s < dr.y;
        sm.tab[2 * i] = make_float4((float)(2 * Dx), (float)(2 * Dy), (float)(2 * Dz), (float)(R * R));
        sm.tab[2 * i + 1] = make_float4((float)R, reduce_phase(A.k0.x * R), own ? reduce_phase(kj.x * R) : 0.f, 0.f);
    }
    if (tid == 0) {
        for (int s = 0; s < NSTAGE; s++) {
            mbar_init(&sm.full[s], 1);
            sm.cnt[s] = 0;
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    inputs_ready();
    dependents_may_start();
    __syncthreads();

    auto issue = [&](int i, int st) {
        const int s = sb + i;
        Stage& S = sm.st[st];
        mbar_arrive_expect_tx(&sm.full[st], STAGE_BYTES);
        bulk_g2s(S.pg, A.pgp + (int64_t)s * TP, TP * 16, &sm.full[st]);
        bulk_g2s(S.pd, A.pd + (int64_t)s * TP, TP * 16, &sm.full[st]);
        bulk_g2s(S.tg, A.tg + (int64_t)s * TT, TT * 16, &sm.full[st]);
        bulk_g2s(S.tc, A.tcurl + (int64_t)s * 2 * TT, 2 * TT * 16, &sm.full[st]);
    };
    if (tid == 0)
        for (int i = 0; i < min(NSTAGE, nsrc); i++) issue(i, i);

    Acc a0, a1;
#pragma unroll
    for (int c = 0; c < NCOMP; c++) {
        a0.v[c] = 0.f;
        a1.v[c] = 0.f;
    }
    for (int i = 0; i < nsrc; i++) {
        const int st = i % NSTAGE;
        mbar_wait_bounded(&sm.full[st], (uint32_t)((i / NSTAGE) & 1), A.err);
        const int s = sb + i;
        const Stage& S = sm.st[st];
        const int ntri = A.tntri[s];
        const int skip = (s == tt) ? mt : -1;
        const float4 c0 = sm.tab[2 * i], c1 = sm.tab[2 * i + 1];
        const bool two = A.slot1 && s >= dr.x && s < dr.y;
        if (two) {
            if (lossy0) {
                if (lossy1) tile_body<true, true, true>(S, ntri, skip, X, c0, c1, k0, k1, a0, a1);
                else tile_body<true, true, false>(S, ntri, skip, X, c0, c1, k0, k1, a0, a1);
            } else {
                if (lossy1) tile_body<true, false, true>(S, ntri, skip, X, c0, c1, k0, k1, a0, a1);
                else tile_body<true, false, false>(S, ntri, skip, X, c0, c1, k0, k1, a0, a1);
            }
        } else {
            if (lossy0) tile_body<false, true, false>(S, ntri, skip, X, c0, c1, k0, k1, a0, a1);
            else tile_body<false, false, false>(S, ntri, skip, X, c0, c1, k0, k1, a0, a1);
        }
        // leave the stage; the last warp out refills it with the tile NSTAGE ahead
        __syncwarp();
        if (lane == 0) {
            const int old = atomicAdd(&sm.cnt[st], 1);
            if (old == NWARP - 1) {
                sm.cnt[st] = 0;
                if (i + NSTAGE < nsrc) issue(i + NSTAGE, st);
            }
        }
    }

    float* out = A.partial + (int64_t)cy * 2 * NCOMP * A.n_pts + (p - A.p_off);
#pragma unroll
    for (int c = 0; c < NCOMP; c++) {
        out[(int64_t)c * A.n_pts] = a0.v[c];
        out[(int64_t)(NCOMP + c) * A.n_pts] = a1.v[c];
    }
}

__global__ void __launch_bounds__(TP, 2) far32_kernel(FarArgs32 A) {
    int tx = blockIdx.x, cy = blockIdx.y;
    if (A.work) {
        const int2 w = A.work[blockIdx.x];
        tx = w.x;
        cy = w.y;
    }
    far32_item(A, tx, cy);
}

// Several meshes in one launch: work item blockIdx.x is (mesh, target tile,
// chunk) = gwork[blockIdx.x], and the mesh's arguments are group[mesh].
__global__ void __launch_bounds__(TP, 2) far32_group_kernel(const FarArgs32* __restrict__ group,
                                                            const int4* __restrict__ gwork) {
    const int4 w = gwork[blockIdx.x];
    const FarArgs32 A = group[w.x];
    far32_item(A, w.y, w.z);
}

size_t far32_smem_bytes() { return sizeof(FarSmem); }

cudaError_t launch_far32(const FarArgs32& a, int n_tgt_tiles, int n_chunks, cudaStream_t s) {
    const size_t smem = far32_smem_bytes();
    static const cudaError_t attr_e =
        cudaFuncSetAttribute(far32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (attr_e != cudaSuccess) return attr_e;
    if (n_tgt_tiles <= 0 || n_chunks <= 0) return cudaSuccess;
    const dim3 grid = a.work ? dim3((unsigned)((int64_t)n_tgt_tiles * n_chunks)) : dim3(n_tgt_tiles, n_chunks);
    return launch_after(far32_kernel, grid, TP, smem, s, a);
}

cudaError_t launch_far32_group(const FarArgs32* group, const int4* gwork, int64_t n_work, cudaStream_t s) {
    const size_t smem = far32_smem_bytes();
    static const cudaError_t attr_e =
        cudaFuncSetAttribute(far32_group_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (attr_e != cudaSuccess) return attr_e;
    if (n_work <= 0) return cudaSuccess;
    far32_group_kernel<<<(unsigned)n_work, TP, smem, s>>>(group, gwork);
    return cudaGetLastError();
}

// ----------------------------------------------------------------- FP32 far field, several right-hand sides
//
// The Green's function G and the gradient factor F of a (target point,
// source point) pair do not depend on the densities, so a work item that
// serves MRG right-hand sides evaluates the geometry, the phase and the MUFU
// functions once and accumulates MRG sets of potentials.  One wavenumber
// slot per work item keeps the per-thread state (14 potentials and eight
// packed triangle sums per right-hand side) within the register budget of
// the one-vector kernel; own-domain sources are visited once per slot.

constexpr int NSTAGE_M = 3;

struct __align__(16) StageM {
    float4 pg[TP];           // source points (dx, dy, dz, w), pair-interleaved
    float4 tg[TT];           // triangles (n, h)
    float4 pd[MRG][TP];      // densities of each right-hand side, pair-interleaved
    float4 tc[MRG][2 * TT];  // curl densities of each right-hand side
};
constexpr uint32_t STAGE_M_BYTES = sizeof(StageM);
static_assert(STAGE_M_BYTES == 3584 + MRG * 4096, "multi stage layout");

struct FarSmemM {
    StageM st[NSTAGE_M];
    float4 tab[2 * CHUNK_MAX];
    int src[CHUNK_MAX];  // source tiles of the item
    int nsrc;
    uint64_t full[NSTAGE_M];
    int cnt[NSTAGE_M];
};

// Per right-hand side: the V and K' sums run packed over the whole item
// (no per-triangle factor; folded once at the end), the K and W terms need
// per-triangle sums (K' and K kept with the sign of -F, as in the one-vector
// kernel).
struct AccM {
    f2 Vr, Vi, nKpr, nKpi;
    float K[2], Wm[2], Wc[6];
};
struct PairTriM {
    f2 nS1r, nS1i, S3r, S3i;
};

template <bool LOSSY>
__device__ __forceinline__ void tile_body_m(const StageM& st, int ntri, int skip_tl, const PairTgt& X, float4 c0,
                                            float Rcf, PairK k, AccM (&acc)[MRG]) {
    const float D2x = c0.x, D2y = c0.y, D2z = c0.z;
    const f2 m2x = bc2(-fmaf(2.f, X.dx, D2x)), m2y = bc2(-fmaf(2.f, X.dy, D2y)), m2z = bc2(-fmaf(2.f, X.dz, D2z));
    const f2 cb = bc2(fmaf(D2x, X.dx, fmaf(D2y, X.dy, fmaf(D2z, X.dz, X.dd))));
    const f2 cn = bc2(fmaf(0.5f, X.nx * D2x + X.ny * D2y + X.nz * D2z, X.nd));
    const f2 Rc2 = bc2(c0.w), Rc = bc2(Rcf);
    const float Xx = fmaf(0.5f, D2x, X.dx), Xy = fmaf(0.5f, D2y, X.dy), Xz = fmaf(0.5f, D2z, X.dz);  // x - c_source
    const f2 z2 = make_float2(0.f, 0.f);
    for (int tl = 0; tl < ntri; tl++) {
        if (tl == skip_tl) continue;  // identical triangle: near-field correction only
        PairTriM S[MRG];
#pragma unroll
        for (int q = 0; q < MRG; q++) S[q] = PairTriM{z2, z2, z2, z2};
        f2 S2r = z2, S2i = z2;
#pragma unroll
        for (int j = 0; j < QP / 2; j++) {
            const float4 GA = st.pg[tl * QP + 2 * j], GB = st.pg[tl * QP + 2 * j + 1];
            const f2 gx = lo2(GA), gy = hi2(GA), gz = lo2(GB), w = hi2(GB);
            const f2 s = fma2(gx, add2(gx, m2x), fma2(gy, add2(gy, m2y), fma2(gz, add2(gz, m2z), cb)));
            const f2 r2 = add2(s, Rc2);
            const f2 rinv = make_float2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
            const f2 rinv2 = mul2(rinv, rinv);
            const f2 den = fma2(r2, rinv, Rc);  // r + R_c
            const f2 rho = mul2(s, make_float2(rcp_approx(den.x), rcp_approx(den.y)));
            const f2 ndot = fma2(X.nnx, gx, fma2(X.nny, gy, fma2(X.nnz, gz, cn)));
            const f2 arg = fma2(k.kr, rho, k.th);
            f2 sn, cs;
            sincos_approx(arg.x, &sn.x, &cs.x);
            sincos_approx(arg.y, &sn.y, &cs.y);
            f2 a = rinv;
            if constexpr (LOSSY) {
                const f2 e = mul2(k.nkil2, mul2(r2, rinv));
                a = mul2(make_float2(ex2_approx(e.x), ex2_approx(e.y)), rinv);
            }
            const f2 Gr = mul2(a, cs), Gi = mul2(a, sn);
            const f2 B = mul2(k.kr, rinv);
            const f2 P = LOSSY ? fma2(k.ki, rinv, rinv2) : rinv2;
            const f2 nFr = fma2(P, Gr, mul2(B, Gi));
            const f2 nFi = fma2(P, Gi, neg2(mul2(B, Gr)));
            const f2 nFnr = mul2(ndot, nFr), nFni = mul2(ndot, nFi);
            S2r = fma2(Gr, w, S2r);
            S2i = fma2(Gi, w, S2i);
#pragma unroll
            for (int q = 0; q < MRG; q++) {
                const float4 DA = st.pd[q][tl * QP + 2 * j], DB = st.pd[q][tl * QP + 2 * j + 1];
                const f2 d1r = lo2(DA), d1i = hi2(DA), d2r = lo2(DB), d2i = hi2(DB);
                const f2 nd1i = neg2(d1i), nd2i = neg2(d2i);  // folded into the packed FMAs' operands
                PairTriM& T = S[q];
                AccM& U = acc[q];
                U.Vr = fma2(Gr, d1r, fma2(Gi, nd1i, U.Vr));
                U.Vi = fma2(Gr, d1i, fma2(Gi, d1r, U.Vi));
                U.nKpr = fma2(nFnr, d1r, fma2(nFni, nd1i, U.nKpr));
                U.nKpi = fma2(nFnr, d1i, fma2(nFni, d1r, U.nKpi));
                T.nS1r = fma2(nFr, d2r, fma2(nFi, nd2i, T.nS1r));
                T.nS1i = fma2(nFr, d2i, fma2(nFi, d2r, T.nS1i));
                T.S3r = fma2(Gr, d2r, fma2(Gi, nd2i, T.S3r));
                T.S3i = fma2(Gr, d2i, fma2(Gi, d2r, T.S3i));
            }
        }
        const float4 tg = st.tg[tl];
        const float fK = tg.w - (tg.x * Xx + tg.y * Xy + tg.z * Xz);  // n_t.(y - x)
        const float nn = X.nx * tg.x + X.ny * tg.y + X.nz * tg.z;      // n_x.n_t
        const float s2r = S2r.x + S2r.y, s2i = S2i.x + S2i.y;
#pragma unroll
        for (int q = 0; q < MRG; q++) {
            const PairTriM& T = S[q];
            AccM& t = acc[q];
            const float4 cre = st.tc[q][2 * tl], cim = st.tc[q][2 * tl + 1];
            t.K[0] = fmaf(-fK, T.nS1r.x + T.nS1r.y, t.K[0]);
            t.K[1] = fmaf(-fK, T.nS1i.x + T.nS1i.y, t.K[1]);
            t.Wm[0] = fmaf(nn, T.S3r.x + T.S3r.y, t.Wm[0]);
            t.Wm[1] = fmaf(nn, T.S3i.x + T.S3i.y, t.Wm[1]);
            t.Wc[0] = fmaf(s2r, cre.x, fmaf(-s2i, cim.x, t.Wc[0]));
            t.Wc[1] = fmaf(s2r, cre.y, fmaf(-s2i, cim.y, t.Wc[1]));
            t.Wc[2] = fmaf(s2r, cre.z, fmaf(-s2i, cim.z, t.Wc[2]));
            t.Wc[3] = fmaf(s2r, cim.x, fmaf(s2i, cre.x, t.Wc[3]));
            t.Wc[4] = fmaf(s2r, cim.y, fmaf(s2i, cre.y, t.Wc[4]));
            t.Wc[5] = fmaf(s2r, cim.z, fmaf(s2i, cre.z, t.Wc[5]));
        }
    }
}

// Work item: target tile tx (offset from A.tgt_begin) against source chunk
// cy at wavenumber slot `slot` (0: k0 on every source tile; 1: the target
// domain's k_j on its own tiles), right-hand sides grp * MRG ... + MRG - 1.
template <bool LOSSY>
__device__ __forceinline__ void far32m_item(const FarArgs32M& A, int tx, int cy, int slot, int grp) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    FarSmemM& sm = *reinterpret_cast<FarSmemM*>(smem_raw);

    const int tid = threadIdx.x, lane = tid & 31;
    const int tt = A.tgt_begin + tx;
    const int mydom = A.tdom[tt];
    const int2 dr = A.dom_tiles[mydom];
    // the item's source tiles (slot 1: those of the target's domain)
    if (tid < 32) {
        const int sb = A.near_ptr ? A.near_ptr[tt] : A.src_begin + cy * A.chunk_tiles;
        const int se = A.near_ptr ? min(A.near_ptr[tt + 1], sb + CHUNK_MAX) : min(sb + A.chunk_tiles, A.src_end);
        int n = 0;
        for (int b = sb; b < se; b += 32) {
            const int s = b + lane < se ? (A.near_ptr ? A.near_idx[b + lane] : b + lane) : -1;
            const bool in = s >= 0 && (!slot || (s >= dr.x && s < dr.y));
            const uint32_t m = __ballot_sync(0xffffffffu, in);
            if (in) sm.src[n + __popc(m & ((1u << lane) - 1))] = s;
            n += __popc(m);
        }
        if (lane == 0) sm.nsrc = n;
    }
    __syncthreads();
    const int nsrc = sm.nsrc;
    const int r0 = grp * MRG;
    const int nq = min(MRG, A.R - r0);

    const int64_t p = (int64_t)tt * TP + tid;
    const float4 g = A.pg[p];
    const int mt = tid / QP;
    const float4 ng = A.tg[(int64_t)tt * TT + mt];
    const double4 ct = A.tc[tt];
    const double2 kk = slot ? A.kdom[mydom] : A.k0;
    const PairK k{bc2((float)kk.x), bc2(0.f), bc2((float)kk.y),
                  bc2((float)(-kk.y * 1.4426950408889634))};
    const PairTgt X{g.x, g.y, g.z, ng.x, ng.y, ng.z, g.x * g.x + g.y * g.y + g.z * g.z,
                    ng.x * g.x + ng.y * g.y + ng.z * g.z, bc2(-ng.x), bc2(-ng.y), bc2(-ng.z)};

    // tile-pair table: 2D, R_c^2, R_c and the FP64-reduced phase
    for (int i = tid; i < nsrc; i += TP) {
        const double4 cs = A.tc[sm.src[i]];
        const double Dx = ct.x - cs.x, Dy = ct.y - cs.y, Dz = ct.z - cs.z;
        const double R = sqrt(Dx * Dx + Dy * Dy + Dz * Dz);
        sm.tab[2 * i] = make_float4((float)(2 * Dx), (float)(2 * Dy), (float)(2 * Dz), (float)(R * R));
        sm.tab[2 * i + 1] = make_float4((float)R, reduce_phase(kk.x * R), 0.f, 0.f);
    }
    if (tid == 0) {
        for (int s = 0; s < NSTAGE_M; s++) {
            mbar_init(&sm.full[s], 1);
            sm.cnt[s] = 0;
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    auto issue = [&](int i, int st) {
        const int s = sm.src[i];
        StageM& S = sm.st[st];
        mbar_arrive_expect_tx(&sm.full[st], STAGE_M_BYTES);
        bulk_g2s(S.pg, A.pgp + (int64_t)s * TP, TP * 16, &sm.full[st]);
        bulk_g2s(S.tg, A.tg + (int64_t)s * TT, TT * 16, &sm.full[st]);
#pragma unroll
        for (int q = 0; q < MRG; q++) {
            const int64_t r = min(r0 + q, A.R - 1);  // a short last group repeats the last vector (not written)
            bulk_g2s(S.pd[q], A.pd + r * A.n_pts + (int64_t)s * TP, TP * 16, &sm.full[st]);
            bulk_g2s(S.tc[q], A.tcurl + r * 2 * A.n_slots + (int64_t)s * 2 * TT, 2 * TT * 16, &sm.full[st]);
        }
    };
    if (tid == 0)
        for (int i = 0; i < min(NSTAGE_M, nsrc); i++) issue(i, i);

    AccM acc[MRG];
#pragma unroll
    for (int q = 0; q < MRG; q++) {
        const f2 z2 = make_float2(0.f, 0.f);
        acc[q].Vr = acc[q].Vi = acc[q].nKpr = acc[q].nKpi = z2;
        acc[q].K[0] = acc[q].K[1] = acc[q].Wm[0] = acc[q].Wm[1] = 0.f;
#pragma unroll
        for (int c = 0; c < 6; c++) acc[q].Wc[c] = 0.f;
    }
    for (int i = 0; i < nsrc; i++) {
        const int st = i % NSTAGE_M;
        mbar_wait_bounded(&sm.full[st], (uint32_t)((i / NSTAGE_M) & 1), A.err);
        const int s = sm.src[i];
        const int ntri = A.tntri[s];
        const int skip = (s == tt) ? mt : -1;
        const float4 c0 = sm.tab[2 * i], c1 = sm.tab[2 * i + 1];
        PairK kt = k;
        kt.th = bc2(c1.y);
        tile_body_m<LOSSY>(sm.st[st], ntri, skip, X, c0, c1.x, kt, acc);
        // leave the stage; the last warp out refills it with the tile NSTAGE_M ahead
        __syncwarp();
        if (lane == 0) {
            const int old = atomicAdd(&sm.cnt[st], 1);
            if (old == NWARP - 1) {
                sm.cnt[st] = 0;
                if (i + NSTAGE_M < nsrc) issue(i + NSTAGE_M, st);
            }
        }
    }

    const int64_t po = A.perm ? (int64_t)A.perm[(int64_t)tt * TT + mt] * QP + tid % QP : p;
#pragma unroll
    for (int q = 0; q < MRG; q++) {
        if (q >= nq) break;
        const AccM& t = acc[q];
        // the 14 potentials in the order of the one-vector kernel: PV, PK, PK', PWm, PWc
        const float v[NCOMP] = {t.Vr.x + t.Vr.y, t.Vi.x + t.Vi.y, t.K[0], t.K[1], -(t.nKpr.x + t.nKpr.y),
                                -(t.nKpi.x + t.nKpi.y), t.Wm[0], t.Wm[1], t.Wc[0], t.Wc[1], t.Wc[2], t.Wc[3],
                                t.Wc[4], t.Wc[5]};
        float* out = A.partial + (int64_t)(r0 + q) * A.rstride + ((int64_t)cy * 2 + slot) * NCOMP * A.n_pts + po;
#pragma unroll
        for (int c = 0; c < NCOMP; c++) out[(int64_t)c * A.n_pts] = v[c];
    }
}

__global__ void __launch_bounds__(TP, 2) far32m_kernel(FarArgs32M A) {
    const int4 w = A.work[blockIdx.x];
    const int mydom = A.tdom[A.tgt_begin + w.x];
    const double ki = w.z ? A.kdom[mydom].y : A.k0.y;
    if (ki != 0.0) far32m_item<true>(A, w.x, w.y, w.z, w.w);
    else far32m_item<false>(A, w.x, w.y, w.z, w.w);
}

cudaError_t launch_far32_multi(const FarArgs32M& a, int64_t n_work, cudaStream_t s) {
    const size_t smem = sizeof(FarSmemM);
    static const cudaError_t attr_e =
        cudaFuncSetAttribute(far32m_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (attr_e != cudaSuccess) return attr_e;
    if (n_work <= 0) return cudaSuccess;
    far32m_kernel<<<(unsigned)n_work, TP, smem, s>>>(a);
    return cudaGetLastError();
}

// ----------------------------------------------------------------- FP64 far field

// One vector at FP64: the multi-vector kernel with a single group.
cudaError_t launch_far64(const FarArgs64& a, int n_tgt_tiles, int n_chunks, cudaStream_t s) {
    FarArgs64M m{};
    m.pg = a.pg; m.tg = a.tg; m.tc = a.tc; m.tdom = a.tdom; m.tntri = a.tntri; m.pd = a.pd; m.tcurl = a.tcurl;
    m.dom_tiles = a.dom_tiles; m.kdom = a.kdom; m.k0 = a.k0;
    m.src_begin = a.src_begin; m.src_end = a.src_end; m.tgt_begin = a.tgt_begin; m.chunk_tiles = a.chunk_tiles;
    m.slot1 = a.slot1; m.groups = 1; m.R = 1; m.n_pts = a.n_pts; m.n_slots = 0; m.rstride = 0; m.partial = a.partial;
    return launch_far64_multi(m, n_tgt_tiles, n_chunks, s);
}

// Several vectors per FP64 far-field CTA.  The Green's function G, its radial
// factor F and the geometric weights of a (target point, source point) pair
// are computed once and applied to each of the group's vectors, with the
// target-normal and source-edge factors folded into the point terms:
// 16 FP64 FMAs per vector and pair beside the shared evaluation (sqrt, the
// reciprocal, sincos and, for a complex wavenumber, exp).  Sums per vector
// and component in source order, so results do not depend on the group.
template <int RG, bool ATTEN>
__device__ __forceinline__ void far64m_body(const FarArgs64M& A, int sl, int grp) {
    const int tid = threadIdx.x;
    const int tt = A.tgt_begin + blockIdx.x;
    const int chunk = blockIdx.y;
    int sb = A.src_begin + chunk * A.chunk_tiles;
    int se = min(sb + A.chunk_tiles, A.src_end);
    const int64_t p = (int64_t)tt * TP + tid;
    const double4 g = A.pg[p];
    const int mt = tid / QP;
    const double4 ng = A.tg[(int64_t)tt * TT + mt];
    const double4 ct = A.tc[tt];
    const int mydom = A.tdom[tt];
    if (sl == 1) {
        const int2 dr = A.dom_tiles[mydom];
        sb = max(sb, dr.x);
        se = min(se, dr.y);
    }
    const double2 kk = sl ? A.kdom[mydom] : A.k0;
    const double kr = kk.x, ki = kk.y;
    const int r0 = grp * RG, nv = min(RG, A.R - r0);
    double acc[RG][NCOMP];
#pragma unroll
    for (int v = 0; v < RG; v++)
#pragma unroll
        for (int c = 0; c < NCOMP; c++) acc[v][c] = 0.0;
    for (int s = sb; s < se; s++) {
        const double4 cs = A.tc[s];
        const double Xx = g.x + (ct.x - cs.x), Xy = g.y + (ct.y - cs.y), Xz = g.z + (ct.z - cs.z);  // x - c_source
        const int ntri = A.tntri[s];
        for (int tl = 0; tl < ntri; tl++) {
            if (s == tt && tl == mt) continue;
            const int64_t ts = (int64_t)s * TT + tl;
            const double4 tg = A.tg[ts];
            const double fK = tg.w - (tg.x * Xx + tg.y * Xy + tg.z * Xz);
            const double nn = ng.x * tg.x + ng.y * tg.y + ng.z * tg.z;
            double S2r = 0, S2i = 0;
            for (int q = 0; q < QP; q++) {
                const double4 y = A.pg[ts * QP + q];
                const double ex = Xx - y.x, ey = Xy - y.y, ez = Xz - y.z;  // x - y
                const double r = sqrt(ex * ex + ey * ey + ez * ez);
                const double rinv = 1.0 / r;
                double sn, cs2;
                sincos(kr * r, &sn, &cs2);
                const double a = (ATTEN ? exp(-ki * r) : 1.0) * rinv;
                const double Gr = a * cs2, Gi = a * sn;
                const double u = -ki - rinv;
                const double Fr = (Gr * u - Gi * kr) * rinv, Fi = (Gr * kr + Gi * u) * rinv;
                const double ndot = ng.x * ex + ng.y * ey + ng.z * ez;
                const double nFr = ndot * Fr, nFi = ndot * Fi;  // K' point factor
                const double kFr = fK * Fr, kFi = fK * Fi;      // K point factor
                const double wGr = nn * Gr, wGi = nn * Gi;      // W (normal-normal) point factor
                S2r += Gr * y.w;
                S2i += Gi * y.w;
#pragma unroll
                for (int v = 0; v < RG; v++) {
                    if (v >= nv) break;
                    const double4 d = A.pd[(int64_t)(r0 + v) * A.n_pts + ts * QP + q];
                    acc[v][0] += Gr * d.x - Gi * d.y;
                    acc[v][1] += Gr * d.y + Gi * d.x;
                    acc[v][2] += kFr * d.z - kFi * d.w;
                    acc[v][3] += kFr * d.w + kFi * d.z;
                    acc[v][4] += nFr * d.x - nFi * d.y;
                    acc[v][5] += nFr * d.y + nFi * d.x;
                    acc[v][6] += wGr * d.z - wGi * d.w;
                    acc[v][7] += wGr * d.w + wGi * d.z;
                }
            }
#pragma unroll
            for (int v = 0; v < RG; v++) {
                if (v >= nv) break;
                const double4* tcv = A.tcurl + (int64_t)(r0 + v) * 2 * A.n_slots;
                const double4 cre = tcv[2 * ts], cim = tcv[2 * ts + 1];
                acc[v][8] += S2r * cre.x - S2i * cim.x;
                acc[v][9] += S2r * cre.y - S2i * cim.y;
                acc[v][10] += S2r * cre.z - S2i * cim.z;
                acc[v][11] += S2r * cim.x + S2i * cre.x;
                acc[v][12] += S2r * cim.y + S2i * cre.y;
                acc[v][13] += S2r * cim.z + S2i * cre.z;
            }
        }
    }
#pragma unroll
    for (int v = 0; v < RG; v++) {
        if (v >= nv) break;
        double* out = A.partial + (int64_t)(r0 + v) * A.rstride + ((int64_t)chunk * 2 + sl) * NCOMP * A.n_pts + p;
#pragma unroll
        for (int c = 0; c < NCOMP; c++) out[(int64_t)c * A.n_pts] = acc[v][c];
    }
}

template <int RG>
__global__ void __launch_bounds__(TP, RG == 1 ? 2 : 1) far64m_kernel(FarArgs64M A) {
    const int sl = blockIdx.z / A.groups, grp = blockIdx.z % A.groups;
    const double ki = sl ? A.kdom[A.tdom[A.tgt_begin + blockIdx.x]].y : A.k0.y;
    if (ki != 0.0) far64m_body<RG, true>(A, sl, grp);
    else far64m_body<RG, false>(A, sl, grp);
}

// One vector (groups = R = 1) or groups of RG64; slot 1 only with a.slot1.
cudaError_t launch_far64_multi(const FarArgs64M& a, int n_tgt_tiles, int n_chunks, cudaStream_t s) {
    if (n_tgt_tiles <= 0 || n_chunks <= 0 || a.groups <= 0) return cudaSuccess;
    const dim3 grid(n_tgt_tiles, n_chunks, (a.slot1 ? 2 : 1) * a.groups);
    if (a.R == 1) far64m_kernel<1><<<grid, TP, 0, s>>>(a);
    else far64m_kernel<RG64><<<grid, TP, 0, s>>>(a);
    return cudaGetLastError();
}

// ----------------------------------------------------------------- projection onto P1 test functions

// One CTA per PS = 8 slots (a quarter of a target tile), three phases:
//  1. near pairs (touching and near band), one warp per slot, one pair per
//     lane and pass: the combined 3x3 sub-blocks (row1<-psi, row1<-phi,
//     row2<-psi, row2<-phi) times the pair's source values.  The FP32
//     operator takes FP32 products; a lane sums its two or three pairs.
//  2. chunk partials: the CTA's 2 x NCOMP x 48 sums over the chunks, one
//     (component, point) per thread and pass, points coalesced.  FP32
//     partials are summed with a compensated (TwoSum) FP32 sum in chunk
//     order, converted to FP64 once: the GPU's FP64 rate is a small fraction
//     of its FP32 rate, and the compensation carries the rounding error of
//     every addition, so the result matches an FP64 sum of the same FP32
//     values to about 1e-15 of the sum of their magnitudes.
//  3. the projection onto the P1 test functions in FP64, spread over the
//     (slot, point) and (slot, vertex) pairs, and the lanes' near sums
//     (compensated again) in lane order.
// The kernel is a chain of dependent loads and of FP64 operations at 1/64 of
// the FP32 rate, so its time at small sizes is the length of that chain on
// one SM.  One CTA per tile with six threads per slot walked ten pairs one
// after another and ran a tile's FP64 on one SM; a quarter of a tile per CTA
// and 32 lanes per slot shorten both: 76 -> 24 us on 300 triangles, 234 -> 98 us
// on 8,172 (FP32), 319 -> 159 us on 1,452 (FP64), cold caches.
constexpr int PS = 8;                  // slots per CTA
constexpr int PP = PS * QP;            // points per CTA
constexpr int PROJ_THREADS = PS * 32;
constexpr int PROJ_PAD = 32 * 12 + 4;  // near partial sums of one slot, padded against bank conflicts
static_assert(TT % PS == 0, "a CTA's slots lie in one tile");
static_assert(2 * PP + 12 * PS <= PROJ_THREADS && 3 * PS <= 32 && 32 + 6 * PS <= PROJ_THREADS, "phase 3 work fits the CTA");

__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float x) {
    const float u = hi + x;  // TwoSum: hi + x = u + (rounding error)
    const float xb = u - hi;
    lo += (hi - (u - xb)) + (x - xb);
    hi = u;
}

template <bool F64>
__global__ void __launch_bounds__(PROJ_THREADS) project_kernel(ProjectArgs a) {
    typedef typename std::conditional<F64, double, float>::type real_t;
    __shared__ double Ps[2][NCOMP][PP];
    __shared__ real_t red[PS * PROJ_PAD];
    __shared__ double nsum[PS][12], csum[PS][6];
    const int64_t s0 = (int64_t)a.tgt_begin * TT + (int64_t)blockIdx.x * PS;  // first slot
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tdom = a.tdom[s0 / TT];  // a tile holds triangles of one domain
    // 1. near pairs
    if (a.np_ptr) {
        const int64_t s = s0 + warp;
        real_t f[12];
#pragma unroll
        for (int c = 0; c < 12; c++) f[c] = 0;
        if (a.slot_v[s].x >= 0) {
            const int64_t pe = a.np_ptr[s + 1];
            // two pairs per pass: the dependent loads pair -> slot -> unknowns -> values overlap
            for (int64_t pi = a.np_ptr[s] + lane; pi < pe; pi += 64) {
                const int64_t pj[2] = {pi, min(pi + 32, pe - 1)};
                int4 vt[2];
#pragma unroll
                for (int u = 0; u < 2; u++) vt[u] = a.slot_v[a.np_src[pj[u]]];
                real_t xv[2][2][3][2];
#pragma unroll
                for (int u = 0; u < 2; u++)
#pragma unroll
                    for (int b = 0; b < 3; b++) {
                        const int vid = b == 0 ? vt[u].x : b == 1 ? vt[u].y : vt[u].z;
                        const double2 x1 = a.x[a.v_dof1[vid]], x2 = a.x[a.v_dof2[vid]];
                        xv[u][0][b][0] = (real_t)x1.x;
                        xv[u][0][b][1] = (real_t)x1.y;
                        xv[u][1][b][0] = (real_t)x2.x;
                        xv[u][1][b][1] = (real_t)x2.y;
                    }
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    if (u && pi + 32 >= pe) break;
                    // 36 complex entries as 18 loads of two (FP32, 16-byte aligned: pair stride 288 bytes) or 36 of one
#pragma unroll
                    for (int e = 0; e < 36; e++) {
                        real_t br, bi;
                        if constexpr (F64) {
                            const double2 B = a.nb64[pj[u] * 36 + e];
                            br = B.x;
                            bi = B.y;
                        } else {
                            const float4 B = reinterpret_cast<const float4*>(a.nb32 + pj[u] * 36)[e >> 1];
                            br = (e & 1) ? B.z : B.x;
                            bi = (e & 1) ? B.w : B.y;
                        }
                        const int blk = e / 9, k = (e % 9) / 3, b = e % 3, o = (blk < 2 ? 0 : 6) + 2 * k;
                        const real_t xr = xv[u][blk & 1][b][0], xi = xv[u][blk & 1][b][1];
                        f[o] += br * xr - bi * xi;
                        f[o + 1] += br * xi + bi * xr;
                    }
                }
            }
        }
#pragma unroll
        for (int c = 0; c < 12; c++) red[warp * PROJ_PAD + lane * 12 + c] = f[c];
    }
    // 2. chunk partials
    inputs_ready();
    dependents_may_start();
    const int64_t p0 = s0 * QP - a.p_off;
    const int64_t step = 2 * NCOMP * a.n_pts;  // one chunk
    // a thread's sums side by side: their loads of one chunk are independent
    constexpr int NS = (2 * NCOMP * PP + PROJ_THREADS - 1) / PROJ_THREADS;
    const SlotCoef &cf0 = a.coef[tdom * 2], &cf1 = a.coef[tdom * 2 + 1];
    const bool on[2] = {cf0.cV != 0 || cf0.cK != 0 || cf0.cKp != 0 || cf0.cW != 0,
                        cf1.cV != 0 || cf1.cK != 0 || cf1.cKp != 0 || cf1.cW != 0};
    int64_t at[NS];
    bool use[NS];
#pragma unroll
    for (int u = 0; u < NS; u++) {
        const int i = tid + u * PROJ_THREADS, row = i / PP;
        use[u] = i < 2 * NCOMP * PP && on[row >= NCOMP];
        at[u] = (int64_t)row * a.n_pts + p0 + (i - row * PP);
    }
    if constexpr (F64) {
        double sum[NS];
#pragma unroll
        for (int u = 0; u < NS; u++) sum[u] = 0.0;
#pragma unroll 2
        for (int ch = 0; ch < a.n_chunks; ch++)
#pragma unroll
            for (int u = 0; u < NS; u++)
                if (use[u]) sum[u] += a.partial64[ch * step + at[u]];
#pragma unroll
        for (int u = 0; u < NS; u++)
            if (use[u]) (&Ps[0][0][0])[tid + u * PROJ_THREADS] = sum[u];
    } else {
        float hi[NS], lo[NS];
#pragma unroll
        for (int u = 0; u < NS; u++) hi[u] = lo[u] = 0.f;
#pragma unroll 4
        for (int ch = 0; ch < a.n_chunks; ch++) {
            float x[NS];
#pragma unroll
            for (int u = 0; u < NS; u++) x[u] = use[u] ? a.partial32[ch * step + at[u]] : 0.f;
#pragma unroll
            for (int u = 0; u < NS; u++) two_sum_acc(hi[u], lo[u], x[u]);
        }
#pragma unroll
        for (int u = 0; u < NS; u++)
            if (use[u]) (&Ps[0][0][0])[tid + u * PROJ_THREADS] = (double)hi[u] + (double)lo[u];
    }
    __syncthreads();
    // 3a. one thread per (slot, wavenumber slot, point): the point's weighted
    // row potentials and curl terms, in place; beside them one thread per
    // (slot, component) adds the lanes' near sums
    if (tid < 2 * PP) {
        const int sl = tid / PP, pt = tid - sl * PP;
        if (on[sl] && a.slot_v[s0 + pt / QP].x >= 0) {
            const SlotCoef& cf = sl ? cf1 : cf0;
            const double w = a.pt_w[s0 * QP + pt] * 0.07957747154594767;  // 1 / (4 pi)
            const double P6 = Ps[sl][6][pt], P7 = Ps[sl][7][pt];
            // row1 potential: cV PV - cK PK ; row2 (pointwise part): cKp PKp - cW k^2 PWm
            const double t1r = cf.cV * Ps[sl][0][pt] - cf.cK * Ps[sl][2][pt];
            const double t1i = cf.cV * Ps[sl][1][pt] - cf.cK * Ps[sl][3][pt];
            const double t2r = cf.cKp * Ps[sl][4][pt] - cf.cW * (cf.k2re * P6 - cf.k2im * P7);
            const double t2i = cf.cKp * Ps[sl][5][pt] - cf.cW * (cf.k2re * P7 + cf.k2im * P6);
            Ps[sl][0][pt] = w * t1r;
            Ps[sl][1][pt] = w * t1i;
            Ps[sl][2][pt] = w * t2r;
            Ps[sl][3][pt] = w * t2i;
            const double wc = w * cf.cW;
#pragma unroll
            for (int c = 8; c < NCOMP; c++) Ps[sl][c][pt] *= wc;
        }
    } else if (a.np_ptr && tid < 2 * PP + PS * 12) {
        const int u = tid - 2 * PP, j = u / 12, c = u - 12 * j;
        real_t n = 0, lo = 0;
        for (int l = 0; l < 32; l++) {
            const real_t x = red[j * PROJ_PAD + l * 12 + c];
            if constexpr (F64) n += x;
            else two_sum_acc(n, lo, x);
        }
        nsum[j][c] = (double)n + (double)lo;
    }
    __syncthreads();
    // 3b. thread (j, k): rows of vertex k of slot s0 + j; beside them the slots' curl sums, one component per thread
    const int j = tid / 3, k = tid - 3 * j;
    const bool own = tid < 3 * PS && a.slot_v[s0 + j].x >= 0;
    double r[4] = {0, 0, 0, 0};
    if (own) {
#pragma unroll
        for (int sl = 0; sl < 2; sl++)
            if (on[sl])
#pragma unroll
                for (int q = 0; q < QP; q++)
#pragma unroll
                    for (int c = 0; c < 4; c++) r[c] += a.lam[q][k] * Ps[sl][c][j * QP + q];
    } else if (tid >= 32 && tid < 32 + 6 * PS) {
        const int jj = (tid - 32) / 6, c = tid - 32 - 6 * jj;
        double t = 0;
#pragma unroll
        for (int sl = 0; sl < 2; sl++)
            if (on[sl])
#pragma unroll
                for (int q = 0; q < QP; q++) t += Ps[sl][8 + c][jj * QP + q];
        csum[jj][c] = t;
    }
    __syncthreads();
    if (!own) return;
    const int64_t s = s0 + j;
    const double* cu = &a.slot_curl[s * 9 + 3 * k];
    r[2] += cu[0] * csum[j][0] + cu[1] * csum[j][1] + cu[2] * csum[j][2];
    r[3] += cu[0] * csum[j][3] + cu[1] * csum[j][4] + cu[2] * csum[j][5];
    if (a.np_ptr) {
        r[0] += nsum[j][2 * k];
        r[1] += nsum[j][2 * k + 1];
        r[2] += nsum[j][6 + 2 * k];
        r[3] += nsum[j][6 + 2 * k + 1];
    }
    a.tri_out[(s * 3 + k) * 2] = make_double2(r[0], r[1]);
    a.tri_out[(s * 3 + k) * 2 + 1] = make_double2(r[2], r[3]);
}

cudaError_t launch_project(const ProjectArgs& a, cudaStream_t s) {
    const int n_tiles = a.tgt_end - a.tgt_begin;
    if (n_tiles <= 0) return cudaSuccess;
    const unsigned grid = (unsigned)n_tiles * (TT / PS);
    return launch_after(a.partial32 ? project_kernel<false> : project_kernel<true>, dim3(grid), PROJ_THREADS, 0, s, a);
}

// ----------------------------------------------------------------- vertex reduction

__global__ void reduce_kernel(ReduceArgs a) {
    inputs_ready();
    const int64_t v = a.v_begin + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= a.v_end) return;
    double s1r = 0, s1i = 0, s2r = 0, s2i = 0;
    const int64_t e = a.vc_ptr[v + 1];
#pragma unroll 4
    for (int64_t i = a.vc_ptr[v]; i < e; i++) {
        const int64_t c = a.vc_idx[i];
        const double2 u = a.tri_out[c * 2], w = a.tri_out[c * 2 + 1];
        s1r += u.x;
        s1i += u.y;
        s2r += w.x;
        s2i += w.y;
    }
    a.y[a.v_dof1[v]] = make_double2(s1r, s1i);
    a.y[a.v_dof2[v]] = make_double2(s2r, s2i);
}

cudaError_t launch_reduce(const ReduceArgs& a, cudaStream_t s) {
    int64_t n = a.v_end - a.v_begin;
    if (n <= 0) return cudaSuccess;
    return launch_after(reduce_kernel, dim3((unsigned)((n + 63) / 64)), 64, 0, s, a);
}

cudaError_t launch_gather(const GatherArgs& a, cudaStream_t s) {
    int64_t n = a.s_end - a.s_begin;
    if (n <= 0) return cudaSuccess;
    gather_kernel<<<(unsigned)((n * QP + GATHER_THREADS - 1) / GATHER_THREADS), GATHER_THREADS, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace gbem
