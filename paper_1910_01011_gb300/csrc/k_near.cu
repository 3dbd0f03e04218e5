// k_near.cu -- near-field correction for touching and near triangle pairs
// (FP64, or FP64-accurate double-float point evaluations by default).
//
// For every pair of triangles of one surface that shares a vertex, an edge
// or is identical, the far-field kernel's regular 6-point x 6-point rule is
// wrong (or, for the identical pair, skipped).  This file integrates the
// pair with the Sauter-Schwab regularising maps (Sauter & Schwab, Boundary
// Element Methods, Sec. 5.2; the paper leaves quadrature to its BEM library,
// Sec. 3).  Pairs without a common vertex whose centroids are closer than
// twice the longer of their longest edges (within a surface or across
// domains) are integrated with a collapsed Gauss-Legendre rule on each
// triangle (table 0).  Either way the kernel subtracts exactly what the
// far-field kernel adds, giving
// per-pair 3x3 corrections of V, K, K' (paper App. A); W follows from V by
// its integration-by-parts form: W_ab = curl_a.curl_b sum(V) - k^2 (n_x.n_y) V_ab.
// The corrections of both wavenumbers of a domain are combined with the
// block coefficients of the PMCHWT system (Sec. 2.2) into four 3x3 blocks
// (row1<-psi, row1<-phi, row2<-psi, row2<-phi), applied per matvec by the
// projection kernel.
#include "df_math.cuh"
#include "internal.h"

namespace gbem {

constexpr int NEAR_THREADS = 128;
constexpr int NACC = 27;  // V, K, K' (3x3 complex each)

__device__ __forceinline__ void kernel_eval(const double* x, const double* y, const double* nx, const double* ny,
                                            double kr, double ki, double w, const double* lx, const double* ly,
                                            double (*acc)[2]) {
    const double d0 = x[0] - y[0], d1 = x[1] - y[1], d2 = x[2] - y[2];
    const double r = sqrt(d0 * d0 + d1 * d1 + d2 * d2);
    const double rinv = 1.0 / r;
    double sn, cs;
    sincos(kr * r, &sn, &cs);
    const double a = exp(-ki * r) * rinv * 0.07957747154594767 * w;  // w G magnitude
    const double Gr = a * cs, Gi = a * sn;
    const double u = -ki - rinv;                                   // Re(ik - 1/r)
    const double Fr = (Gr * u - Gi * kr) * rinv, Fi = (Gr * kr + Gi * u) * rinv;
    const double dny = -(d0 * ny[0] + d1 * ny[1] + d2 * ny[2]);    // (y - x).n_y
    const double dnx = d0 * nx[0] + d1 * nx[1] + d2 * nx[2];       // (x - y).n_x
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) {
            const double pp = lx[i] * ly[j];
            acc[3 * i + j][0] += Gr * pp;
            acc[3 * i + j][1] += Gi * pp;
            acc[9 + 3 * i + j][0] += Fr * dny * pp;
            acc[9 + 3 * i + j][1] += Fi * dny * pp;
            acc[18 + 3 * i + j][0] += Fr * dnx * pp;
            acc[18 + 3 * i + j][1] += Fi * dnx * pp;
        }
}

// grid: (pair, wavenumber slot); one CTA integrates one pair at one k.
__global__ void __launch_bounds__(NEAR_THREADS) near_build_kernel(NearArgs A) {
    const int64_t pi = blockIdx.x;
    const int sl = blockIdx.y;
    const int tgt = A.pair_tgt[pi], src = A.pair_src[pi];
    const int code = A.pair_code[pi];
    const int rel = code & 15;
    int pa[3], pb[3];
    for (int i = 0; i < 3; i++) {
        pa[i] = (code >> (4 + 2 * i)) & 3;
        pb[i] = (code >> (10 + 2 * i)) & 3;
    }
    const int dom = A.slot_dom[4 * tgt + 3];
    const double2 k = sl == 0 ? A.k[0] : A.kdom[dom];
    // the own-domain wavenumber applies only to pairs within the target's domain
    const bool live = sl == 0 || A.slot_dom[4 * src + 3] == dom;
    // reordered vertices: shared ones first, in matching order
    double PX[3][3], PY[3][3], OX[3][3], OY[3][3], nx[3], ny[3];
    for (int i = 0; i < 3; i++)
        for (int c = 0; c < 3; c++) {
            PX[i][c] = A.slot_P[(int64_t)tgt * 9 + 3 * pa[i] + c];
            PY[i][c] = A.slot_P[(int64_t)src * 9 + 3 * pb[i] + c];
            OX[i][c] = A.slot_P[(int64_t)tgt * 9 + 3 * i + c];
            OY[i][c] = A.slot_P[(int64_t)src * 9 + 3 * i + c];
        }
    for (int c = 0; c < 3; c++) {
        nx[c] = A.slot_n[(int64_t)tgt * 3 + c];
        ny[c] = A.slot_n[(int64_t)src * 3 + c];
    }
    const double ax = A.slot_area[tgt], ay = A.slot_area[src];
    double acc[NACC][2];
    for (int i = 0; i < NACC; i++) acc[i][0] = acc[i][1] = 0.0;
    // Sauter-Schwab part, accumulated in the ORIGINAL local order
    const double* tab = A.ss_tab[rel];
    const int n = live ? A.ss_n[rel] : 0;
    const double scale = 4.0 * ax * ay;
    for (int idx = threadIdx.x; idx < n; idx += NEAR_THREADS) {
        const double s1 = tab[5 * idx], s2 = tab[5 * idx + 1], t1 = tab[5 * idx + 2], t2 = tab[5 * idx + 3];
        const double w = tab[5 * idx + 4] * scale;
        double x[3], y[3], lxr[3] = {1 - s1, s1 - s2, s2}, lyr[3] = {1 - t1, t1 - t2, t2}, lx[3], ly[3];
        for (int c = 0; c < 3; c++) {
            x[c] = PX[0][c] + s1 * (PX[1][c] - PX[0][c]) + s2 * (PX[2][c] - PX[1][c]);
            y[c] = PY[0][c] + t1 * (PY[1][c] - PY[0][c]) + t2 * (PY[2][c] - PY[1][c]);
        }
        for (int i = 0; i < 3; i++) {
            lx[pa[i]] = lxr[i];
            ly[pb[i]] = lyr[i];
        }
        kernel_eval(x, y, nx, ny, k.x, k.y, w, lx, ly, acc);
    }
    // minus the regular rule the far-field kernel applied (not for identical pairs)
    if (rel != 3 && live) {
        for (int idx = threadIdx.x; idx < QP * QP; idx += NEAR_THREADS) {
            const int qa = idx / QP, qb = idx % QP;
            const double l1 = A.rule[3 * qa], l2 = A.rule[3 * qa + 1], wa = A.rule[3 * qa + 2];
            const double m1 = A.rule[3 * qb], m2 = A.rule[3 * qb + 1], wb = A.rule[3 * qb + 2];
            double x[3], y[3];
            for (int c = 0; c < 3; c++) {
                x[c] = OX[0][c] + l1 * (OX[1][c] - OX[0][c]) + l2 * (OX[2][c] - OX[0][c]);
                y[c] = OY[0][c] + m1 * (OY[1][c] - OY[0][c]) + m2 * (OY[2][c] - OY[0][c]);
            }
            const double lx[3] = {1 - l1 - l2, l1, l2}, ly[3] = {1 - m1 - m2, m1, m2};
            kernel_eval(x, y, nx, ny, k.x, k.y, -wa * wb * ax * ay, lx, ly, acc);
        }
    }
    // block reduction
    __shared__ double red[NEAR_THREADS / 32][NACC][2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = 0; i < NACC; i++)
        for (int c = 0; c < 2; c++) {
            double v = acc[i][c];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) red[warp][i][c] = v;
        }
    __syncthreads();
    if (threadIdx.x < NACC * 2) {
        const int i = threadIdx.x >> 1, c = threadIdx.x & 1;
        double v = 0;
        for (int w = 0; w < NEAR_THREADS / 32; w++) v += red[w][i][c];
        double* out = reinterpret_cast<double*>(A.raw + ((int64_t)pi * A.n_slot_k + sl) * NACC);
        out[2 * i + c] = v;
    }
}

// ---- the same integrals with double-float point evaluations (df_math.cuh):
// GB300 runs FP64 at ~1/64 of its FP32 rate and every point pair costs a
// square root, a reciprocal and a sincos.
//
// Every rule is a tensor product whose innermost direction moves the point of
// one triangle along a line and leaves the other point where it is, so a
// table row is a group: the fixed point, the line of the moving one, the
// weight without the innermost factor.  A thread evaluates the points of one
// group.  Along the line the moving P1 functions and the one of (y - x).n_y,
// (x - y).n_x that is not constant are linear in the innermost coordinate, so
// five complex sums per point carry everything: G, G g, F, F g, F g^2.
// They are expanded to three sums per moving vertex for each of V, K and K'
// (relative accuracy ~1e-13, as the evaluations), and the CTA's groups meet
// in shared memory, where lane (operator, i, j) of each warp multiplies them
// with the fixed point's P1 values and adds up 32 groups; these sums are
// added in FP64.  One point per thread with all 27 complex moments in
// registers (255 of them, eight warps per SM), each reduced over the CTA by
// FP64 shuffles, which ran on the 1/64-rate pipe for longer than the points
// on theirs, took 198 ms (4,620-triangle rib scene); now 57.6 ms.
//
// The regular rule is subtracted by six more groups (one per fixed point)
// whose points do not lie on a line; they sum the expanded form directly.

constexpr int NEAR_S = 9;                    // complex sums of a group: V, K, K' x moving vertex
constexpr int NEAR_ROW = 2 * NEAR_S + 3 + 1;  // (h, l) pairs of a group in shared memory: sums, P1 values, side

struct NearGeomDF {
    dfl v[14][3];  // X0, X1, X2, Y0, Y1, Y2 (reordered vertices), O0, Ou, Ov, Q0, Qu, Qv (original), nx, ny
    dfl scale, axay;
};

__device__ __forceinline__ dfl split_d(double v) {
    const float h = (float)v;
    return dfl{h, (float)(v - (double)h)};
}

__device__ __forceinline__ dfl ddot3(const dfl (&a)[3], const dfl (&b)[3]) {
    return dadd(dadd(dmul(a[0], b[0]), dmul(a[1], b[1])), dmul(a[2], b[2]));
}

// G r^0 = e^{ikr} / r and F = G (ik - 1/r) / r at the difference e (without the 1 / (4 pi))
// (atten: uniform over the CTA; one body for both, which the instruction cache holds)
__device__ __forceinline__ void near_gf(const dfl (&e)[3], dfl kr, dfl ki, bool atten, const NearArgs& A,
                                        const float4* __restrict__ tab, const float2* __restrict__ etab, dfl& Gr, dfl& Gi,
                                        dfl& Fr, dfl& Fi) {
    dfl r, ri;
    dsqrt_rinv(dadd(dadd(dsqr(e[0]), dsqr(e[1])), dsqr(e[2])), r, ri);
    dfl sn, cs;
    dsincos(dmul(kr, r), A.c, tab, sn, cs);
    dfl a = ri, u = dneg(ri);  // Re(ik - 1/r)
    if (atten) {
        a = dmul(a, dexp_neg(dmul(ki, r), A.c, etab));
        u = dsub(u, ki);
    }
    Gr = dmul(a, cs);
    Gi = dmul(a, sn);
    Fr = dmul(dsub(dmul(Gr, u), dmul(Gi, kr)), ri);
    Fi = dmul(dadd(dmul(Gr, kr), dmul(Gi, u)), ri);
}

// out[j] = v[i] with pa[i] = j, without run-time register indexing
__device__ __forceinline__ void permute3(const dfl (&v)[3], const int (&pa)[3], dfl (&out)[3]) {
#pragma unroll
    for (int j = 0; j < 3; j++) out[j] = pa[0] == j ? v[0] : pa[1] == j ? v[1] : v[2];
}
// P1 values (1 - s1, s1 - s2, s2), or with c = 0 their change along (s1, s2)
__device__ __forceinline__ void bary(dfl s1, dfl s2, float c, const int (&pa)[3], dfl (&out)[3]) {
    const dfl v[3] = {dsub(dfl{c, 0.0f}, s1), dsub(s1, s2), s2};
    permute3(v, pa, out);
}

__device__ __forceinline__ void near_group(const NearArgs& A, const NearGeomDF& G, int rel, int idx, const int (&pa)[3],
                                           const int (&pb)[3], dfl kr, dfl ki, bool atten, const float4* __restrict__ tab,
                                           const float2* __restrict__ etab, const float2 (*__restrict__ inner)[4],
                                           float2* __restrict__ row) {
    const float4* T = A.grp[rel] + 4 * (int64_t)idx;
    const float4 fh = T[0], wh = T[1], fl = T[2], wl = T[3];
    const dfl f1 = {fh.x, fl.x}, f2 = {fh.y, fl.y}, m1 = {fh.z, fl.z}, m2 = {fh.w, fl.w};
    const dfl d1 = {wh.x, wl.x}, d2 = {wh.y, wl.y}, w = dmul(dfl{wh.z, wl.z}, G.scale);
    const bool ymoves = wh.w == 0.0f;  // x fixed
    // e = x - y = e0 + g dv along the line
    const dfl(*Fx)[3] = G.v + (ymoves ? 0 : 3);
    const dfl(*Mv)[3] = G.v + (ymoves ? 3 : 0);
    dfl e0[3], dv[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const dfl fx = dadd(dadd(Fx[0][c], dmul(f1, Fx[1][c])), dmul(f2, Fx[2][c]));
        const dfl mv = dadd(dadd(Mv[0][c], dmul(m1, Mv[1][c])), dmul(m2, Mv[2][c]));
        const dfl sl = dadd(dmul(d1, Mv[1][c]), dmul(d2, Mv[2][c]));
        e0[c] = ymoves ? dsub(fx, mv) : dsub(mv, fx);
        dv[c] = ymoves ? dneg(sl) : sl;
    }
    dfl g0[2], g1[2], h0[2], h1[2], h2[2];
#pragma unroll
    for (int c = 0; c < 2; c++) g0[c] = g1[c] = h0[c] = h1[c] = h2[c] = dfl{0.0f, 0.0f};
    for (int q = 0; q < A.ng; q++) {
        const float2 gq = inner[q][0], w0 = inner[q][1], w1 = inner[q][2], w2 = inner[q][3];
        const dfl g = {gq.x, gq.y}, c0 = {w0.x, w0.y}, c1 = {w1.x, w1.y}, c2 = {w2.x, w2.y};
        dfl e[3];
#pragma unroll
        for (int c = 0; c < 3; c++) e[c] = dadd(e0[c], dmul(g, dv[c]));
        dfl Gr, Gi, Fr, Fi;
        near_gf(e, kr, ki, atten, A, tab, etab, Gr, Gi, Fr, Fi);
        dmac(g0[0], Gr, c0, 1.0f);
        dmac(g0[1], Gi, c0, 1.0f);
        dmac(g1[0], Gr, c1, 1.0f);
        dmac(g1[1], Gi, c1, 1.0f);
        dmac(h0[0], Fr, c0, 1.0f);
        dmac(h0[1], Fi, c0, 1.0f);
        dmac(h1[0], Fr, c1, 1.0f);
        dmac(h1[1], Fi, c1, 1.0f);
        dmac(h2[0], Fr, c2, 1.0f);
        dmac(h2[1], Fi, c2, 1.0f);
    }
    // (y - x).n_y = -e.n_y and (x - y).n_x = e.n_x: the one of the moving triangle is constant along the line
    const dfl(&nf)[3] = G.v[ymoves ? 12 : 13];
    const dfl(&nm)[3] = G.v[ymoves ? 13 : 12];
    dfl cst = ddot3(e0, nm), lr = ddot3(e0, nf), ls = ddot3(dv, nf);
    if (ymoves) cst = dneg(cst);
    else {
        lr = dneg(lr);
        ls = dneg(ls);
    }
    dfl u[3], p[3], s[3];
    bary(f1, f2, 1.0f, ymoves ? pa : pb, u);
    bary(m1, m2, 1.0f, ymoves ? pb : pa, p);
    bary(d1, d2, 0.0f, ymoves ? pb : pa, s);
    // sums per moving vertex: V from G; the constant factor's operator and the linear one's from F
    const int oc = ymoves ? 3 : 6, ol = ymoves ? 6 : 3;  // K, K' rows
#pragma unroll
    for (int c = 0; c < 2; c++) {
        g0[c] = two_sum(g0[c].h, g0[c].l);
        g1[c] = two_sum(g1[c].h, g1[c].l);
        h0[c] = two_sum(h0[c].h, h0[c].l);
        h1[c] = two_sum(h1[c].h, h1[c].l);
        h2[c] = two_sum(h2[c].h, h2[c].l);
        // F times the linear factor: l0 + l1 g, as moments 0 and 1
        const dfl l0 = dadd(dmul(lr, h0[c]), dmul(ls, h1[c])), l1 = dadd(dmul(lr, h1[c]), dmul(ls, h2[c]));
        const dfl k0 = dmul(cst, h0[c]), k1 = dmul(cst, h1[c]);
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const dfl pw = dmul(p[j], w), sw = dmul(s[j], w);
            const dfl V = dadd(dmul(pw, g0[c]), dmul(sw, g1[c]));
            const dfl K = dadd(dmul(pw, k0), dmul(sw, k1)), L = dadd(dmul(pw, l0), dmul(sw, l1));
            row[2 * j + c] = make_float2(V.h, V.l);
            row[2 * (oc + j) + c] = make_float2(K.h, K.l);
            row[2 * (ol + j) + c] = make_float2(L.h, L.l);
        }
    }
#pragma unroll
    for (int i = 0; i < 3; i++) row[2 * NEAR_S + i] = make_float2(u[i].h, u[i].l);
    row[2 * NEAR_S + 3] = make_float2(ymoves ? 0.0f : 1.0f, 0.0f);
}

// Minus the regular rule the far-field kernel applied: point qa of the target against the source's points.
__device__ __forceinline__ void near_regular(const NearArgs& A, const NearGeomDF& G, int qa, dfl kr, dfl ki, bool atten,
                                             const float4* __restrict__ tab, const float2* __restrict__ etab,
                                             float2* __restrict__ row) {
    const dfl l1 = {A.rule_h[3 * qa], A.rule_l[3 * qa]}, l2 = {A.rule_h[3 * qa + 1], A.rule_l[3 * qa + 1]};
    const dfl wa = {A.rule_h[3 * qa + 2], A.rule_l[3 * qa + 2]};
    const dfl w = dneg(dmul(wa, G.axay));
    dfl x[3];
#pragma unroll
    for (int c = 0; c < 3; c++) x[c] = dadd(dadd(G.v[6][c], dmul(l1, G.v[7][c])), dmul(l2, G.v[8][c]));
    dfl acc[NEAR_S][2];
#pragma unroll
    for (int k = 0; k < NEAR_S; k++) acc[k][0] = acc[k][1] = dfl{0.0f, 0.0f};
    for (int qb = 0; qb < QP; qb++) {
        const dfl m1 = {A.rule_h[3 * qb], A.rule_l[3 * qb]}, m2 = {A.rule_h[3 * qb + 1], A.rule_l[3 * qb + 1]};
        const dfl wb = {A.rule_h[3 * qb + 2], A.rule_l[3 * qb + 2]};
        dfl e[3];
#pragma unroll
        for (int c = 0; c < 3; c++)
            e[c] = dsub(x[c], dadd(dadd(G.v[9][c], dmul(m1, G.v[10][c])), dmul(m2, G.v[11][c])));
        dfl Gr, Gi, Fr, Fi;
        near_gf(e, kr, ki, atten, A, tab, etab, Gr, Gi, Fr, Fi);
        const dfl wt = dmul(w, wb), dy = dneg(ddot3(e, G.v[13])), dx = ddot3(e, G.v[12]);
        const dfl ly[3] = {dsub(dsub(dfl{1.0f, 0.0f}, m1), m2), m1, m2};
        const dfl f[3][2] = {{dmul(Gr, wt), dmul(Gi, wt)},
                             {dmul(dmul(Fr, wt), dy), dmul(dmul(Fi, wt), dy)},
                             {dmul(dmul(Fr, wt), dx), dmul(dmul(Fi, wt), dx)}};
#pragma unroll
        for (int o = 0; o < 3; o++)
#pragma unroll
            for (int j = 0; j < 3; j++)
#pragma unroll
                for (int c = 0; c < 2; c++) dmac(acc[3 * o + j][c], f[o][c], ly[j], 1.0f);
    }
#pragma unroll
    for (int k = 0; k < NEAR_S; k++)
#pragma unroll
        for (int c = 0; c < 2; c++) {
            const dfl v = two_sum(acc[k][c].h, acc[k][c].l);
            row[2 * k + c] = make_float2(v.h, v.l);
        }
    const dfl lx[3] = {dsub(dsub(dfl{1.0f, 0.0f}, l1), l2), l1, l2};
#pragma unroll
    for (int i = 0; i < 3; i++) row[2 * NEAR_S + i] = make_float2(lx[i].h, lx[i].l);
    row[2 * NEAR_S + 3] = make_float2(0.0f, 0.0f);
}

// grid: (pair, wavenumber slot); one CTA integrates one pair at one k.
__global__ void __launch_bounds__(NEAR_THREADS, 4) near_build_df_kernel(NearArgs A) {
    __shared__ float4 tab[128];
    __shared__ float2 etab[64];
    __shared__ float2 inner[NEAR_NG_MAX][4];  // innermost rule: g, w, w g, w g^2
    __shared__ NearGeomDF G;
    __shared__ float2 rows[NEAR_THREADS][NEAR_ROW];
    __shared__ double red[NEAR_THREADS / 32][NACC][2];
    const int64_t pi = blockIdx.x;
    const int sl = blockIdx.y, tid = threadIdx.x;
    const int tgt = A.pair_tgt[pi], src = A.pair_src[pi];
    const int code = A.pair_code[pi];
    const int rel = code & 15;
    double* out = reinterpret_cast<double*>(A.raw + ((int64_t)pi * A.n_slot_k + sl) * NACC);
    const int dom = A.slot_dom[4 * tgt + 3];
    // the own-domain wavenumber applies only to pairs within the target's domain
    if (sl != 0 && A.slot_dom[4 * src + 3] != dom) {
        if (tid < NACC * 2) out[tid] = 0.0;
        return;
    }
    int pa[3], pb[3];
#pragma unroll
    for (int i = 0; i < 3; i++) {
        pa[i] = (code >> (4 + 2 * i)) & 3;
        pb[i] = (code >> (10 + 2 * i)) & 3;
    }
    const float4 kk = sl == 0 ? A.k0df : A.kdf[dom];
    const dfl kr = {kk.x, kk.y}, ki = {kk.z, kk.w};
    for (int i = tid; i < 128; i += NEAR_THREADS) tab[i] = A.sctab[i];
    for (int i = tid; i < 64; i += NEAR_THREADS) etab[i] = A.extab[i];
    for (int i = tid; i < 4 * A.ng; i += NEAR_THREADS) (&inner[0][0])[i] = A.inner[i];
    if (tid < 42) {
        // the pair's geometry, one component per thread; FP64 differences formed before the split
        const int v = tid / 3, c = tid - 3 * v;
        double val;
        if (v < 12) {
            const bool y = (v / 3) & 1, orig = v >= 6;
            const double* P = A.slot_P + (int64_t)(y ? src : tgt) * 9 + c;
            const int m = v % 3;
            // reordered: (P0, P1 - P0, P2 - P1) of the rule's vertex order; original: (P0, P1 - P0, P2 - P0)
            const int sh = y ? 10 : 4, at = orig ? m : (code >> (sh + 2 * m)) & 3;
            const int from = orig ? 0 : (code >> (sh + 2 * (m - 1))) & 3;
            val = P[3 * at];
            if (m > 0) val -= P[3 * from];
        } else {
            val = A.slot_n[(int64_t)(v == 12 ? tgt : src) * 3 + c];
        }
        G.v[v][c] = split_d(val);
    } else if (tid == 42) {
        G.scale = split_d(4.0 * A.slot_area[tgt] * A.slot_area[src] * 0.07957747154594767);
    } else if (tid == 43) {
        G.axay = split_d(A.slot_area[tgt] * A.slot_area[src] * 0.07957747154594767);
    }
    __syncthreads();
    const bool atten = kk.z != 0.0f || kk.w != 0.0f;
    const int n = A.grp_n[rel];
    // the regular groups take the last warp of the last batch where that is free, else a batch of their own
    const int base = (n - 1) / NEAR_THREADS * NEAR_THREADS;
    const int reg0 = rel == 3 ? n : base + (n - base <= NEAR_THREADS - 32 ? NEAR_THREADS - 32 : NEAR_THREADS);
    const int n_all = rel == 3 ? n : reg0 + QP;  // (not for identical pairs)
    // lane (operator, i, j) sums its moment over its warp's groups
    const int lane = tid & 31, warp = tid >> 5;
    const int op = lane / 9, ij = lane - 9 * op, mi = ij / 3, mj = ij - 3 * mi;
    double tr = 0, ti = 0;
    for (int b = 0; b < n_all; b += NEAR_THREADS) {
        const int idx = b + tid;
        float2* row = rows[tid];
        if (idx < n) {
            near_group(A, G, rel, idx, pa, pb, kr, ki, atten, tab, etab, inner, row);
        } else if (idx >= reg0 && idx < n_all) {
            near_regular(A, G, idx - reg0, kr, ki, atten, tab, etab, row);
        }
        __syncwarp();
        if (lane < NACC) {
            dfl sr = {0.0f, 0.0f}, si = {0.0f, 0.0f};
            for (int g = 0; g < 32; g++) {
                const int i = b + warp * 32 + g;
                if (!(i < n || (i >= reg0 && i < n_all))) continue;
                const float2* r = rows[warp * 32 + g];
                const bool xmoves = r[2 * NEAR_S + 3].x != 0.0f;
                const float2 u = r[2 * NEAR_S + (xmoves ? mj : mi)];
                const float2 *v = r + 2 * (3 * op + (xmoves ? mi : mj)), vr = v[0], vi = v[1];
                dmac(sr, dfl{vr.x, vr.y}, dfl{u.x, u.y}, 1.0f);
                dmac(si, dfl{vi.x, vi.y}, dfl{u.x, u.y}, 1.0f);
            }
            // 32 groups in FP32 pairs, the rest in FP64: mean error of 24 FP64 products on four small scenes against
            // native FP64 1.490e-14 (1.515e-14 with pairs over a whole rule, 1.524e-14 with FP64 sums of every thread's points)
            tr += (double)sr.h + (double)sr.l;
            ti += (double)si.h + (double)si.l;
        }
        __syncwarp();
    }
    if (lane < NACC) {
        red[warp][lane][0] = tr;
        red[warp][lane][1] = ti;
    }
    __syncthreads();
    if (tid < NACC * 2) {
        const int i = tid >> 1, c = tid & 1;
        double v = 0;
        for (int w = 0; w < NEAR_THREADS / 32; w++) v += red[w][i][c];
        out[2 * i + c] = v;
    }
}

__global__ void near_combine_kernel(NearCombineArgs A) {
    const int64_t pi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (pi >= A.n_pairs) return;
    const int tgt = A.pair_tgt[pi], src = A.pair_src[pi];
    const int dom = A.slot_v[tgt].w;
    double cc[3][3], nn = 0;
    for (int c = 0; c < 3; c++) nn += A.slot_n[(int64_t)tgt * 3 + c] * A.slot_n[(int64_t)src * 3 + c];
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) {
            double s = 0;
            for (int c = 0; c < 3; c++)
                s += A.slot_curl[(int64_t)tgt * 9 + 3 * i + c] * A.slot_curl[(int64_t)src * 9 + 3 * j + c];
            cc[i][j] = s;
        }
    double B[4][9][2];
    for (int b = 0; b < 4; b++)
        for (int e = 0; e < 9; e++) B[b][e][0] = B[b][e][1] = 0.0;
    for (int sl = 0; sl < A.n_slot_k; sl++) {
        const SlotCoef cf = A.coef[dom * 2 + sl];
        const double2* R = A.raw + (pi * A.n_slot_k + sl) * NACC;
        double ig_r = 0, ig_i = 0;
        for (int e = 0; e < 9; e++) {
            ig_r += R[e].x;
            ig_i += R[e].y;
        }
        for (int i = 0; i < 3; i++)
            for (int j = 0; j < 3; j++) {
                const int e = 3 * i + j;
                const double2 V = R[e], K = R[9 + e], Kp = R[18 + e];
                // W = curl.curl * sum(V) - k^2 (n_x.n_y) V
                const double kvr = cf.k2re * V.x - cf.k2im * V.y, kvi = cf.k2re * V.y + cf.k2im * V.x;
                const double Wr = cc[i][j] * ig_r - nn * kvr, Wi = cc[i][j] * ig_i - nn * kvi;
                B[0][e][0] += cf.cV * V.x;
                B[0][e][1] += cf.cV * V.y;
                B[1][e][0] -= cf.cK * K.x;
                B[1][e][1] -= cf.cK * K.y;
                B[2][e][0] += cf.cKp * Kp.x;
                B[2][e][1] += cf.cKp * Kp.y;
                B[3][e][0] += cf.cW * Wr;
                B[3][e][1] += cf.cW * Wi;
            }
    }
    for (int b = 0; b < 4; b++)
        for (int e = 0; e < 9; e++) {
            A.nb64[(pi * 4 + b) * 9 + e] = make_double2(B[b][e][0], B[b][e][1]);
            A.nb32[(pi * 4 + b) * 9 + e] = make_float2((float)B[b][e][0], (float)B[b][e][1]);
        }
}

cudaError_t launch_near_build(const NearArgs& a, cudaStream_t s) {
    if (a.n_pairs <= 0) return cudaSuccess;
    // one launch per <= 65535 pairs is not needed: grid.x may be up to 2^31-1
    if (a.use_df) near_build_df_kernel<<<dim3((unsigned)a.n_pairs, a.n_slot_k), NEAR_THREADS, 0, s>>>(a);
    else near_build_kernel<<<dim3((unsigned)a.n_pairs, a.n_slot_k), NEAR_THREADS, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_near_combine(const NearCombineArgs& a, cudaStream_t s) {
    if (a.n_pairs <= 0) return cudaSuccess;
    near_combine_kernel<<<(unsigned)((a.n_pairs + 127) / 128), 128, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace gbem
