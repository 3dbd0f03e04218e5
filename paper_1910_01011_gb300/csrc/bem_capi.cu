// bem_capi.cu -- the C ABI (include/bem.h): context, device memory, and the
// operator application pipeline
//   gather (trial densities) -> far field (FP32 or FP64) -> projection onto
//   P1 test functions with the touching-pair correction -> vertex reduction.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <vector>

#include "ctx.h"
#include "internal.h"

using namespace gbem;

// ------------------------------------------------------------------ helpers

#define CK(expr)                                                                   \
    do {                                                                           \
        cudaError_t e_ = (expr);                                                   \
        if (e_ != cudaSuccess) return ctx->fail(BEM_ERR_CUDA, std::string(#expr) + ": " + cudaGetErrorString(e_)); \
    } while (0)

int bem_ctx::fail(int code, const std::string& msg) {
    err = msg;
    return code;
}

// Allocation generations are unique across contexts, so a cached group
// launch never mistakes a new context at a reused address for the old one.
static uint64_t next_gen() {
    static std::atomic<uint64_t> g{0};
    return ++g;
}

// One allocation within the context's budget and the shared one; null, *rc and why otherwise.
void* bem_ctx::take(size_t bytes, int* rc, std::string& why) {
    if (bytes == 0) bytes = 16;
    if (opts.hbm_budget_bytes > 0 && (int64_t)(used_bytes + bytes) > opts.hbm_budget_bytes) {
        *rc = BEM_ERR_OUT_OF_BUDGET;
        why = "device memory budget exceeded (" + std::to_string(used_bytes + bytes) + " > " +
              std::to_string(opts.hbm_budget_bytes) + " bytes)";
        return nullptr;
    }
    if (pool) {
        const int64_t after = pool->fetch_add((int64_t)bytes) + (int64_t)bytes;
        if (pool_limit > 0 && after > pool_limit) {
            pool->fetch_sub((int64_t)bytes);
            *rc = BEM_ERR_OUT_OF_BUDGET;
            why = "shared device memory budget exceeded (" + std::to_string(after) + " > " + std::to_string(pool_limit) +
                  " bytes)";
            return nullptr;
        }
    }
    void* p = nullptr;
    cudaError_t e = cudaMalloc(&p, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        if (pool) pool->fetch_sub((int64_t)bytes);
        *rc = BEM_ERR_CUDA;
        why = std::string("cudaMalloc: ") + cudaGetErrorString(e);
        return nullptr;
    }
    allocs.push_back({p, bytes});
    used_bytes += bytes;
    gen = next_gen();
    peak_bytes = std::max(peak_bytes, used_bytes);
    *rc = BEM_OK;
    return p;
}

// Memory that a call cannot do without: what only speeds calls up goes before it is refused.
void* bem_ctx::dalloc(size_t bytes, int* rc) {
    std::string why;
    void* p = take(bytes, rc, why);
    if (!p && give_back()) p = take(bytes, rc, why);
    if (p) {
        note_need();
    } else {
        short_of_memory = true;
        fail(*rc, why);
    }
    return p;
}

// Memory that only speeds calls up: nothing else goes for it, and a refusal is not an error.
void* bem_ctx::try_alloc(size_t bytes) {
    int rc;
    std::string why;
    void* p = take(bytes, &rc, why);
    if (!p) optional_wait = OPTIONAL_WAIT;
    return p;
}

// Whether `grow` bytes more may go to such memory: within the context's budget,
// within half of a shared one next to all that is held of and promised out of
// it, and as much again left free on the device.  After a refusal by the device
// the next OPTIONAL_WAIT calls do not ask it again.
bool bem_ctx::room_for(size_t grow) {
    if (grow == 0) return true;
    if (frugal) return false;
    if (opts.hbm_budget_bytes > 0 && (int64_t)(used_bytes + grow) > opts.hbm_budget_bytes) return false;
    if (pool_wanted && pool_wanted->load()) return false;
    if (pool && pool_limit > 0 &&
        2 * (pool->load() + (pool_reserved ? pool_reserved->load() : 0) + (int64_t)grow) > pool_limit)
        return false;
    if (optional_wait > 0) {
        optional_wait--;
        return false;
    }
    size_t free = 0, total = 0;
    if (cudaMemGetInfo(&free, &total) != cudaSuccess || free < 2 * grow) {
        cudaGetLastError();
        optional_wait = OPTIONAL_WAIT;
        return false;
    }
    return true;
}

// Frees what only speeds calls up, unless a call in progress holds pointers into it.
bool bem_ctx::give_back() {
    if (pinned > 0) return false;
    const bool part = partial && partial_bytes > partial_need, multi = multi_buf && multi_buf_bytes > multi_need;
    if (!part && !multi && !mm_buf && !mmg.buf) return false;
    cudaStreamSynchronize(stream);
    if (part) {
        dfree(partial);
        partial = nullptr;
        partial_bytes = 0;
    }
    if (multi) {
        dfree(multi_buf);
        multi_buf = nullptr;
        multi_buf_bytes = 0;
    }
    dfree(mm_buf);
    mm_buf = nullptr;
    mm_bytes = 0;
    if (mmg.buf) {
        dfree(mmg.buf);
        mmg = MmGeom();
    }
    note_need();
    return true;
}

size_t bem_ctx::optional_bytes() const {
    return (partial_bytes > partial_need ? partial_bytes - partial_need : 0) +
           (multi_buf_bytes > multi_need ? multi_buf_bytes - multi_need : 0) + mm_bytes + mmg.bytes;
}

void bem_ctx::note_need() {
    const size_t o = optional_bytes();
    optional_now.store((int64_t)o);
    peak_need = std::max(peak_need, used_bytes - std::min(o, used_bytes));
}

void bem_ctx::dfree(void* p) {
    if (!p) return;
    for (size_t i = 0; i < allocs.size(); i++)
        if (allocs[i].first == p) {
            gen = next_gen();
            used_bytes -= allocs[i].second;
            if (pool) pool->fetch_sub((int64_t)allocs[i].second);
            cudaFree(p);
            allocs.erase(allocs.begin() + i);
            return;
        }
}

template <class T>
static int upload(bem_ctx* ctx, T** dst, const std::vector<T>& v) {
    int rc;
    *dst = (T*)ctx->dalloc(v.size() * sizeof(T), &rc);
    if (rc) return rc;
    if (!v.empty()) CK(cudaMemcpyAsync(*dst, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, ctx->stream));
    return BEM_OK;
}

void destroy_solver_state(bem_ctx* ctx);  // bem_solve.cu / k_sparse.cu (objects only; memory is freed here)

static void release_group(bem_ctx* ctx) {
    if (!ctx->group) return;
    if (ctx->group->exec) cudaGraphExecDestroy(ctx->group->exec);
    if (ctx->group->cap) cudaStreamDestroy(ctx->group->cap);
    delete ctx->group;  // its device buffers belong to ctx->allocs
    ctx->group = nullptr;
}

static void release_device(bem_ctx* ctx) {
    cudaSetDevice(ctx->device);
    cudaStreamSynchronize(ctx->stream);
    release_group(ctx);
    ctx->gen = next_gen();
    for (auto& a : ctx->allocs) cudaFree(a.first);
    ctx->allocs.clear();
    if (ctx->pool) ctx->pool->fetch_sub((int64_t)ctx->used_bytes);
    ctx->used_bytes = 0;
    ctx->dev = DeviceGeom();
    ctx->ready = false;
    ctx->near_ready = false;
    ctx->block_cache.clear();
    ctx->osrc_ready = false;
    ctx->rhs_ready = false;
    ctx->asm_ready = false;
    ctx->asm64_ready = false;
    ctx->asm64 = nullptr;
    ctx->asm64_exp = nullptr;
    ctx->dg_work = nullptr;
    ctx->dg_work_bytes = 0;
    ctx->df_exp = nullptr;
    ctx->df_work = nullptr;
    ctx->df_work_bytes = 0;
    ctx->asm_planes = nullptr;
    ctx->asm_work = nullptr;
    ctx->asm_work_bytes = 0;
    ctx->partial = nullptr;
    ctx->partial_bytes = ctx->partial_need = 0;
    ctx->optional_wait = 0;
    ctx->field_buf = nullptr;
    ctx->field_buf_bytes = 0;
    ctx->far_work = nullptr;
    for (int& k : ctx->far_work_key) k = -1;
    ctx->multi_buf = nullptr;
    ctx->multi_buf_bytes = ctx->multi_need = 0;
    ctx->multi64_buf = nullptr;
    ctx->multi64_buf_bytes = 0;
    ctx->dfg = bem_ctx::DfGeom();
    ctx->dfv_buf = nullptr;
    ctx->dfv_bytes = 0;
    ctx->multi_work = nullptr;
    ctx->multi_n_work = 0;
    for (int& k : ctx->multi_key) k = -1;
    ctx->mmg = bem_ctx::MmGeom();
    ctx->mm_buf = nullptr;
    ctx->mm_bytes = 0;
    ctx->optional_now.store(0);
    ctx->pmchwt_near = NearSet();
    destroy_solver_state(ctx);
}

namespace gbem {

void invalidate_basis(bem_ctx* ctx);
void invalidate_recycle(bem_ctx* ctx);
size_t gemm_work_bytes(int64_t mpad, int64_t kpad, int64_t n_rhs);  // k_gemm.cu

// Eviction by the request loop: every device allocation of the context goes;
// the host description (meshes, materials, transducer) stays and the device
// state is rebuilt on next use.
void release_device_memory(bem_ctx* ctx) { release_device(ctx); }

void multi_chunking(int n_tiles, int64_t n_pts, int64_t R, int* n_chunks, int* chunk_tiles) {
    const int groups = (int)((R + MRG - 1) / MRG);
    int nc = std::max(1, (152 * 2 * 8 + n_tiles * groups - 1) / std::max(1, n_tiles * groups));
    nc = std::max(nc, (n_tiles + CHUNK_MAX - 1) / CHUNK_MAX);
    const size_t per_chunk = (size_t)R * 2 * NCOMP * n_pts * sizeof(float);
    const int nc_mem = (int)std::max<size_t>(1, ((size_t)2 << 30) / std::max<size_t>(1, per_chunk));
    if (nc > nc_mem) nc = std::max(nc_mem, (n_tiles + CHUNK_MAX - 1) / CHUNK_MAX);
    nc = std::max(1, std::min(nc, n_tiles));
    const int ct = (n_tiles + nc - 1) / nc;
    *chunk_tiles = ct;
    *n_chunks = (n_tiles + ct - 1) / ct;
}

// Chunks of the FP64 multi-vector far field: about 8 CTAs per SM over
// (target tile, chunk, slot, group of RG64), no more (each chunk adds R x 2 x
// NCOMP x n_pts doubles of partial potentials).  The double-float kernel has
// groups of two, so up to twice as many CTAs: 2,964-triangle rib scene, 5
// vectors, 40.2 ms; with its own groups counted, and so longer chunks, 41.0 ms.
void multi64_chunking(int n_tiles, int64_t R, int* n_chunks, int* chunk_tiles) {
    const int64_t groups = (R + RG64 - 1) / RG64;
    int64_t nc = (152 * 8 + 2 * groups * n_tiles - 1) / std::max<int64_t>(1, 2 * groups * n_tiles);
    nc = std::max<int64_t>(1, std::min<int64_t>(nc, n_tiles));
    const int ct = (int)((n_tiles + nc - 1) / nc);
    *chunk_tiles = ct;
    *n_chunks = (n_tiles + ct - 1) / ct;
}

// Device bytes a solve of n_exc excitations with options o may need at its
// peak, from the mesh sizes alone (no device state is needed); every term
// follows one allocation of the solver, rounded up, with a 10 % margin.
int64_t estimate_solve_bytes(const bem_ctx* ctx, int64_t n_exc, const bem_solve_opts& o_in) {
    int64_t T = 0, nv = 0, tiles = 0;
    for (auto& d : ctx->doms) {
        T += d.nt;
        nv += d.nv;
        tiles += (d.nt + TT - 1) / TT;
    }
    bem_solve_opts o = o_in;
    o.operator_mode = resolved_operator_mode(o.operator_mode, 2 * nv);
    // correction pairs: touching (about 13 per triangle) and near (20-80 per
    // triangle on the meshes measured): the exact count once the geometry exists
    const int64_t pairs = ctx->ready ? (int64_t)ctx->geo.np_src.size() : 96 * T;
    const int64_t N = 2 * nv, pts = tiles * TP, slots = tiles * TT;
    const int64_t ne = (int64_t)ctx->tr_r.size();
    int64_t b = 0;
    // geometry, densities, staging vectors
    b += pts * 152 + slots * 460 + pairs * 12 + N * 64 + tiles * 64;
    // near-field blocks (c128 + c64) and their build scratch
    b += pairs * 36 * 24 + std::min<int64_t>(pairs, 1 << 20) * 2 * 27 * 16;
    // far-field partial potentials of the longest chunks (one buffer for the FP32 operator and the FP64 residual, which
    // is the larger); short chunks' and the tensor-core far field's memory is not needed and not counted
    int nc = 1, ct = 1;
    ctx->chunking((int)tiles, (int)tiles, &nc, &ct, true);
    b += (int64_t)nc * 2 * NCOMP * pts * 8;
    // right-hand sides, solutions, piston data
    b += n_exc * (2 * N * 16 + slots * 6 * 16 + ne * 16) + ne * 32 * 32 + 3 * N * 16;
    // GMRES basis and work (per lockstep column)
    const int64_t R = o.batch_rhs > 1 ? solve_batch_width(o, n_exc) : 1;
    b += (int64_t)(o.restart + 1) * R * N * 16 + 2 * R * N * 16 + (int64_t)(o.restart + 2) * 120 * R * 16 * 3 + 8 * R;
    b += (int64_t)R * ((o.restart + 1) * o.restart + 3 * o.restart + 1) * 16 + 32 * R + 16;  // device least squares
    if (o.precondition && o.flexible) b += (int64_t)o.restart * R * N * 16;  // flexible basis
    if (o.block_gmres) {  // FP32 basis and work blocks, dot partials, coefficient blocks
        const int64_t gx = ((int64_t)(o.restart + 1) * R + 63) / 64;
        b += (int64_t)(o.restart + 3) * R * N * 8 +
             16 * std::max<int64_t>((int64_t)(o.restart + 1) * R * R * 8, R * 64 * std::max<int64_t>(gx, 608)) +
             16 * (2 * (int64_t)(o.restart + 1) * R * R + R * R) + 8 * (int64_t)(o.restart + 1) * R * R + 8 +
             16 * ((int64_t)(o.restart + 1) * R * o.restart * R + (int64_t)(o.restart + 1) * R * R);  // Hessenberg mirror
    }
    b += 4 * R * N * 16;
    if (o.precondition) {
        const int64_t L = ctx->opts.n_pade, nnz = 8 * nv, ms = 2 * L * R, nd = (int64_t)ctx->doms.size();
        b += nnz * 20 + (nv + 1) * 8 + 2 * nv * 8 + nv * 4 + nd * (L + 4) * 16;
        b += 6 * ms * nv * 16 + ms * (16 * nd + 128 * 4 * 8 + 64) + 4 * R * nv * 16;
        b += 5 * ms * nv * 8 + 16 * nv * 8 + 2 * nv * 4;  // FP32 vectors and matrix copies of the loose solves
    }
    // several right-hand sides in one matrix-free FP32 far-field launch
    if (o.operator_mode == 0 && o.precision == BEM_PREC_FP32 && R > 1) {
        int ncm = 1, ctm = 1;
        multi_chunking((int)tiles, pts, R, &ncm, &ctm);
        b += R * (pts * 16 + 2 * slots * 16 + (int64_t)ncm * 2 * NCOMP * pts * 4) +
             tiles * ncm * 2 * ((R + MRG - 1) / MRG) * 16;
    }
    // FP64 residuals of several vectors in one matrix-free launch
    if (o.operator_mode == 0 && R > 1) {
        int nc64 = 1, ct64 = 1;
        multi64_chunking((int)tiles, R, &nc64, &ct64);
        b += R * (pts * 32 + 2 * slots * 32 + (int64_t)nc64 * 2 * NCOMP * pts * 8);
    }
    // double-float far field: split geometry and tables; split densities of R vectors
    if (o.operator_mode == 0 && ctx->opts.fp64_far == 0)
        b += 32 * (pts + slots + tiles) + 4096 + R * (pts * 32 + 2 * slots * 32 + 16);
    // recycled solution space: Q, U' and their coefficients
    if (o.recycle > 0) b += (int64_t)o.recycle * (2 * N * 16 + 64 * 16);
    if (o.operator_mode == 1) {
        const int64_t mp = (N + 127) / 128 * 128, kp = (N + 31) / 32 * 32;
        const int64_t planes = 6 * mp * kp * 2;
        const int64_t a64 = (int64_t)(digits_bytes(N) + digits_convert_bytes(N) + digits_exp_bytes(N)) +
                            (int64_t)digits_work_bytes(N, std::min<int64_t>(R, 16));
        if (o.precision == BEM_PREC_FP32)
            b += std::max(planes + 8 * N * N, planes + a64) + (int64_t)gemm_work_bytes(mp, kp, R);
        else
            b += a64;
    }
    return b + b / 10 + ((int64_t)64 << 20);
}

}  // namespace gbem

// ------------------------------------------------------------------ set-up

int bem_ctx::finalize() {
    bem_ctx* const ctx = this;
    if (ready) return BEM_OK;
    CK(cudaSetDevice(device));
    if (!build_quadrature(quad, opts.n_gauss_singular)) return fail(BEM_ERR_STATE, "quadrature derivation failed");
    std::string msg = build_geometry(doms, quad, geo);
    if (!msg.empty()) return fail(BEM_ERR_MESH_INVALID, msg);
    const Geometry& g = geo;
    DeviceGeom& d = dev;
    int rc;
    // fp32 / fp64 point and triangle data
    std::vector<float4> pg32(g.n_pts), tg32(g.n_slots);
    std::vector<double4> pg64(g.n_pts), tg64(g.n_slots), tc(g.n_tiles);
    for (int64_t p = 0; p < g.n_pts; p++) {
        pg32[p] = make_float4((float)g.pt_delta[3 * p], (float)g.pt_delta[3 * p + 1], (float)g.pt_delta[3 * p + 2],
                              (float)g.pt_w[p]);
        pg64[p] = make_double4(g.pt_delta[3 * p], g.pt_delta[3 * p + 1], g.pt_delta[3 * p + 2], g.pt_w[p]);
    }
    std::vector<float4> pgp32(g.n_pts);
    for (int64_t s = 0; s < g.n_slots; s++) {
        float4 tri[QP];
        for (int q = 0; q < QP; q++) tri[q] = pg32[s * QP + q];
        pair_interleave(tri, pgp32.data() + s * QP);
    }
    for (int64_t s = 0; s < g.n_slots; s++) {
        tg32[s] = make_float4((float)g.slot_n[3 * s], (float)g.slot_n[3 * s + 1], (float)g.slot_n[3 * s + 2],
                              (float)g.slot_h[s]);
        tg64[s] = make_double4(g.slot_n[3 * s], g.slot_n[3 * s + 1], g.slot_n[3 * s + 2], g.slot_h[s]);
    }
    for (int t = 0; t < g.n_tiles; t++)
        tc[t] = make_double4(g.tile_c[4 * t], g.tile_c[4 * t + 1], g.tile_c[4 * t + 2], g.tile_c[4 * t + 3]);
    std::vector<int2> dt(g.n_dom);
    for (int i = 0; i < g.n_dom; i++) dt[i] = make_int2(g.dom_tile_begin[i], g.dom_tile_end[i]);
    std::vector<int4> sv(g.n_slots);
    for (int64_t s = 0; s < g.n_slots; s++)
        sv[s] = make_int4(g.slot_v[4 * s], g.slot_v[4 * s + 1], g.slot_v[4 * s + 2], g.slot_v[4 * s + 3]);
    if ((rc = upload(this, &d.pg32, pg32)) || (rc = upload(this, &d.pgp32, pgp32)) || (rc = upload(this, &d.tg32, tg32)) || (rc = upload(this, &d.pg64, pg64)) ||
        (rc = upload(this, &d.tg64, tg64)) || (rc = upload(this, &d.tc, tc)) || (rc = upload(this, &d.tdom, g.tile_dom)) ||
        (rc = upload(this, &d.tntri, g.tile_ntri)) || (rc = upload(this, &d.dom_tiles, dt)) ||
        (rc = upload(this, &d.slot_v, sv)) || (rc = upload(this, &d.slot_P, g.slot_P)) ||
        (rc = upload(this, &d.slot_n, g.slot_n)) || (rc = upload(this, &d.slot_area, g.slot_area)) ||
        (rc = upload(this, &d.slot_curl, g.slot_curl)) || (rc = upload(this, &d.pt_w, g.pt_w)) ||
        (rc = upload(this, &d.vc_ptr, g.vc_ptr)) || (rc = upload(this, &d.vc_idx, g.vc_idx)) ||
        (rc = upload(this, &d.v_dof1, g.v_dof1)) || (rc = upload(this, &d.v_dof2, g.v_dof2)) ||
        (rc = upload(this, &d.np_ptr, g.np_ptr)) || (rc = upload(this, &d.np_src, g.np_src)) ||
        (rc = upload(this, &d.np_code, g.np_code)))
        return rc;
    // pair target list (for the near build)
    std::vector<int32_t> ptgt(g.np_src.size());
    for (int64_t s = 0; s < g.n_slots; s++)
        for (int64_t i = g.np_ptr[s]; i < g.np_ptr[s + 1]; i++) ptgt[i] = (int32_t)s;
    if ((rc = upload(this, &d.np_tgt, ptgt))) return rc;
    for (int r = 0; r <= 3; r++) {  // 0: the near-pair rule, 1-3: Sauter-Schwab
        if ((rc = upload(this, &d.ss_tab[r], quad.ss[r]))) return rc;
        std::vector<float4> f;  // groups of the double-float near build: hi, then lo of each row
        for (size_t i = 0; i < quad.grp[r].size(); i += 8) {
            float h[8], l[8];
            for (int c = 0; c < 8; c++) {
                h[c] = (float)quad.grp[r][i + c];
                l[c] = (float)(quad.grp[r][i + c] - (long double)h[c]);
            }
            for (const float* v : {h, h + 4, l, l + 4}) f.push_back(make_float4(v[0], v[1], v[2], v[3]));
        }
        if ((rc = upload(this, &d.grp[r], f))) return rc;
    }
    {
        std::vector<float2> f;
        for (const long double v : quad.inner) f.push_back(make_float2((float)v, (float)(v - (long double)(float)v)));
        if ((rc = upload(this, &d.inner, f))) return rc;
    }
    // working buffers
    d.pd32 = (float4*)dalloc(g.n_pts * sizeof(float4), &rc); if (rc) return rc;
    d.tcurl32 = (float4*)dalloc(2 * g.n_slots * sizeof(float4), &rc); if (rc) return rc;
    d.pd64 = (double4*)dalloc(g.n_pts * sizeof(double4), &rc); if (rc) return rc;
    d.tcurl64 = (double4*)dalloc(2 * g.n_slots * sizeof(double4), &rc); if (rc) return rc;
    d.tri_out = (double2*)dalloc(g.n_slots * 6 * sizeof(double2), &rc); if (rc) return rc;
    d.kdom = (double2*)dalloc(g.n_dom * sizeof(double2), &rc); if (rc) return rc;
    d.coef = (SlotCoef*)dalloc(g.n_dom * 2 * sizeof(SlotCoef), &rc); if (rc) return rc;
    d.err = (int*)dalloc(sizeof(int), &rc); if (rc) return rc;
    d.xs = (double2*)dalloc(g.n_dof * sizeof(double2), &rc); if (rc) return rc;
    d.ys = (double2*)dalloc(g.n_dof * sizeof(double2), &rc); if (rc) return rc;
    d.ys2 = (double2*)dalloc(g.n_dof * sizeof(double2), &rc); if (rc) return rc;
    CK(cudaMemsetAsync(d.err, 0, sizeof(int), stream));
    ready = true;
    return upload_materials();
}

int bem_ctx::upload_materials() {
    bem_ctx* const ctx = this;
    std::vector<double2> kd(geo.n_dom);
    std::vector<SlotCoef> cf(geo.n_dom * 2);
    for (int i = 0; i < geo.n_dom; i++) {
        kd[i] = make_double2(doms[i].kre, doms[i].kim);
        const double r = doms[i].rho / rho0;
        const double k0r = k0re, k0i = k0im, kr = doms[i].kre, ki = doms[i].kim;
        cf[2 * i] = SlotCoef{1.0, 1.0, 1.0, 1.0, k0r * k0r - k0i * k0i, 2 * k0r * k0i};
        cf[2 * i + 1] = SlotCoef{r, 1.0, 1.0, 1.0 / r, kr * kr - ki * ki, 2 * kr * ki};
    }
    CK(cudaMemcpyAsync(dev.kdom, kd.data(), kd.size() * sizeof(double2), cudaMemcpyHostToDevice, stream));
    CK(cudaMemcpyAsync(dev.coef, cf.data(), cf.size() * sizeof(SlotCoef), cudaMemcpyHostToDevice, stream));
    CK(cudaStreamSynchronize(stream));
    return dfg.ready ? upload_df_wavenumbers() : BEM_OK;
}

// Near-field corrections: n_slot_k = 2 for the PMCHWT system (exterior and
// own-domain wavenumbers), 1 for a single Calderon block at wavenumber k.
int bem_ctx::build_near(NearSet& ns, int n_slot_k, double kre, double kim, const SlotCoef* coef_dev) {
    bem_ctx* const ctx = this;
    const int64_t np = (int64_t)geo.np_src.size();
    int rc;
    ns.n_pairs = np;
    ns.nb64 = (double2*)dalloc(std::max<int64_t>(1, np) * 36 * sizeof(double2), &rc); if (rc) return rc;
    ns.nb32 = (float2*)dalloc(std::max<int64_t>(1, np) * 36 * sizeof(float2), &rc); if (rc) return rc;
    if (np == 0) return BEM_OK;
    const int64_t max_batch = 1 << 20;  // bound the raw scratch
    double2* raw = (double2*)dalloc(std::min(np, max_batch) * n_slot_k * 27 * sizeof(double2), &rc);
    if (rc) return rc;
    for (int64_t b0 = 0; b0 < np; b0 += max_batch) {
        const int64_t nb = std::min(max_batch, np - b0);
        NearArgs a{};
        a.n_pairs = nb;
        a.pair_tgt = dev.np_tgt + b0;
        a.pair_src = dev.np_src + b0;
        a.pair_code = dev.np_code + b0;
        a.slot_P = dev.slot_P;
        a.slot_n = dev.slot_n;
        a.slot_area = dev.slot_area;
        a.slot_curl = dev.slot_curl;
        for (int r = 0; r <= 3; r++) {
            a.ss_tab[r] = dev.ss_tab[r];
            a.ss_n[r] = (int)(quad.ss[r].size() / 5);
        }
        for (int q = 0; q < QP; q++) {
            a.rule[3 * q] = quad.l1[q];
            a.rule[3 * q + 1] = quad.l2[q];
            a.rule[3 * q + 2] = quad.w[q];
        }
        a.k[0] = make_double2(kre, kim);
        a.k[1] = make_double2(0, 0);
        a.kdom = dev.kdom;
        a.slot_dom = (const int*)dev.slot_v;
        a.n_slot_k = n_slot_k;
        a.raw = raw;
        if (opts.fp64_far == 0) {  // double-float point evaluations (the default), else native FP64
            if ((rc = ensure_fardf()) || (rc = check_df_phase(kre, false))) return rc;
            a.use_df = 1;
            for (int r = 0; r <= 3; r++) {
                a.grp[r] = dev.grp[r];
                a.grp_n[r] = (int)(quad.grp[r].size() / 8);
            }
            a.inner = dev.inner;
            a.ng = quad.ng;
            a.sctab = dfg.sctab;
            a.extab = dfg.extab;
            a.c = dfg.c;
            a.kdf = dfg.kdf;
            auto split = [](long double v, float& h, float& l) {
                h = (float)v;
                l = (float)(v - (long double)h);
            };
            split((long double)kre, a.k0df.x, a.k0df.y);
            split((long double)kim, a.k0df.z, a.k0df.w);
            for (int q = 0; q < 3 * QP; q++) split((long double)a.rule[q], a.rule_h[q], a.rule_l[q]);
        }
        CK(launch_near_build(a, stream));
        NearCombineArgs c{};
        c.n_pairs = nb;
        c.pair_tgt = dev.np_tgt + b0;
        c.pair_src = dev.np_src + b0;
        c.slot_n = dev.slot_n;
        c.slot_curl = dev.slot_curl;
        c.slot_v = dev.slot_v;
        c.coef = coef_dev;
        c.n_slot_k = n_slot_k;
        c.raw = raw;
        c.nb64 = ns.nb64 + b0 * 36;
        c.nb32 = ns.nb32 + b0 * 36;
        CK(launch_near_combine(c, stream));
    }
    CK(cudaStreamSynchronize(stream));
    dfree(raw);
    return BEM_OK;
}

int bem_ctx::ensure_near() {
    if (near_ready) return BEM_OK;
    if (pmchwt_near.nb64) { dfree(pmchwt_near.nb64); dfree(pmchwt_near.nb32); pmchwt_near = NearSet(); }
    int rc = build_near(pmchwt_near, 2, k0re, k0im, dev.coef);
    if (rc) return rc;
    near_ready = true;
    return BEM_OK;
}

// Partial potentials of `need` bytes; optional: where that only allows shorter chunks.
int bem_ctx::ensure_partial(size_t need, bool optional) {
    if (need <= partial_bytes) return BEM_OK;
    if (optional && !room_for(need - partial_bytes)) return BEM_ERR_OUT_OF_BUDGET;
    dfree(partial);
    partial_bytes = 0;
    int rc = BEM_OK;
    partial = optional ? try_alloc(need) : dalloc(need, &rc);
    if (!partial) return optional ? BEM_ERR_OUT_OF_BUDGET : rc;
    partial_bytes = need;
    return BEM_OK;
}

// Launch order of the far-field work items: every (target tile, source chunk)
// pair, heaviest first (cost = source triangles, twice for sources in the
// target's own domain, which carry both wavenumbers), so that the light items
// fill the last wave instead of a long one trailing alone.
int bem_ctx::ensure_far_work(int tgt_b, int tgt_e, int src_b, int src_e, int chunk_tiles, int n_chunks, int slot1) {
    const int key[6] = {tgt_b, tgt_e, src_b, src_e, chunk_tiles, slot1};
    if (far_work && std::equal(key, key + 6, far_work_key)) return BEM_OK;
    const Geometry& g = geo;
    const int n_tgt = tgt_e - tgt_b;
    std::vector<std::pair<int64_t, int>> cost((size_t)n_tgt * n_chunks);
    for (int t = 0; t < n_tgt; t++) {
        const int d = g.tile_dom[tgt_b + t];
        const int own_b = g.dom_tile_begin[d], own_e = g.dom_tile_end[d];
        for (int c = 0; c < n_chunks; c++) {
            const int sb = src_b + c * chunk_tiles, se = std::min(sb + chunk_tiles, src_e);
            int64_t w = 0;
            for (int s = sb; s < se; s++) w += (int64_t)g.tile_ntri[s] * (1 + (slot1 && s >= own_b && s < own_e));
            cost[(size_t)t * n_chunks + c] = {-w, t * n_chunks + c};
        }
    }
    std::stable_sort(cost.begin(), cost.end());
    std::vector<int2> work(cost.size());
    for (size_t i = 0; i < cost.size(); i++) work[i] = make_int2(cost[i].second / n_chunks, cost[i].second % n_chunks);
    if (far_work) dfree(far_work);
    far_work = nullptr;
    int rc = upload(this, &far_work, work);
    if (rc) return rc;
    std::copy(key, key + 6, far_work_key);
    return BEM_OK;
}

// FP32 chunks are at most FAR32_CHUNK tiles long: the six warps of a CTA drift
// apart inside its four-stage ring, and in a long chunk the leading warps end
// up waiting for the slowest one at every tile (long-scoreboard stalls, FMA
// pipe 63 % busy at 128 tiles against 74 % at 16).  Measured far-field time on
// the 20,988-triangle rib scene: 31.7-31.9 ms at 6-16 tiles, 33.4 at 24, 36.8
// at 64, 39.1 at the up to 219 tiles taken before; on 41,292 triangles 123 ms
// against 147.5.  The double-float far field has no ring and keeps its own rule.
constexpr int FAR32_CHUNK = 12;

void bem_ctx::chunking(int n_tgt, int n_src, int* n_chunks, int* chunk_tiles, bool fp64) const {
    int want = std::max(1, (152 * 2 * 8 + n_tgt - 1) / std::max(1, n_tgt));
    int nc = std::max(want, (n_src + CHUNK_MAX - 1) / CHUNK_MAX);
    if (!fp64) nc = std::max(nc, (n_src + FAR32_CHUNK - 1) / FAR32_CHUNK);
    if (opts.chunk_tiles > 0) nc = (n_src + opts.chunk_tiles - 1) / opts.chunk_tiles;
    // the partial potentials grow as chunks x points: at most 8 GiB of them at
    // FP64 (4 GiB at FP32), unless CHUNK_MAX forces more chunks
    const int64_t per_chunk = (int64_t)2 * NCOMP * n_tgt * TP * sizeof(double);
    const int nc_mem = (int)std::max<int64_t>(1, ((int64_t)8 << 30) / std::max<int64_t>(1, per_chunk));
    nc = std::min(nc, std::max(nc_mem, (n_src + CHUNK_MAX - 1) / CHUNK_MAX));
    nc = std::max(1, std::min(nc, n_src));
    int ct = (n_src + nc - 1) / nc;
    ct = std::min(ct, CHUNK_MAX);
    *chunk_tiles = ct;
    *n_chunks = (n_src + ct - 1) / ct;
}

// Buffers and launch arguments of one operator application (no launches).
// fill_tiles > 0: the target tiles of all meshes launched together (a group),
// which the chunking spreads over the SMs instead of this mesh's alone.
int bem_ctx::plan_apply(const double2* x, double2* y, int precision, const ApplyMode& m, ApplyPlan& P,
                        int fill_tiles) {
    const Geometry& g = geo;
    const bool fp64 = precision == BEM_PREC_FP64;
    P = ApplyPlan();
    P.fp64 = fp64;
    const int tgt_b = g.dom_tile_begin[m.tgt_dom_lo], tgt_e = g.dom_tile_end[m.tgt_dom_hi - 1];
    const int src_b = g.dom_tile_begin[m.src_dom_lo], src_e = g.dom_tile_end[m.src_dom_hi - 1];
    // FP32: short source chunks where there is room for their partials, else the longer ones
    const int fill = fill_tiles > 0 ? fill_tiles : tgt_e - tgt_b;
    const size_t per_chunk = (size_t)2 * NCOMP * g.n_pts * (fp64 ? sizeof(double) : sizeof(float));
    int n_chunks, chunk_tiles, nc, ct, rc;
    chunking(fill, src_e - src_b, &n_chunks, &chunk_tiles, true);
    partial_need = std::max(partial_need, n_chunks * per_chunk);
    chunking(fill, src_e - src_b, &nc, &ct, fp64);
    if (nc != n_chunks && ensure_partial(nc * per_chunk, true) == BEM_OK) {
        n_chunks = nc;
        chunk_tiles = ct;
    } else if ((rc = ensure_partial(n_chunks * per_chunk, false))) {
        return rc;
    }
    P.n_tgt = tgt_e - tgt_b;
    P.n_chunks = n_chunks;
    // 1. trial densities on the source slots
    GatherArgs& ga = P.ga;
    ga.slot_v = dev.slot_v;
    ga.v_dof1 = dev.v_dof1;
    ga.v_dof2 = dev.v_dof2;
    ga.pt_w = dev.pt_w;
    ga.slot_curl = dev.slot_curl;
    ga.x = x;
    ga.s_begin = (int64_t)src_b * TT;
    ga.s_end = (int64_t)src_e * TT;
    for (int q = 0; q < QP; q++)
        for (int k = 0; k < 3; k++) ga.lam[q][k] = quad.lam[q][k];
    if (fp64) { ga.pd64 = dev.pd64; ga.tcurl64 = dev.tcurl64; }
    else { ga.pd32 = dev.pd32; ga.tcurl32 = dev.tcurl32; }
    // 2. far field
    if (fp64) {
        FarArgs64& fa = P.fa64;
        fa.pg = dev.pg64; fa.tg = dev.tg64; fa.tc = dev.tc; fa.tdom = dev.tdom; fa.tntri = dev.tntri;
        fa.pd = dev.pd64; fa.tcurl = dev.tcurl64; fa.dom_tiles = dev.dom_tiles; fa.kdom = dev.kdom;
        fa.k0 = make_double2(m.kre, m.kim);
        fa.src_begin = src_b; fa.src_end = src_e; fa.tgt_begin = tgt_b; fa.chunk_tiles = chunk_tiles;
        fa.slot1 = m.slot1; fa.n_pts = g.n_pts; fa.partial = (double*)partial;
    } else {
        FarArgs32& fa = P.fa32;
        fa.pg = dev.pg32; fa.pgp = dev.pgp32; fa.tg = dev.tg32; fa.tc = dev.tc; fa.tdom = dev.tdom; fa.tntri = dev.tntri;
        fa.pd = dev.pd32; fa.tcurl = dev.tcurl32; fa.dom_tiles = dev.dom_tiles; fa.kdom = dev.kdom;
        fa.k0 = make_double2(m.kre, m.kim);
        fa.src_begin = src_b; fa.src_end = src_e; fa.tgt_begin = tgt_b; fa.chunk_tiles = chunk_tiles;
        fa.slot1 = m.slot1; fa.n_pts = g.n_pts; fa.partial = (float*)partial; fa.err = dev.err;
        if ((rc = ensure_far_work(tgt_b, tgt_e, src_b, src_e, chunk_tiles, n_chunks, m.slot1))) return rc;
        fa.work = far_work;
    }
    // 3. projection (+ touching-pair correction)
    ProjectArgs& pa = P.pa;
    pa.slot_v = dev.slot_v; pa.pt_w = dev.pt_w; pa.slot_curl = dev.slot_curl; pa.tntri = dev.tntri; pa.tdom = dev.tdom;
    pa.coef = m.coef; pa.tgt_begin = tgt_b; pa.tgt_end = tgt_e; pa.n_chunks = n_chunks; pa.n_pts = g.n_pts;
    if (fp64) pa.partial64 = (const double*)partial; else pa.partial32 = (const float*)partial;
    if (m.near && m.near->n_pairs > 0) {
        pa.np_ptr = dev.np_ptr; pa.np_src = dev.np_src;
        if (fp64) pa.nb64 = m.near->nb64; else pa.nb32 = m.near->nb32;
    }
    pa.v_dof1 = dev.v_dof1; pa.v_dof2 = dev.v_dof2; pa.x = x; pa.tri_out = dev.tri_out;
    for (int q = 0; q < QP; q++)
        for (int k = 0; k < 3; k++) pa.lam[q][k] = quad.lam[q][k];
    // 4. vertex reduction
    ReduceArgs& ra = P.ra;
    ra.vc_ptr = dev.vc_ptr; ra.vc_idx = dev.vc_idx; ra.v_dof1 = dev.v_dof1; ra.v_dof2 = dev.v_dof2;
    ra.tri_out = dev.tri_out; ra.y = y;
    ra.v_begin = g.dom_vert_off[m.tgt_dom_lo];
    ra.v_end = g.dom_vert_off[m.tgt_dom_hi - 1] + g.dom_nv[m.tgt_dom_hi - 1];
    return BEM_OK;
}

// A call whose buffers do not fit beside memory that only speeds calls up gives that back and starts over.
int bem_ctx::run_apply(const double2* x, double2* y, int precision, const ApplyMode& m) {
    return without_optional_if_short([&] { return run_apply_once(x, y, precision, m); });
}

// The pipeline.  x, y: device, system order.  Modes: PMCHWT (all targets,
// all sources at k0 plus own-domain sources at k_j), or BLOCK (targets of
// domain j, sources of domain i, one wavenumber).
int bem_ctx::run_apply_once(const double2* x, double2* y, int precision, const ApplyMode& m) {
    bem_ctx* const ctx = this;
    ApplyPlan P;
    int rc = plan_apply(x, y, precision, m, P);
    if (rc) return rc;
    CK(launch_gather(P.ga, stream));
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    if (profiling) {
        CK(cudaEventCreate(&ev0));
        CK(cudaEventCreate(&ev1));
        CK(cudaEventRecord(ev0, stream));
    }
    if (P.fp64 && opts.fp64_far == 0) {
        const FarArgs64& f = P.fa64;
        if ((rc = far_df(dev.pd64, dev.tcurl64, 1, f.tgt_begin, f.tgt_begin + P.n_tgt, f.src_begin, f.src_end,
                         f.chunk_tiles, P.n_chunks, f.slot1, f.k0.x, f.k0.y, f.partial, 0)))
            return rc;
    } else if (P.fp64) {
        CK(launch_far64(P.fa64, P.n_tgt, P.n_chunks, stream));
    } else {
        CK(launch_far32(P.fa32, P.n_tgt, P.n_chunks, stream));
    }
    if (profiling) {
        CK(cudaEventRecord(ev1, stream));
        far_events.push_back({ev0, ev1});
    }
    CK(launch_project(P.pa, stream));
    CK(launch_reduce(P.ra, stream));
    launches += 4;
    return BEM_OK;
}

// Geometry of the tensor-core far field, on compact tiles of its own (an A
// operand is scaled per pair of tiles, and pairs closer than the sum of their
// radii stay with the FP32 kernel: of 382 tiles on a 12,184-triangle kidney
// scene 19 % of the pairs with runs of a Morton curve, 6.6 % with these): what
// gather, the far-field kernels and the operands read, in those tiles' order,
// the slot of each in the order of the rest, a frame with the mean normal of
// every tile, and the close pairs of tiles.
int bem_ctx::ensure_farmm() {
    bem_ctx* const ctx = this;
    if (mmg.ready) return BEM_OK;
    const Geometry& g = geo;
    const int nt = g.n_tiles;
    CompactTiles ct;
    compact_tiles(g, ct);
    std::vector<float4> gq(g.n_pts), pg(g.n_pts), pgp(g.n_pts), tg(g.n_slots);
    std::vector<double4> tc(nt);
    std::vector<int4> sv(g.n_slots);
    std::vector<double> pw(g.n_pts), curl(9 * g.n_slots);
    for (int64_t s = 0; s < g.n_slots; s++) {
        const int64_t o = ct.perm[s];
        float4 tri[QP];
        for (int q = 0; q < QP; q++) {
            const int64_t p = s * QP + q;
            const float x = (float)ct.pt_delta[3 * p], y = (float)ct.pt_delta[3 * p + 1], z = (float)ct.pt_delta[3 * p + 2];
            pw[p] = g.pt_w[o * QP + q];
            pg[p] = make_float4(x, y, z, (float)pw[p]);
            tri[q] = make_float4(x, y, z, (float)((double)x * x + (double)y * y + (double)z * z));
        }
        pair_interleave(tri, gq.data() + s * QP);
        for (int q = 0; q < QP; q++) tri[q] = pg[s * QP + q];
        pair_interleave(tri, pgp.data() + s * QP);
        tg[s] = make_float4((float)g.slot_n[3 * o], (float)g.slot_n[3 * o + 1], (float)g.slot_n[3 * o + 2], (float)ct.slot_h[s]);
        sv[s] = make_int4(g.slot_v[4 * o], g.slot_v[4 * o + 1], g.slot_v[4 * o + 2], g.slot_v[4 * o + 3]);
        for (int k = 0; k < 9; k++) curl[9 * s + k] = g.slot_curl[9 * o + k];
    }
    for (int t = 0; t < nt; t++) tc[t] = make_double4(ct.tile_c[4 * t], ct.tile_c[4 * t + 1], ct.tile_c[4 * t + 2], ct.tile_c[4 * t + 3]);
    std::vector<float> fr((size_t)nt * 9);
    double rmax = 0;
    for (int t = 0; t < nt; t++) {
        rmax = std::max(rmax, ct.tile_c[4 * t + 3]);
        double m[3] = {0, 0, 0};
        for (int64_t s = (int64_t)t * TT; s < (int64_t)t * TT + g.tile_ntri[t]; s++)
            for (int c = 0; c < 3; c++) m[c] += g.slot_n[3 * ct.perm[s] + c] * g.slot_area[ct.perm[s]];
        double l = std::sqrt(m[0] * m[0] + m[1] * m[1] + m[2] * m[2]);
        if (!(l > 0)) { m[0] = m[1] = 0; m[2] = l = 1; }
        for (double& c : m) c /= l;
        const int ax = std::fabs(m[0]) < std::fabs(m[1]) ? (std::fabs(m[0]) < std::fabs(m[2]) ? 0 : 2)
                                                         : (std::fabs(m[1]) < std::fabs(m[2]) ? 1 : 2);
        double u[3] = {0, 0, 0}, d = m[ax];
        for (int c = 0; c < 3; c++) u[c] = (c == ax) - d * m[c];
        l = std::sqrt(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
        for (double& c : u) c /= l;
        const double v[3] = {m[1] * u[2] - m[2] * u[1], m[2] * u[0] - m[0] * u[2], m[0] * u[1] - m[1] * u[0]};
        for (int c = 0; c < 3; c++) {
            fr[9 * t + c] = (float)u[c];
            fr[9 * t + 3 + c] = (float)v[c];
            fr[9 * t + 6 + c] = (float)m[c];
        }
    }
    int e = 0;
    std::frexp(rmax, &e);
    mmg.rho = std::ldexp(1.0f, std::max(-100, std::min(100, e)));
    mmg.near_words = (nt + 31) / 32;
    std::vector<uint32_t> mask((size_t)nt * mmg.near_words, 0);
    mmg.h_ptr.assign(nt + 1, 0);
    mmg.h_idx.clear();
    mmg.fits = true;
    for (int t = 0; t < nt; t++) {
        const double* a = &ct.tile_c[4 * t];
        for (int s = 0; s < nt; s++) {
            const double* b = &ct.tile_c[4 * s];
            const double x = a[0] - b[0], y = a[1] - b[1], z = a[2] - b[2], r = FARMM_SEP * (a[3] + b[3]);
            if (x * x + y * y + z * z < r * r || s == t) {
                mask[(size_t)t * mmg.near_words + s / 32] |= 1u << (s % 32);
                mmg.h_idx.push_back(s);
            }
        }
        mmg.h_ptr[t + 1] = (int)mmg.h_idx.size();
        mmg.fits &= mmg.h_ptr[t + 1] - mmg.h_ptr[t] <= CHUNK_MAX;
    }
    if (!mmg.fits) {  // never used
        mmg.ready = true;
        return BEM_OK;
    }
    // one buffer, pieces at 256 bytes
    size_t total = 0;
    for (int pass = 0; pass < 2; pass++) {
        size_t at = 0;
        cudaError_t e = cudaSuccess;
        auto put = [&](auto** p, const auto& v) {
            const size_t n = v.size() * sizeof(v[0]);
            if (pass) {
                *p = (std::remove_reference_t<decltype(**p)>*)((char*)mmg.buf + at);
                if (n && e == cudaSuccess) e = cudaMemcpyAsync(*p, v.data(), n, cudaMemcpyHostToDevice, stream);
            }
            at += (n + 255) / 256 * 256;
        };
        put(&mmg.geo, gq); put(&mmg.pg, pg); put(&mmg.pgp, pgp); put(&mmg.tg, tg); put(&mmg.tc, tc); put(&mmg.slot_v, sv);
        put(&mmg.pt_w, pw); put(&mmg.slot_curl, curl); put(&mmg.perm, ct.perm); put(&mmg.near, mask); put(&mmg.frame, fr);
        put(&mmg.near_ptr, mmg.h_ptr); put(&mmg.near_idx, mmg.h_idx);
        CK(e);
        if (!pass) {
            total = at;
            mmg.buf = try_alloc(total);
            if (!mmg.buf) return BEM_ERR_OUT_OF_BUDGET;
            mmg.bytes = total;
        }
    }
    CK(cudaStreamSynchronize(stream));
    mmg.ready = true;
    return BEM_OK;
}

// Bytes of mmg.buf, at most.
static size_t farmm_geometry_bytes(const Geometry& g) {
    const size_t nt = g.n_tiles;
    return (size_t)g.n_pts * 56 + (size_t)g.n_slots * 108 +
           nt * (32 + 36 + 4 + 4 * ((nt + 31) / 32) + 4 * std::min<size_t>(nt, CHUNK_MAX)) + 14 * 256;
}

// Whether n_rhs vectors go to the tensor cores, with the memory for it in
// place (`multi`: that of their densities and partials): enough tiles for most
// pairs not to be close, and room.  Nothing is built or allocated where there is none.
bool bem_ctx::reserve_farmm(int64_t n_rhs, size_t multi) {
    if (geo.n_tiles < FARMM_MIN_TILES || (mmg.ready && !mmg.fits)) return false;
    const size_t need = farmm_bytes(geo.n_tiles, n_rhs);
    const size_t grow = (mmg.ready ? 0 : farmm_geometry_bytes(geo)) + (need > mm_bytes ? need - mm_bytes : 0) +
                        (multi > multi_buf_bytes ? multi - multi_buf_bytes : 0);
    if (!room_for(grow) || ensure_farmm() || !mmg.fits) return false;
    if (need > mm_bytes) {
        dfree(mm_buf);
        mm_buf = try_alloc(need);
        mm_bytes = mm_buf ? need : 0;
    }
    if (mm_buf && multi > multi_buf_bytes) {
        dfree(multi_buf);
        multi_buf = try_alloc(multi);
        multi_buf_bytes = multi_buf ? multi : 0;
    }
    return mm_buf && multi <= multi_buf_bytes;
}

// A_hat applied to n_rhs vectors x [n_rhs][N] -> y [n_rhs][N] at FP32 with
// the far field of all of them at once, then the projection (with the
// near-field correction) and the reduction of each vector.  Meshes of at least
// FARMM_MIN_TILES tiles take the tensor cores for the pairs of tiles that are
// not close (k_farmm.cu) and far32m_kernel for the close ones, whose partials
// are one chunk more; smaller ones, and budgets that do not hold the operands,
// far32m_kernel for all (the Green's function and gradient factor of a pair
// are evaluated once per group of MRG vectors).
int bem_ctx::apply_ahat_multi(const double2* x, double2* y, int64_t n_rhs) {
    int rc = ensure_near();
    if (rc) return rc;
    return without_optional_if_short([&] { return apply_ahat_multi_once(x, y, n_rhs); });
}

int bem_ctx::apply_ahat_multi_once(const double2* x, double2* y, int64_t n_rhs) {
    bem_ctx* const ctx = this;
    int rc;
    const Geometry& g = geo;
    const int n_tiles = g.n_tiles;
    const int groups = (int)((n_rhs + MRG - 1) / MRG);
    int n_chunks, chunk_tiles, nc, ct;  // partial rows; source tiles per item
    const size_t b_pd = (size_t)n_rhs * g.n_pts * sizeof(float4);
    const size_t b_tc = (size_t)n_rhs * 2 * g.n_slots * sizeof(float4);
    const size_t b_row = (size_t)n_rhs * 2 * NCOMP * g.n_pts * sizeof(float);
    multi_chunking(n_tiles, g.n_pts, n_rhs, &n_chunks, &chunk_tiles);
    const size_t need = b_pd + b_tc + n_chunks * b_row;
    multi_need = std::max(multi_need, need);
    farmm_chunking(n_tiles, g.n_pts, n_rhs, &nc, &ct);
    const bool mm = reserve_farmm(n_rhs, b_pd + b_tc + (nc + 1) * b_row);
    if (mm) {
        n_chunks = nc + 1;  // one more: the close tiles
        chunk_tiles = ct;
    } else if (need > multi_buf_bytes) {
        dfree(multi_buf);
        multi_buf_bytes = 0;
        multi_buf = dalloc(need, &rc);
        if (rc) return rc;
        multi_buf_bytes = need;
    }
    const int64_t rstride = (int64_t)n_chunks * 2 * NCOMP * g.n_pts;
    float4* pdm = (float4*)multi_buf;
    float4* tcm = (float4*)((char*)multi_buf + b_pd);
    float* part = (float*)((char*)multi_buf + b_pd + b_tc);
    // work list: tensor-core items (block, chunk, slot, group), groups and chunks outermost so that the CTAs of a
    // wave share a chunk's operands through L2, then items of the FP32 kernel (target tile, chunk, slot, group),
    // heaviest first
    const int key[4] = {n_chunks, chunk_tiles, groups, (int)mm};
    if (!multi_work || !std::equal(key, key + 4, multi_key)) {
        std::vector<int4> work;
        if (mm)
            for (int gr = 0; gr < farmm_groups(n_rhs); gr++)
                for (int c = 0; c + 1 < n_chunks; c++)
                    for (int sl = 0; sl < 2; sl++)
                        for (int b = 0; b < farmm_blocks(g.n_pts); b++) work.push_back(make_int4(b, c, sl, gr));
        const int64_t n_far = (int64_t)work.size();
        std::vector<std::pair<int64_t, int4>> items;
        for (int t = 0; t < n_tiles; t++) {
            const int d = g.tile_dom[t];
            const int own_b = g.dom_tile_begin[d], own_e = g.dom_tile_end[d];
            for (int c = mm ? n_chunks - 1 : 0; c < n_chunks; c++) {
                const int sb = mm ? mmg.h_ptr[t] : c * chunk_tiles, se = mm ? mmg.h_ptr[t + 1] : std::min(sb + chunk_tiles, n_tiles);
                int64_t w0 = 0, w1 = 0;
                for (int i = sb; i < se; i++) {
                    const int s = mm ? mmg.h_idx[i] : i;
                    w0 += g.tile_ntri[s];
                    if (s >= own_b && s < own_e) w1 += g.tile_ntri[s];
                }
                for (int gr = 0; gr < groups; gr++) {
                    items.push_back({-w0, make_int4(t, c, 0, gr)});
                    items.push_back({-w1, make_int4(t, c, 1, gr)});  // empty ranges write zeros
                }
            }
        }
        std::stable_sort(items.begin(), items.end(),
                         [](const std::pair<int64_t, int4>& a, const std::pair<int64_t, int4>& b) { return a.first < b.first; });
        for (const auto& it : items) work.push_back(it.second);
        dfree(multi_work);
        multi_work = nullptr;
        for (int& k : multi_key) k = -1;
        multi_work = (int4*)dalloc(work.size() * sizeof(int4), &rc);
        if (rc) return rc;
        CK(cudaMemcpyAsync(multi_work, work.data(), work.size() * sizeof(int4), cudaMemcpyHostToDevice, stream));
        CK(cudaStreamSynchronize(stream));
        multi_n_work = (int64_t)work.size();
        multi_n_far = n_far;
        std::copy(key, key + 4, multi_key);
    }
    const int64_t N = g.n_dof;
    // 1. trial densities of every vector
    for (int64_t r = 0; r < n_rhs; r++) {
        GatherArgs ga{};
        ga.slot_v = mm ? mmg.slot_v : dev.slot_v; ga.v_dof1 = dev.v_dof1; ga.v_dof2 = dev.v_dof2;
        ga.pt_w = mm ? mmg.pt_w : dev.pt_w; ga.slot_curl = mm ? mmg.slot_curl : dev.slot_curl;
        ga.x = x + r * N; ga.s_begin = 0; ga.s_end = g.n_slots;
        for (int q = 0; q < QP; q++)
            for (int k = 0; k < 3; k++) ga.lam[q][k] = quad.lam[q][k];
        ga.pd32 = pdm + r * g.n_pts;
        ga.tcurl32 = tcm + r * 2 * g.n_slots;
        CK(launch_gather(ga, stream));
    }
    // 2. far field of all vectors
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    if (profiling) {
        CK(cudaEventCreate(&ev0));
        CK(cudaEventCreate(&ev1));
        CK(cudaEventRecord(ev0, stream));
    }
    if (mm) {
        FarMmPlan p{};
        p.pg = mmg.pg; p.tg = mmg.tg; p.tc = mmg.tc; p.tdom = dev.tdom; p.dom_tiles = dev.dom_tiles; p.kdom = dev.kdom;
        p.perm = mmg.perm;
        p.k0 = make_double2(k0re, k0im);
        p.pd = pdm; p.tcurl = tcm; p.frame = mmg.frame; p.near = mmg.near; p.near_words = mmg.near_words; p.geo = mmg.geo;
        p.rho = mmg.rho; p.n_tiles = n_tiles; p.chunk_tiles = chunk_tiles; p.R = (int)n_rhs; p.n_pts = g.n_pts;
        p.n_slots = g.n_slots; p.rstride = rstride; p.n_work = multi_n_far; p.partial = part; p.err = dev.err;
        p.work = multi_work; p.buf = mm_buf;
        CK(launch_farmm(p, stream));
        launches += 3;
    }
    FarArgs32M fa{};
    fa.pg = dev.pg32; fa.pgp = dev.pgp32; fa.tg = dev.tg32; fa.tc = dev.tc; fa.tdom = dev.tdom; fa.tntri = dev.tntri;
    fa.pd = pdm; fa.tcurl = tcm; fa.dom_tiles = dev.dom_tiles; fa.kdom = dev.kdom;
    fa.k0 = make_double2(k0re, k0im);
    fa.src_begin = 0; fa.src_end = n_tiles; fa.tgt_begin = 0; fa.chunk_tiles = chunk_tiles;
    fa.R = (int)n_rhs; fa.n_pts = g.n_pts; fa.n_slots = g.n_slots; fa.rstride = rstride; fa.partial = part;
    fa.err = dev.err; fa.work = multi_work + (mm ? multi_n_far : 0);
    if (mm) {
        fa.pg = mmg.pg; fa.pgp = mmg.pgp; fa.tg = mmg.tg; fa.tc = mmg.tc; fa.perm = mmg.perm;
        fa.near_ptr = mmg.near_ptr;
        fa.near_idx = mmg.near_idx;
    }
    CK(launch_far32_multi(fa, multi_n_work - (mm ? multi_n_far : 0), stream));
    if (profiling) {
        CK(cudaEventRecord(ev1, stream));
        far_events.push_back({ev0, ev1});
    }
    // 3. projection and reduction of each vector
    for (int64_t r = 0; r < n_rhs; r++) {
        ProjectArgs pa{};
        pa.slot_v = dev.slot_v; pa.pt_w = dev.pt_w; pa.slot_curl = dev.slot_curl; pa.tntri = dev.tntri; pa.tdom = dev.tdom;
        pa.coef = dev.coef; pa.tgt_begin = 0; pa.tgt_end = n_tiles; pa.n_chunks = n_chunks; pa.n_pts = g.n_pts;
        pa.partial32 = part + r * rstride;
        if (pmchwt_near.n_pairs > 0) { pa.np_ptr = dev.np_ptr; pa.np_src = dev.np_src; pa.nb32 = pmchwt_near.nb32; }
        pa.v_dof1 = dev.v_dof1; pa.v_dof2 = dev.v_dof2; pa.x = x + r * N; pa.tri_out = dev.tri_out;
        for (int q = 0; q < QP; q++)
            for (int k = 0; k < 3; k++) pa.lam[q][k] = quad.lam[q][k];
        CK(launch_project(pa, stream));
        ReduceArgs ra{};
        ra.vc_ptr = dev.vc_ptr; ra.vc_idx = dev.vc_idx; ra.v_dof1 = dev.v_dof1; ra.v_dof2 = dev.v_dof2;
        ra.tri_out = dev.tri_out; ra.y = y + r * N; ra.v_begin = 0; ra.v_end = g.n_vert;
        CK(launch_reduce(ra, stream));
    }
    launches += 3 * n_rhs + 1;
    return BEM_OK;
}

// A_hat applied to n_rhs vectors at FP64 with one far-field launch for all of
// them (the kernel values of a pair evaluated once per group: two vectors in
// fardf_kernel, RG64 in far64m_kernel where native FP64 is asked for), then the
// projection (with the FP64 near-field correction) and the reduction of each
// vector.
int bem_ctx::apply_ahat64_multi(const double2* x, double2* y, int64_t n_rhs) {
    bem_ctx* const ctx = this;
    int rc = ensure_near();
    if (rc) return rc;
    const Geometry& g = geo;
    const int n_tiles = g.n_tiles;
    int n_chunks, chunk_tiles;
    multi64_chunking(n_tiles, n_rhs, &n_chunks, &chunk_tiles);
    const int64_t rstride = (int64_t)n_chunks * 2 * NCOMP * g.n_pts;
    const size_t b_pd = (size_t)n_rhs * g.n_pts * sizeof(double4);
    const size_t b_tc = (size_t)n_rhs * 2 * g.n_slots * sizeof(double4);
    const size_t need = b_pd + b_tc + (size_t)n_rhs * rstride * sizeof(double);
    if (need > multi64_buf_bytes) {
        dfree(multi64_buf);
        multi64_buf = dalloc(need, &rc);
        if (rc) { multi64_buf = nullptr; multi64_buf_bytes = 0; return rc; }
        multi64_buf_bytes = need;
    }
    double4* pdm = (double4*)multi64_buf;
    double4* tcm = (double4*)((char*)multi64_buf + b_pd);
    double* part = (double*)((char*)multi64_buf + b_pd + b_tc);
    const int64_t N = g.n_dof;
    for (int64_t r = 0; r < n_rhs; r++) {
        GatherArgs ga{};
        ga.slot_v = dev.slot_v; ga.v_dof1 = dev.v_dof1; ga.v_dof2 = dev.v_dof2; ga.pt_w = dev.pt_w;
        ga.slot_curl = dev.slot_curl; ga.x = x + r * N; ga.s_begin = 0; ga.s_end = g.n_slots;
        for (int q = 0; q < QP; q++)
            for (int k = 0; k < 3; k++) ga.lam[q][k] = quad.lam[q][k];
        ga.pd64 = pdm + r * g.n_pts;
        ga.tcurl64 = tcm + r * 2 * g.n_slots;
        CK(launch_gather(ga, stream));
    }
    FarArgs64M fa{};
    fa.pg = dev.pg64; fa.tg = dev.tg64; fa.tc = dev.tc; fa.tdom = dev.tdom; fa.tntri = dev.tntri;
    fa.pd = pdm; fa.tcurl = tcm; fa.dom_tiles = dev.dom_tiles; fa.kdom = dev.kdom;
    fa.k0 = make_double2(k0re, k0im);
    fa.src_begin = 0; fa.src_end = n_tiles; fa.tgt_begin = 0; fa.chunk_tiles = chunk_tiles; fa.slot1 = 1;
    fa.groups = (int)((n_rhs + RG64 - 1) / RG64); fa.R = (int)n_rhs;
    fa.n_pts = g.n_pts; fa.n_slots = g.n_slots; fa.rstride = rstride; fa.partial = part;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    if (profiling) {
        CK(cudaEventCreate(&ev0));
        CK(cudaEventCreate(&ev1));
        CK(cudaEventRecord(ev0, stream));
    }
    if (opts.fp64_far == 0) {
        if ((rc = far_df(pdm, tcm, n_rhs, 0, n_tiles, 0, n_tiles, chunk_tiles, n_chunks, 1, k0re, k0im, part, rstride)))
            return rc;
    } else {
        CK(launch_far64_multi(fa, n_tiles, n_chunks, stream));
    }
    if (profiling) {
        CK(cudaEventRecord(ev1, stream));
        far_events.push_back({ev0, ev1});
    }
    for (int64_t r = 0; r < n_rhs; r++) {
        ProjectArgs pa{};
        pa.slot_v = dev.slot_v; pa.pt_w = dev.pt_w; pa.slot_curl = dev.slot_curl; pa.tntri = dev.tntri; pa.tdom = dev.tdom;
        pa.coef = dev.coef; pa.tgt_begin = 0; pa.tgt_end = n_tiles; pa.n_chunks = n_chunks; pa.n_pts = g.n_pts;
        pa.partial64 = part + r * rstride;
        if (pmchwt_near.n_pairs > 0) { pa.np_ptr = dev.np_ptr; pa.np_src = dev.np_src; pa.nb64 = pmchwt_near.nb64; }
        pa.v_dof1 = dev.v_dof1; pa.v_dof2 = dev.v_dof2; pa.x = x + r * N; pa.tri_out = dev.tri_out;
        for (int q = 0; q < QP; q++)
            for (int k = 0; k < 3; k++) pa.lam[q][k] = quad.lam[q][k];
        CK(launch_project(pa, stream));
        ReduceArgs ra{};
        ra.vc_ptr = dev.vc_ptr; ra.vc_idx = dev.vc_idx; ra.v_dof1 = dev.v_dof1; ra.v_dof2 = dev.v_dof2;
        ra.tri_out = dev.tri_out; ra.y = y + r * N; ra.v_begin = 0; ra.v_end = g.n_vert;
        CK(launch_reduce(ra, stream));
    }
    launches += 3 * n_rhs + 1;
    return BEM_OK;
}

int bem_ctx::apply_ahat(const double2* x, double2* y, int precision) {
    int rc = ensure_near();
    if (rc) return rc;
    ApplyMode m;
    m.tgt_dom_lo = 0; m.tgt_dom_hi = geo.n_dom; m.src_dom_lo = 0; m.src_dom_hi = geo.n_dom;
    m.kre = k0re; m.kim = k0im; m.slot1 = 1; m.coef = dev.coef; m.near = &pmchwt_near;
    return run_apply(x, y, precision, m);
}

int bem_ctx::check_device_error() {
    bem_ctx* const ctx = this;
    int h = 0;
    CK(cudaMemcpyAsync(&h, dev.err, sizeof(int), cudaMemcpyDeviceToHost, stream));
    CK(cudaStreamSynchronize(stream));
    if (h) {
        CK(cudaMemsetAsync(dev.err, 0, sizeof(int), stream));
        if (h & 4) return fail(BEM_ERR_INVALID_ARG, "a device-side input index was out of range (checked by a kernel)");
        return fail(BEM_ERR_TIMEOUT, "a device-side wait timed out (error flag set by a kernel)");
    }
    return BEM_OK;
}

// ------------------------------------------------------------------ C ABI

extern "C" {

int bem_default_opts(bem_opts* o) {
    if (!o) return BEM_ERR_INVALID_ARG;
    std::memset(o, 0, sizeof *o);
    o->n_gauss_singular = 6;
    o->chunk_tiles = 0;
    o->hbm_budget_bytes = 0;
    o->n_pade = 4;
    o->pade_theta = M_PI / 3.0;
    o->r_eps = 0.0;
    o->eps_exponent = 1.0 / 3.0;
    o->osrc_tol = 1e-11;
    o->osrc_solver = 0;
    o->osrc_wavenumber = 0;
    o->fp64_far = 0;
    return BEM_OK;
}

int bem_create(bem_ctx** out, int device, void* cuda_stream, const bem_opts* opts) {
    if (!out) return BEM_ERR_INVALID_ARG;
    *out = nullptr;
    int n = 0;
    if (cudaGetDeviceCount(&n) != cudaSuccess || device < 0 || device >= n) return BEM_ERR_CUDA;
    if (cudaSetDevice(device) != cudaSuccess) return BEM_ERR_CUDA;
    bem_ctx* c = new (std::nothrow) bem_ctx();
    if (!c) return BEM_ERR_OUT_OF_BUDGET;
    c->device = device;
    c->stream = (cudaStream_t)cuda_stream;
    bem_default_opts(&c->opts);
    if (opts) c->opts = *opts;
    if (c->opts.n_gauss_singular < 2 || c->opts.n_gauss_singular > NEAR_NG_MAX || !(c->opts.osrc_tol > 0) ||
        !(c->opts.osrc_tol < 1) || c->opts.osrc_solver < 0 || c->opts.osrc_solver > 4 ||
        c->opts.osrc_wavenumber < 0 || c->opts.osrc_wavenumber > 1 || c->opts.fp64_far < 0 || c->opts.fp64_far > 1) {
        delete c;
        return BEM_ERR_INVALID_ARG;
    }
    c->osrc_tol = c->opts.osrc_tol;
    *out = c;
    return BEM_OK;
}

int bem_destroy(bem_ctx* ctx) {
    if (!ctx) return BEM_OK;
    release_device(ctx);
    release_group(ctx);
    if (ctx->own_stream) cudaStreamDestroy(ctx->stream);
    delete ctx;
    return BEM_OK;
}

int bem_set_exterior(bem_ctx* ctx, bem_z k0, double rho0) {
    if (!ctx) return BEM_ERR_INVALID_ARG;
    if (!(rho0 > 0) || !(k0.im >= 0) || !std::isfinite(k0.re)) return ctx->fail(BEM_ERR_INVALID_ARG, "bad exterior medium");
    ctx->k0re = k0.re;
    ctx->k0im = k0.im;
    ctx->rho0 = rho0;
    invalidate_basis(ctx);
    invalidate_recycle(ctx);
    if (ctx->ready) {
        ctx->near_ready = false;
        ctx->osrc_ready = false;
        ctx->rhs_ready = false;
        ctx->asm_ready = false;
        ctx->asm64_ready = false;
        return ctx->upload_materials();
    }
    return BEM_OK;
}

int bem_add_domain(bem_ctx* ctx, const double* verts, int64_t nv, const int32_t* tris, int64_t nt, bem_z k,
                   double rho, int32_t* domain_id) {
    if (!ctx) return BEM_ERR_INVALID_ARG;
    if (!verts || !tris || nv < 3 || nt < 4) return ctx->fail(BEM_ERR_INVALID_ARG, "empty or null mesh");
    if (!(rho > 0) || !(k.im >= 0)) return ctx->fail(BEM_ERR_INVALID_ARG, "bad material");
    HostDomain d;
    d.verts.assign(verts, verts + 3 * nv);
    d.tris.assign(tris, tris + 3 * nt);
    d.nv = nv;
    d.nt = nt;
    d.kre = k.re;
    d.kim = k.im;
    d.rho = rho;
    std::vector<HostDomain> trial = ctx->doms;
    trial.push_back(d);
    // validate now (cheap host pass) so that errors surface at the call
    Quadrature q;
    if (!build_quadrature(q, 2)) return ctx->fail(BEM_ERR_STATE, "quadrature");
    Geometry g;
    std::vector<HostDomain> one{d};
    std::string msg = build_geometry(one, q, g);
    if (!msg.empty()) return ctx->fail(BEM_ERR_MESH_INVALID, msg);
    if (ctx->ready) release_device(ctx);
    ctx->doms.push_back(d);
    if (domain_id) *domain_id = (int32_t)ctx->doms.size() - 1;
    return BEM_OK;
}

int bem_set_material(bem_ctx* ctx, int32_t id, bem_z k, double rho) {
    if (!ctx) return BEM_ERR_INVALID_ARG;
    if (id < 0 || id >= (int32_t)ctx->doms.size()) return ctx->fail(BEM_ERR_INVALID_ARG, "bad domain id");
    if (!(rho > 0) || !(k.im >= 0)) return ctx->fail(BEM_ERR_INVALID_ARG, "bad material");
    ctx->doms[id].kre = k.re;
    ctx->doms[id].kim = k.im;
    ctx->doms[id].rho = rho;
    invalidate_basis(ctx);
    invalidate_recycle(ctx);
    if (ctx->ready) {
        ctx->near_ready = false;
        ctx->osrc_ready = false;
        ctx->asm_ready = false;
        ctx->asm64_ready = false;
        return ctx->upload_materials();
    }
    return BEM_OK;
}

int bem_num_dofs(const bem_ctx* ctx, int64_t* n) {
    if (!ctx || !n) return BEM_ERR_INVALID_ARG;
    int64_t s = 0;
    for (auto& d : ctx->doms) s += 2 * d.nv;
    *n = s;
    return BEM_OK;
}

int bem_interaction_count(const bem_ctx* ctx, int64_t* n) {
    if (!ctx || !n) return BEM_ERR_INVALID_ARG;
    // regular-rule point pairs: all (target, source) points at k0, own-domain pairs at k_j
    int64_t P = 0, own = 0;
    for (auto& d : ctx->doms) {
        P += d.nt * QP;
        own += (d.nt * QP) * (d.nt * QP);
    }
    *n = P * P + own;
    return BEM_OK;
}

static int io_in(bem_ctx* ctx, const bem_z* x, int64_t n, int on_device, const double2** out) {
    if (on_device) {
        *out = (const double2*)x;
        return BEM_OK;
    }
    CK(cudaMemcpyAsync(ctx->dev.xs, x, n * sizeof(double2), cudaMemcpyHostToDevice, ctx->stream));
    *out = ctx->dev.xs;
    return BEM_OK;
}

int bem_apply(bem_ctx* ctx, int op, const bem_z* x, bem_z* y, int64_t n_rhs, int precision, int on_device) {
    if (!ctx) return BEM_ERR_INVALID_ARG;
    if (!x || !y || n_rhs < 1) return ctx->fail(BEM_ERR_INVALID_ARG, "null vector or n_rhs < 1");
    if (precision < BEM_PREC_FP64 || precision > BEM_PREC_FP64_ASSEMBLED)
        return ctx->fail(BEM_ERR_INVALID_ARG, "bad precision");
    if (op < BEM_OP_AHAT || op > BEM_OP_PREC_AHAT) return ctx->fail(BEM_ERR_INVALID_ARG, "bad op");
    CK(cudaSetDevice(ctx->device));
    int rc = ctx->finalize();
    if (rc) return rc;
    const int64_t N = ctx->geo.n_dof;
    const bool multi = (precision == BEM_PREC_FP32 || precision == BEM_PREC_FP64) && n_rhs > 1;
    if ((precision == BEM_PREC_BF16X3 || precision == BEM_PREC_FP64_ASSEMBLED || multi) && op != BEM_OP_PREC) {
        // all right-hand sides at once: one product on the assembled operator, or
        // one matrix-free far-field launch for all of them
        const double2* xd = (const double2*)x;
        double2* yd = (double2*)y;
        double2* stage = nullptr;
        if (!on_device) {
            stage = (double2*)ctx->dalloc((size_t)2 * n_rhs * N * sizeof(double2), &rc);
            if (rc) return rc;
            CK(cudaMemcpyAsync(stage, x, n_rhs * N * sizeof(double2), cudaMemcpyHostToDevice, ctx->stream));
            xd = stage;
            yd = stage + n_rhs * N;
        }
        double2* tmp = nullptr;
        if (op == BEM_OP_PREC_AHAT) {
            tmp = (double2*)ctx->dalloc((size_t)n_rhs * N * sizeof(double2), &rc);
            if (rc) return rc;
        }
        double2* dst = tmp ? tmp : yd;
        rc = precision == BEM_PREC_BF16X3         ? ctx->apply_assembled(xd, dst, n_rhs)
             : precision == BEM_PREC_FP64_ASSEMBLED ? ctx->apply_assembled64(xd, dst, n_rhs)
             : precision == BEM_PREC_FP64           ? ctx->apply_ahat64_multi(xd, dst, n_rhs)
                                                    : ctx->apply_ahat_multi(xd, dst, n_rhs);
        if (!rc && tmp) rc = ctx->apply_prec_batch(tmp, yd, n_rhs);
        if (tmp) {
            cudaStreamSynchronize(ctx->stream);
            ctx->dfree(tmp);
        }
        if (!rc && !on_device) {
            CK(cudaMemcpyAsync(y, yd, n_rhs * N * sizeof(double2), cudaMemcpyDeviceToHost, ctx->stream));
            CK(cudaStreamSynchronize(ctx->stream));
        }
        if (stage) {
            cudaStreamSynchronize(ctx->stream);
            ctx->dfree(stage);
        }
        if (rc) return rc;
        return on_device ? BEM_OK : ctx->check_device_error();
    }
    if (op == BEM_OP_PREC && n_rhs > 1) {
        // every right-hand side in one batched preconditioner application
        const double2* xd = (const double2*)x;
        double2* yd = (double2*)y;
        double2* stage = nullptr;
        if (!on_device) {
            stage = (double2*)ctx->dalloc((size_t)2 * n_rhs * N * sizeof(double2), &rc);
            if (rc) return rc;
            CK(cudaMemcpyAsync(stage, x, n_rhs * N * sizeof(double2), cudaMemcpyHostToDevice, ctx->stream));
            xd = stage;
            yd = stage + n_rhs * N;
        }
        rc = ctx->apply_prec_batch(xd, yd, n_rhs);
        if (!rc && !on_device) {
            CK(cudaMemcpyAsync(y, yd, n_rhs * N * sizeof(double2), cudaMemcpyDeviceToHost, ctx->stream));
            CK(cudaStreamSynchronize(ctx->stream));
        }
        if (stage) {
            cudaStreamSynchronize(ctx->stream);
            ctx->dfree(stage);
        }
        if (rc) return rc;
        return on_device ? BEM_OK : ctx->check_device_error();
    }
    for (int64_t r = 0; r < n_rhs; r++) {
        const double2* xd;
        if ((rc = io_in(ctx, x + r * N, N, on_device, &xd))) return rc;
        double2* yd = on_device ? (double2*)(y + r * N) : ctx->dev.ys;
        if (op == BEM_OP_AHAT) rc = ctx->apply_ahat(xd, yd, precision);
        else if (op == BEM_OP_PREC) rc = ctx->apply_prec(xd, yd);
        else rc = ctx->apply_prec_ahat(xd, yd, precision);
        if (rc) return rc;
        if (!on_device) {
            CK(cudaMemcpyAsync(y + r * N, yd, N * sizeof(double2), cudaMemcpyDeviceToHost, ctx->stream));
            CK(cudaStreamSynchronize(ctx->stream));
            if ((rc = ctx->check_device_error())) return rc;
        }
    }
    return BEM_OK;
}

int bem_apply_block(bem_ctx* ctx, int32_t j, int32_t i, bem_z k, const bem_z* x, bem_z* y, int precision,
                    int on_device) {
    if (!ctx) return BEM_ERR_INVALID_ARG;
    const int nd = (int)ctx->doms.size();
    if (j < 0 || j >= nd || i < 0 || i >= nd || !x || !y) return ctx->fail(BEM_ERR_INVALID_ARG, "bad block arguments");
    if (precision != BEM_PREC_FP64 && precision != BEM_PREC_FP32) return ctx->fail(BEM_ERR_INVALID_ARG, "bad precision");
    CK(cudaSetDevice(ctx->device));
    int rc = ctx->finalize();
    if (rc) return rc;
    const Geometry& g = ctx->geo;
    // coefficients: plain Calderon block at k on every domain
    BlockCache* bc = nullptr;
    for (auto& b : ctx->block_cache)
        if (b.dom == i && b.kre == k.re && b.kim == k.im) bc = &b;
    if (!bc) {
        ctx->block_cache.push_back(BlockCache());
        bc = &ctx->block_cache.back();
        bc->dom = i;
        bc->kre = k.re;
        bc->kim = k.im;
        std::vector<SlotCoef> cf(g.n_dom * 2);
        for (int d = 0; d < g.n_dom; d++) {
            cf[2 * d] = SlotCoef{1, 1, 1, 1, k.re * k.re - k.im * k.im, 2 * k.re * k.im};
            cf[2 * d + 1] = SlotCoef{0, 0, 0, 0, 0, 0};
        }
        bc->coef = (SlotCoef*)ctx->dalloc(cf.size() * sizeof(SlotCoef), &rc);
        if (rc) return rc;
        CK(cudaMemcpyAsync(bc->coef, cf.data(), cf.size() * sizeof(SlotCoef), cudaMemcpyHostToDevice, ctx->stream));
        if ((rc = ctx->build_near(bc->near, 1, k.re, k.im, bc->coef))) return rc;
    }
    // scatter x (paper order [phi_i; psi_i]) into a zero system-order vector
    const int64_t nvi = g.dom_nv[i], nvj = g.dom_nv[j], N = g.n_dof;
    CK(cudaMemsetAsync(ctx->dev.xs, 0, N * sizeof(double2), ctx->stream));
    const cudaMemcpyKind kin = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    const int64_t off_i = g.dom_dof_off[i], off_j = g.dom_dof_off[j];
    CK(cudaMemcpyAsync(ctx->dev.xs + off_i + nvi, x, nvi * sizeof(double2), kin, ctx->stream));       // phi
    CK(cudaMemcpyAsync(ctx->dev.xs + off_i, x + nvi, nvi * sizeof(double2), kin, ctx->stream));       // psi
    ApplyMode m;
    m.tgt_dom_lo = j; m.tgt_dom_hi = j + 1; m.src_dom_lo = i; m.src_dom_hi = i + 1;
    m.kre = k.re; m.kim = k.im; m.slot1 = 0; m.coef = bc->coef;
    // touching pairs within domain i and near pairs from domain j to domain i
    // (the other pairs of the set meet zeros of x outside domain i)
    m.near = &bc->near;
    if ((rc = ctx->run_apply(ctx->dev.xs, ctx->dev.ys, precision, m))) return rc;
    const cudaMemcpyKind kout = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    CK(cudaMemcpyAsync(y, ctx->dev.ys + off_j, nvj * sizeof(double2), kout, ctx->stream));            // row1
    CK(cudaMemcpyAsync(y + nvj, ctx->dev.ys + off_j + nvj, nvj * sizeof(double2), kout, ctx->stream)); // row2
    CK(cudaStreamSynchronize(ctx->stream));
    return ctx->check_device_error();
}

static int apply_group_once(bem_ctx* const* ctxs, int32_t n, const bem_z* const* x, bem_z* const* y) {
    bem_ctx* const ctx = ctxs[0];
    CK(cudaSetDevice(ctx->device));
    // buffers and arguments of every member (no launches yet); the source
    // chunks are sized for the whole group's target tiles, so small meshes
    // get long chunks and the group, not each mesh, fills the SMs
    std::vector<ApplyPlan> P(n);
    int rc;
    int fill = 0;
    for (int i = 0; i < n; i++) {
        if ((rc = ctxs[i]->finalize())) return ctx->fail(rc, ctxs[i]->err);
        fill += ctxs[i]->geo.n_tiles;
    }
    for (int i = 0; i < n; i++) {
        bem_ctx* c = ctxs[i];
        if ((rc = c->finalize()) || (rc = c->ensure_near())) return rc == BEM_OK ? rc : ctx->fail(rc, c->err);
        ApplyMode m;
        m.tgt_dom_lo = 0; m.tgt_dom_hi = c->geo.n_dom; m.src_dom_lo = 0; m.src_dom_hi = c->geo.n_dom;
        m.kre = c->k0re; m.kim = c->k0im; m.slot1 = 1; m.coef = c->dev.coef; m.near = &c->pmchwt_near;
        if ((rc = c->plan_apply((const double2*)x[i], (double2*)y[i], BEM_PREC_FP32, m, P[i], fill)))
            return ctx->fail(rc, c->err);
        if (c != ctx && c->stream != ctx->stream) CK(cudaStreamSynchronize(c->stream));  // its own work first
    }
    GroupCache* G = ctx->group;
    bool valid = G && G->exec && (int)G->ctxs.size() == n;
    for (int i = 0; valid && i < n; i++)
        valid = G->ctxs[i] == ctxs[i] && G->gens[i] == ctxs[i]->gen && G->io[2 * i] == x[i] && G->io[2 * i + 1] == y[i];
    if (!valid) {
        // the work list over all members, heaviest first (as for one mesh)
        std::vector<std::pair<int64_t, int4>> items;
        std::vector<FarArgs32> table(n);
        for (int i = 0; i < n; i++) {
            const Geometry& g = ctxs[i]->geo;
            const FarArgs32& fa = P[i].fa32;
            table[i] = fa;
            table[i].work = nullptr;
            for (int t = 0; t < P[i].n_tgt; t++) {
                const int d = g.tile_dom[fa.tgt_begin + t];
                const int own_b = g.dom_tile_begin[d], own_e = g.dom_tile_end[d];
                for (int cch = 0; cch < P[i].n_chunks; cch++) {
                    const int sb = fa.src_begin + cch * fa.chunk_tiles, se = std::min(sb + fa.chunk_tiles, fa.src_end);
                    int64_t w = 0;
                    for (int sidx = sb; sidx < se; sidx++)
                        w += (int64_t)g.tile_ntri[sidx] * (1 + (fa.slot1 && sidx >= own_b && sidx < own_e));
                    items.push_back({-w, make_int4(i, t, cch, 0)});
                }
            }
        }
        std::stable_sort(items.begin(), items.end(),
                         [](const std::pair<int64_t, int4>& a, const std::pair<int64_t, int4>& b) { return a.first < b.first; });
        std::vector<int4> work(items.size());
        for (size_t k = 0; k < items.size(); k++) work[k] = items[k].second;
        if (!G) {
            G = new GroupCache();
            ctx->group = G;
        }
        if (G->exec) {
            cudaGraphExecDestroy(G->exec);
            G->exec = nullptr;
        }
        ctx->dfree(G->table);
        ctx->dfree(G->work);
        G->table = nullptr;
        G->work = nullptr;
        if ((rc = upload(ctx, &G->table, table)) || (rc = upload(ctx, &G->work, work))) return rc;
        G->n_work = (int64_t)work.size();
        if (!G->cap) CK(cudaStreamCreateWithFlags(&G->cap, cudaStreamNonBlocking));
        CK(launch_far32_group(G->table, G->work, 0, G->cap));  // one-time kernel attribute, outside the capture
        CK(cudaStreamSynchronize(ctx->stream));                 // the uploads are done before the graph exists
        cudaGraph_t graph;
        CK(cudaStreamBeginCapture(G->cap, cudaStreamCaptureModeThreadLocal));
        cudaError_t e = cudaSuccess;
        for (int i = 0; i < n && e == cudaSuccess; i++) e = launch_gather(P[i].ga, G->cap);
        if (e == cudaSuccess) e = launch_far32_group(G->table, G->work, G->n_work, G->cap);
        for (int i = 0; i < n && e == cudaSuccess; i++) {
            e = launch_project(P[i].pa, G->cap);
            if (e == cudaSuccess) e = launch_reduce(P[i].ra, G->cap);
        }
        const cudaError_t e2 = cudaStreamEndCapture(G->cap, &graph);
        if (e != cudaSuccess || e2 != cudaSuccess)
            return ctx->fail(BEM_ERR_CUDA, std::string("group capture: ") + cudaGetErrorString(e != cudaSuccess ? e : e2));
        e = cudaGraphInstantiate(&G->exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) return ctx->fail(BEM_ERR_CUDA, std::string("group graph: ") + cudaGetErrorString(e));
        G->ctxs.assign(ctxs, ctxs + n);
        G->gens.resize(n);
        for (int i = 0; i < n; i++) G->gens[i] = ctxs[i]->gen;
        G->io.resize(2 * n);
        for (int i = 0; i < n; i++) {
            G->io[2 * i] = x[i];
            G->io[2 * i + 1] = y[i];
        }
    }
    CK(cudaGraphLaunch(G->exec, ctx->stream));
    ctx->launches += 1 + 3 * n;
    return BEM_OK;
}

// Several meshes in one far-field launch (see include/bem.h).
int bem_apply_group(bem_ctx* const* ctxs, int32_t n, const bem_z* const* x, bem_z* const* y) {
    if (!ctxs || !x || !y || n < 1 || n > 4096) return BEM_ERR_INVALID_ARG;
    bem_ctx* const ctx = ctxs[0];
    if (!ctx) return BEM_ERR_INVALID_ARG;
    for (int i = 0; i < n; i++) {
        if (!ctxs[i] || !x[i] || !y[i]) return ctx->fail(BEM_ERR_INVALID_ARG, "null context or vector in the group");
        if (ctxs[i]->device != ctx->device) return ctx->fail(BEM_ERR_INVALID_ARG, "group contexts on different devices");
        for (int j = 0; j < i; j++)
            if (ctxs[j] == ctxs[i]) return ctx->fail(BEM_ERR_INVALID_ARG, "a context appears twice in the group");
    }
    // (as without_optional_if_short, for every member)
    auto run = [&](bool frugal) {
        for (int i = 0; i < n; i++) {
            ctxs[i]->frugal = frugal;
            ctxs[i]->short_of_memory = false;
            ctxs[i]->pinned++;
        }
        const int rc = apply_group_once(ctxs, n, x, y);
        for (int i = 0; i < n; i++) {
            ctxs[i]->frugal = false;
            ctxs[i]->pinned--;
        }
        return rc;
    };
    const int rc = run(false);
    bool refused = false, given = false;
    for (int i = 0; i < n; i++) refused |= ctxs[i]->short_of_memory;
    if (!rc || !refused) return rc;
    for (int i = 0; i < n; i++) given |= ctxs[i]->give_back();
    return given ? run(true) : rc;
}

int bem_profile_enable(bem_ctx* ctx, int enable) {
    if (!ctx) return BEM_ERR_INVALID_ARG;
    ctx->profiling = enable != 0;
    return BEM_OK;
}

int bem_profile_read(bem_ctx* ctx, double* far_ms, int64_t* far_launches, int64_t* kernel_launches, int reset) {
    if (!ctx) return BEM_ERR_INVALID_ARG;
    CK(cudaStreamSynchronize(ctx->stream));
    for (auto& e : ctx->far_events) {
        float ms = 0;
        CK(cudaEventElapsedTime(&ms, e.first, e.second));
        ctx->far_ms_acc += ms;
        ctx->far_count++;
        cudaEventDestroy(e.first);
        cudaEventDestroy(e.second);
    }
    ctx->far_events.clear();
    if (far_ms) *far_ms = ctx->far_ms_acc;
    if (far_launches) *far_launches = ctx->far_count;
    if (kernel_launches) *kernel_launches = ctx->launches;
    if (reset) {
        ctx->far_ms_acc = 0;
        ctx->far_count = 0;
        ctx->launches = 0;
    }
    return BEM_OK;
}

// Autotuner for the far-field launch shape: the number of source tiles one
// CTA streams (grid = target tiles x source chunks).  Short chunks give more
// CTAs (better balance over 152 SMs) but more partial potentials to write and
// reduce; long chunks the opposite.  Every candidate runs the whole operator
// application (gather, far field, projection, reduction) on the context's
// stream, timed with CUDA events after one warm-up run; the fastest is kept
// in the context's options and a per-process cache keyed by the tile counts.
namespace {
std::mutex g_tune_mu;
std::map<std::tuple<int, int, int, int>, int> g_tune_cache;  // (tiles, domains, lossy, precision) -> chunk
}  // namespace

int bem_autotune(bem_ctx* ctx, int precision, int32_t* chunk_tiles, double* best_ms) {
    if (!ctx) return BEM_ERR_INVALID_ARG;
    if (precision != BEM_PREC_FP32 && precision != BEM_PREC_FP64) return ctx->fail(BEM_ERR_INVALID_ARG, "bad precision");
    CK(cudaSetDevice(ctx->device));
    int rc = ctx->finalize();
    if (rc) return rc;
    if ((rc = ctx->ensure_near())) return rc;
    const Geometry& g = ctx->geo;
    bool lossy = ctx->k0im != 0;
    for (auto& d : ctx->doms) lossy |= d.kim != 0;
    const auto key = std::make_tuple(g.n_tiles, g.n_dom, (int)lossy, precision);
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end() && !best_ms) {
            ctx->opts.chunk_tiles = it->second;
            if (chunk_tiles) *chunk_tiles = it->second;
            return BEM_OK;
        }
    }
    const int64_t N = g.n_dof;
    double2* x = (double2*)ctx->dalloc(2 * N * sizeof(double2), &rc);
    if (rc) return rc;
    double2* y = x + N;
    CK(cudaMemsetAsync(x, 0, N * sizeof(double2), ctx->stream));
    std::vector<int> cand;
    for (int c : {8, 16, 32, 64, 128, 256})
        if (c <= CHUNK_MAX && (c <= g.n_tiles || cand.empty())) cand.push_back(c);
    cand.push_back(0);  // the built-in heuristic
    const int saved = ctx->opts.chunk_tiles;
    cudaEvent_t e0, e1;
    CK(cudaEventCreate(&e0));
    CK(cudaEventCreate(&e1));
    int best = saved;
    double best_t = 1e300;
    for (int c : cand) {
        ctx->opts.chunk_tiles = c;
        if ((rc = ctx->apply_ahat(x, y, precision))) break;  // warm-up (and partial buffer sizing)
        CK(cudaEventRecord(e0, ctx->stream));
        const int reps = 2;
        for (int r = 0; r < reps && !rc; r++) rc = ctx->apply_ahat(x, y, precision);
        if (rc) break;
        CK(cudaEventRecord(e1, ctx->stream));
        CK(cudaEventSynchronize(e1));
        float ms = 0;
        CK(cudaEventElapsedTime(&ms, e0, e1));
        if (ms / reps < best_t) {
            best_t = ms / reps;
            best = c;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaStreamSynchronize(ctx->stream);
    ctx->dfree(x);
    // the partial-potential buffer was sized for the largest candidate; the
    // next application allocates what the chosen shape needs
    if (ctx->partial) {
        ctx->dfree(ctx->partial);
        ctx->partial = nullptr;
        ctx->partial_bytes = ctx->partial_need = 0;
    }
    if (rc) {
        ctx->opts.chunk_tiles = saved;
        return rc;
    }
    ctx->opts.chunk_tiles = best;
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        g_tune_cache[key] = best;
    }
    if (chunk_tiles) *chunk_tiles = best;
    if (best_ms) *best_ms = best_t;
    return ctx->check_device_error();
}

int bem_memory_info(const bem_ctx* ctx, int64_t* used, int64_t* peak) {
    if (!ctx) return BEM_ERR_INVALID_ARG;
    if (used) *used = (int64_t)ctx->used_bytes;
    if (peak) *peak = (int64_t)ctx->peak_bytes;
    return BEM_OK;
}

int bem_estimate_solve_bytes(const bem_ctx* ctx, int64_t n_exc, const bem_solve_opts* opts, int64_t* bytes) {
    if (!ctx || !bytes || n_exc < 1) return BEM_ERR_INVALID_ARG;
    bem_solve_opts o;
    bem_default_solve_opts(&o);
    if (opts) o = *opts;
    *bytes = estimate_solve_bytes(ctx, n_exc, o);
    return BEM_OK;
}

const char* bem_last_error(const bem_ctx* ctx) {
    if (!ctx) return "null context";
    return ctx->err.c_str();
}

int bem_quadrature_table(int which, int n, double* buf, int* n_out) {
    if (!buf || !n_out) return BEM_ERR_INVALID_ARG;
    if (which == 0) {
        Quadrature q;
        if (!build_quadrature(q, 2)) return BEM_ERR_STATE;
        for (int i = 0; i < QP; i++) {
            buf[3 * i] = q.l1[i];
            buf[3 * i + 1] = q.l2[i];
            buf[3 * i + 2] = q.w[i];
        }
        *n_out = QP;
        return BEM_OK;
    }
    if (which == 1) {
        if (n < 1 || n > 64) return BEM_ERR_INVALID_ARG;
        std::vector<double> x, w;
        gauss_legendre01(n, x, w);
        for (int i = 0; i < n; i++) {
            buf[2 * i] = x[i];
            buf[2 * i + 1] = w[i];
        }
        *n_out = n;
        return BEM_OK;
    }
    return BEM_ERR_INVALID_ARG;
}

}  // extern "C"
