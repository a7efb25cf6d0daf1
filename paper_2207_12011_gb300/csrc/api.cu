// Host runtime behind the C ABI declared in include/raypc.h: contexts,
// resident volumes with their levels of detail, brick min/max and brush
// classification, transfer functions, and the render / histogram entry
// points. Every entry point validates its arguments, enqueues its work on
// the caller's stream and reports failures as status codes with a
// thread-local message; nothing aborts the process.
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "host_math.h"
#include "runtime.h"

using namespace raypc;

namespace {
thread_local std::string g_err;
std::atomic<unsigned long long> g_launches{0};
}  // namespace

namespace raypc {

raypc_status fail(raypc_status code, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

raypc_status cuda_fail(cudaError_t e, const char* what) {
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return fail(RAYPC_ERR_OOM, "%s: %s", what, cudaGetErrorString(e));
    }
    return fail(RAYPC_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

}  // namespace raypc

namespace {

void free_level(Level& L) {
    void* ptrs[] = {L.cells, L.pairs, L.bmin, L.bmax, L.active, L.skippable, L.list, L.n_active,
                    L.sbmin, L.sbmax, L.sactive, L.cls, L.tf_sactive, L.sdist, L.tf_sdist};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    L = Level{};
}

void free_bricks(Level& L) {
    void* ptrs[] = {L.bmin, L.bmax, L.active, L.skippable, L.list, L.n_active,
                    L.sbmin, L.sbmax, L.sactive, L.tf_sactive, L.sdist, L.tf_sdist};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    L.bmin = L.bmax = L.sbmin = L.sbmax = nullptr;
    L.active = L.skippable = L.list = L.n_active = L.sactive = L.tf_sactive = nullptr;
    L.sdist = L.tf_sdist = nullptr;
    L.sdist_of = nullptr;
    L.stats.odd = nullptr;
    L.bricks = L.classified = L.cls_valid = false;
}

void free_staging(Volume* V) {
    for (int i = 0; i < 2; ++i) {
        if (V->staging[i]) cudaFree(V->staging[i]);
        if (V->ev_consumed[i]) cudaEventDestroy(V->ev_consumed[i]);
        V->staging[i] = nullptr;
        V->ev_consumed[i] = nullptr;
        V->consumed_pending[i] = false;
    }
    if (V->ev_copied) cudaEventDestroy(V->ev_copied);
    if (V->copy_stream) cudaStreamDestroy(V->copy_stream);
    V->staging_bytes = 0;
    V->stage_next = 0;
    V->ev_copied = nullptr;
    V->copy_stream = nullptr;
}

void free_volume(raypc_ctx* ctx, Volume* V) {
    free_staging(V);
    for (auto& L : V->lv) free_level(L);
    if (V->mags) cudaFree(V->mags);
    if (V->tf) cudaFree(V->tf);
    if (V->tf_prefix) cudaFree(V->tf_prefix);
    ctx->used -= V->bytes < ctx->used ? V->bytes : ctx->used;
    delete V;
}


// The classification is out of date (new values, levels or brush).
void unclassify(Volume* V) {
    for (auto& L : V->lv) {
        L.classified = L.cls_valid = false;
        L.sdist_of = nullptr;
    }
}

// Classify the sub-bricks of every built level under the current brush and compute
// the cell classes of level with_classes (its buffer allocated; null: none), in one launch.
raypc_status classify_all(Volume* V, Level* with_classes, cudaStream_t s) {
    BrushLaunch P{};
    for (int l = 0; l < V->nlev; ++l) {
        Level& L = V->lv[l];
        if (!L.bricks) return fail(RAYPC_ERR_INVALID_ARG, "bricks of level %d are not built", l);
        BrushItem& it = P.items[P.nitems++];
        it = brush_item(V, L, V->brush);
        it.active = L.sactive;
        it.cls = &L == with_classes ? L.cls : nullptr;
    }
    CK(launch_brush(P, V->dtype, s), "classification kernel");
    unclassify(V);
    for (int l = 0; l < V->nlev; ++l) V->lv[l].classified = true;
    if (with_classes) with_classes->cls_valid = true;
    return RAYPC_OK;
}

// Lazily classify when a brush is set but the bricks changed since.
raypc_status ensure_classified(Volume* V, Level& L, cudaStream_t s) {
    if (L.classified) return RAYPC_OK;
    if (!V->brush_set) return fail(RAYPC_ERR_INVALID_ARG, "raypc_set_brush must run first");
    return classify_all(V, nullptr, s);
}

// The level's cell class buffer (allocated on first use; words of cells outside active
// sub-bricks are never written again).
raypc_status alloc_cell_classes(raypc_ctx* ctx, Volume* V, Level& L, cudaStream_t s) {
    if (L.cls) return RAYPC_OK;
    const size_t bytes = (size_t)L.n * L.n * L.n * sizeof(uint16_t);
    raypc_status st = ctx->alloc((void**)&L.cls, bytes, &V->bytes);
    if (st) {
        L.cls = nullptr;
        return st;
    }
    CK(cudaMemsetAsync(L.cls, 0, bytes, s), "clear cell classes");
    return RAYPC_OK;
}

raypc_status alloc_bricks(raypc_ctx* ctx, Volume* V, Level& L) {
    if (L.bmin) return RAYPC_OK;
    size_t nbk = L.nbricks();
    size_t mm = nbk * V->nvars * sizeof(float);
    size_t words = L.nwords() * sizeof(uint32_t);
    size_t smm = L.nsbricks() * V->nvars * sizeof(float);
    raypc_status st;
    if ((st = ctx->alloc((void**)&L.sbmin, smm, &V->bytes)) ||
        (st = ctx->alloc((void**)&L.sbmax, smm, &V->bytes)) ||
        (st = ctx->alloc((void**)&L.sactive, L.nswords() * sizeof(uint32_t) + L.nsbricks() * V->nvars, &V->bytes)) ||
        (st = ctx->alloc((void**)&L.tf_sactive, L.nswords() * sizeof(uint32_t), &V->bytes)) ||
        (st = ctx->alloc((void**)&L.bmin, mm, &V->bytes)) ||
        (st = ctx->alloc((void**)&L.bmax, mm, &V->bytes)) ||
        (st = ctx->alloc((void**)&L.active, words, &V->bytes)) ||
        (st = ctx->alloc((void**)&L.skippable, words, &V->bytes)) ||
        (st = ctx->alloc((void**)&L.list, nbk * sizeof(uint32_t), &V->bytes)) ||
        (st = ctx->alloc((void**)&L.n_active, sizeof(uint32_t), &V->bytes))) {
        free_bricks(L);
        return st;
    }
    L.stats.odd = reinterpret_cast<uint8_t*>(L.sactive + L.nswords());   // behind the words of the same allocation
    return RAYPC_OK;
}

// Staging of a host source for raypc_update_volume: two buffers of the volume's own, used in
// turn, and its copy stream (created on first use, charged to the budget). The copy into a
// buffer waits only until the ingest two updates back has read it, so consecutive time steps'
// copies run back to back and overlap whatever runs on the caller's stream; the caller's stream
// waits for the copy. Returns false when the buffers cannot be had (budget), and the caller
// falls back to a stream-ordered temporary.
bool stage_host_source(raypc_ctx* ctx, Volume* V, const void* src, size_t bytes, cudaStream_t s,
                       const void** dsrc, int* slot, raypc_status* st) {
    *st = RAYPC_OK;
    if (V->staging_bytes != bytes) {
        if (V->copy_stream) cudaStreamSynchronize(V->copy_stream);
        for (int i = 0; i < 2; ++i) {
            if (V->consumed_pending[i]) cudaEventSynchronize(V->ev_consumed[i]);
            if (V->staging[i]) cudaFree(V->staging[i]);
            V->staging[i] = nullptr;
            V->consumed_pending[i] = false;
        }
        V->bytes -= 2 * V->staging_bytes < V->bytes ? 2 * V->staging_bytes : V->bytes;
        ctx->used -= 2 * V->staging_bytes < ctx->used ? 2 * V->staging_bytes : ctx->used;
        V->staging_bytes = 0;
        if (ctx->alloc(&V->staging[0], bytes, &V->bytes) != RAYPC_OK) {
            cudaGetLastError();
            return false;
        }
        if (ctx->alloc(&V->staging[1], bytes, &V->bytes) != RAYPC_OK) {
            cudaGetLastError();
            cudaFree(V->staging[0]);
            V->staging[0] = nullptr;
            V->bytes -= bytes < V->bytes ? bytes : V->bytes;
            ctx->used -= bytes < ctx->used ? bytes : ctx->used;
            return false;
        }
        V->staging_bytes = bytes;
        V->stage_next = 0;
    }
    const int i = V->stage_next;
    cudaError_t e = cudaSuccess;
    if (!V->copy_stream) e = cudaStreamCreateWithFlags(&V->copy_stream, cudaStreamNonBlocking);
    if (e == cudaSuccess && !V->ev_copied) e = cudaEventCreateWithFlags(&V->ev_copied, cudaEventDisableTiming);
    for (int k = 0; k < 2 && e == cudaSuccess; ++k)
        if (!V->ev_consumed[k]) e = cudaEventCreateWithFlags(&V->ev_consumed[k], cudaEventDisableTiming);
    if (e == cudaSuccess && V->consumed_pending[i]) e = cudaStreamWaitEvent(V->copy_stream, V->ev_consumed[i], 0);
    if (e == cudaSuccess) e = cudaMemcpyAsync(V->staging[i], src, bytes, cudaMemcpyHostToDevice, V->copy_stream);
    if (e == cudaSuccess) e = cudaEventRecord(V->ev_copied, V->copy_stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s, V->ev_copied, 0);
    if (e != cudaSuccess) {
        *st = cuda_fail(e, "host to device copy");
        return true;
    }
    *dsrc = V->staging[i];
    *slot = i;
    V->stage_next = i ^ 1;
    return true;
}

raypc_status ingest(raypc_ctx* ctx, Volume* V, const void* src, int src_is_device, int src_dtype,
                    cudaStream_t s, bool own_staging = false) {
    Level& L = V->lv[0];
    const size_t nvox = (size_t)L.n * L.n * L.n;
    const void* dsrc = src;
    void* staging = nullptr;
    cudaError_t e;
    bool staged = false;
    int slot = 0;
    if (!src_is_device && own_staging) {
        raypc_status st;
        staged = stage_host_source(ctx, V, src, nvox * V->nvars * elem_size(src_dtype), s, &dsrc, &slot, &st);
        if (st != RAYPC_OK) return st;
    }
    if (!src_is_device && !staged) {
        size_t src_bytes = nvox * V->nvars * elem_size(src_dtype);
        e = allocate(ctx->device, [&] { return cudaMallocAsync(&staging, src_bytes, s); });
        if (e != cudaSuccess) return cuda_fail(e, "staging allocation");
        e = cudaMemcpyAsync(staging, src, src_bytes, cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) { cudaFreeAsync(staging, s); return cuda_fail(e, "host to device copy"); }
        dsrc = staging;
    }
    // when the next level is allocated (raypc_build_bricks built it before), its cells and
    // x-pairs come out of the same pass over the source
    Level& C = V->lv[1];
    const bool next = C.cells && C.pairs && C.n * 2 == L.n && ingest_next_level_fits(dsrc, L.n);
    e = cudaMemsetAsync(V->mags, 0, kLevelStatsBytes * (1 + RAYPC_MAX_LOD), s);
    if (e == cudaSuccess && next)
        e = launch_ingest_next_level(dsrc, src_dtype, L.cells, L.pairs, V->dtype, L.n, V->nvars, L.bmin, L.bmax,
                                     L.sbmin, L.sbmax, C.cells, C.pairs, L.stats, s);
    else if (e == cudaSuccess)
        e = launch_ingest(dsrc, src_dtype, L.cells, L.pairs, V->dtype, L.n, V->nvars, L.bmin, L.bmax, L.sbmin,
                          L.sbmax, L.stats, s);
    for (auto& l : V->lv) l.fresh = false;
    C.fresh = next && e == cudaSuccess;
    if (staging) cudaFreeAsync(staging, s);
    if (staged && e == cudaSuccess) {
        e = cudaEventRecord(V->ev_consumed[slot], s);  // the staging buffer is free once this ingest ran
        V->consumed_pending[slot] = e == cudaSuccess;
    }
    if (e != cudaSuccess) return cuda_fail(e, "ingest kernel");
    L.bricks = true;               // level-0 brick min/max come out of the ingest pass
    unclassify(V);
    return RAYPC_OK;
}

}  // namespace

void raypc::count_launches(int k) { g_launches.fetch_add((unsigned long long)k, std::memory_order_relaxed); }

namespace raypc {

void set_last_error(const char* msg) { g_err = msg; }

namespace {
std::mutex g_pools_mu;
std::vector<std::pair<int, cudaMemPool_t>> g_pools;
}  // namespace

void pool_opened(int device, cudaMemPool_t pool) {
    std::lock_guard<std::mutex> lk(g_pools_mu);
    g_pools.emplace_back(device, pool);
}

void pool_closed(cudaMemPool_t pool) {
    std::lock_guard<std::mutex> lk(g_pools_mu);
    g_pools.erase(std::remove_if(g_pools.begin(), g_pools.end(), [&](const auto& p) { return p.second == pool; }), g_pools.end());
}

bool trim_pools(int device, bool wait) {
    std::lock_guard<std::mutex> lk(g_pools_mu);
    unsigned long long held = 0;
    for (const auto& p : g_pools) {
        unsigned long long v = 0;
        if (p.first == device && cudaMemPoolGetAttribute(p.second, cudaMemPoolAttrReservedMemCurrent, &v) == cudaSuccess) held += v;
    }
    if (!held) return false;
    if (wait) cudaDeviceSynchronize();
    for (const auto& p : g_pools)
        if (p.first == device) cudaMemPoolTrimTo(p.second, 0);
    cudaGetLastError();
    return true;
}

raypc_status get_volume(raypc_ctx* ctx, int vol, Volume** out) {
    auto it = ctx->vols.find(vol);
    if (it == ctx->vols.end()) return fail(RAYPC_ERR_NOT_FOUND, "unknown volume id %d", vol);
    *out = it->second;
    return RAYPC_OK;
}

raypc_status get_level(Volume* V, int lod, Level** out) {
    if (lod < 0 || lod >= V->nlev) return fail(RAYPC_ERR_NOT_FOUND, "level %d not built (have %d)", lod, V->nlev);
    *out = &V->lv[lod];
    return RAYPC_OK;
}

void finish_position_brush(RenderArgs& a) {
    a.keep_lo2 = a.rin2;
    a.keep_hi2 = a.rout2;
    if ((a.brush.pmask >> 3) & 1u) {
        // lo_r <= sqrt_rn(|p|^2) <= hi_r  <=>  L <= |p|^2 <= H for the exact thresholds L, H
        const float L = radius_threshold2(a.brush.plo[3], false), H = radius_threshold2(a.brush.phi[3], true);
        a.keep_lo2 = fmaxf(a.keep_lo2, L);
        a.keep_hi2 = fminf(a.keep_hi2, H);
    }
    a.keep_lo2 = fminf(a.keep_lo2, 0x1p100f);          // finite (the core-jump bound scales it)
    a.open = a.brush.mask == 0u && a.brush.pmask == 0u;
}

raypc_status make_render_args(Volume* V, Level* L, const raypc_camera* cam, int w, int h,
                              const raypc_render_opts* opts, float* out_rgba_dev,
                              unsigned long long* stats_dev, RenderArgs* out) {
    if (!cam || !out_rgba_dev) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    if (w < 1 || h < 1 || w > 32768 || h > 32768) return fail(RAYPC_ERR_INVALID_ARG, "image size %d x %d out of range", w, h);
    if (((uintptr_t)out_rgba_dev) & 15u) return fail(RAYPC_ERR_INVALID_ARG, "out_rgba_dev must be 16-byte aligned");
    for (int i = 0; i < 3; ++i)
        if (!isfinite(cam->eye[i]) || !isfinite(cam->target[i]) || !isfinite(cam->up[i]))
            return fail(RAYPC_ERR_INVALID_ARG, "non-finite camera");
    if (!(cam->tan_half_vfov > 0.f) || !isfinite(cam->tan_half_vfov)) return fail(RAYPC_ERR_INVALID_ARG, "tan_half_vfov must be > 0");
    {
        float fx = cam->target[0] - cam->eye[0], fy = cam->target[1] - cam->eye[1], fz = cam->target[2] - cam->eye[2];
        if (fx == 0.f && fy == 0.f && fz == 0.f) return fail(RAYPC_ERR_INVALID_ARG, "eye == target");
        float cx = fy * cam->up[2] - fz * cam->up[1], cy = fz * cam->up[0] - fx * cam->up[2], cz = fx * cam->up[1] - fy * cam->up[0];
        if (cx == 0.f && cy == 0.f && cz == 0.f) return fail(RAYPC_ERR_INVALID_ARG, "up is parallel to the view direction");
    }
    raypc_render_opts o{};
    o.ert = 1;
    if (opts) o = *opts;
    for (int i = 0; i < 4; ++i)
        if (!isfinite(o.bg[i])) return fail(RAYPC_ERR_INVALID_ARG, "non-finite background");
    if (V->stale) return fail(RAYPC_ERR_INVALID_ARG, "volume updated: raypc_build_bricks must run before render");
    if (!L->bricks) return fail(RAYPC_ERR_INVALID_ARG, "bricks of the level are not built");
    if (!V->tf_set) return fail(RAYPC_ERR_INVALID_ARG, "set_tf must run before render");
    float dt = o.step > 0.f ? o.step : 1.0f / (float)L->n;
    if (!isfinite(dt) || dt < 2.0f * V->r_out / 4194304.0f)
        return fail(RAYPC_ERR_INVALID_ARG, "step %g too small (at most 2^21 samples per chord)", dt);
    RenderArgs a{};
    a.lv.pairs = L->pairs;
    a.lv.n = L->n;
    a.lv.nsb = L->nsb;
    a.lv.pd = subbrick_pad(L->n);
    a.lv.pbias = narrow_bias(L->n);
    a.lv.plast = (uint32_t)(padded_bytes(L->n) - 1);
    a.lv.sactive = L->sactive;
    a.nvars = V->nvars;
    a.brush = V->brush;
    for (int i = 0; i < 3; ++i) { a.eye[i] = cam->eye[i]; a.target[i] = cam->target[i]; a.up[i] = cam->up[i]; }
    a.tan_half = cam->tan_half_vfov;
    a.w = w;
    a.h = h;
    a.dt = dt;
    // samples that stay in a box of inactive sub-bricks extending 4 (D - 1) cells beyond the current
    // sub-brick, D >= 2, 4, kDistCap (the lattice moves a cell index by at most dt n/2 cells per
    // sample on any axis, 1/16 cell covers its rounding); whole numbers, 0 for coarse steps
    const float cells_per_step = dt * (0.5f * (float)L->n);
    const int box[3] = {1, 3, kDistCap - 1};
    for (int i = 0; i < 3; ++i) a.jump[i] = floorf((4.0f * (float)box[i] - 0.0625f) / cells_per_step);
    // A sample's |p| exceeds r_out by at most about |eye| 2^-20 (rounding of the sphere interval, t
    // and p), so -1 <= u < n on every axis when r_out <= 1 and |eye| n < 2^17.
    const float eye_max = fmaxf(fabsf(cam->eye[0]), fmaxf(fabsf(cam->eye[1]), fabsf(cam->eye[2])));
    const size_t plane_bytes = (size_t)L->n * L->n * L->n * 2 * elem_size(V->dtype);
    a.narrow = V->r_out <= 1.0f && eye_max * (float)L->n < 131072.0f && plane_bytes < ((size_t)1 << 32);
    a.rin2 = V->r_in * V->r_in;
    a.rout2 = V->r_out * V->r_out;
    finish_position_brush(a);
    a.tf = V->tf;
    a.color_var = V->color_var;
    a.tf_lo = V->tf_lo;
    a.tf_scale = 255.0f / (V->tf_hi - V->tf_lo);
    for (int i = 0; i < 4; ++i) a.bg[i] = o.bg[i];
    a.ert = o.ert ? 1 : 0;
    if (o.skip < RAYPC_AUTO || o.skip > RAYPC_SKIP_OFF) return fail(RAYPC_ERR_INVALID_ARG, "bad skip option %d", o.skip);
    if (o.variant < RAYPC_AUTO || o.variant > kNumVariants) return fail(RAYPC_ERR_INVALID_ARG, "bad variant %d", o.variant);
    int variant = o.variant, skip = o.skip;
    int dev = 0;
    cudaGetDevice(&dev);
    resolve_launch(dev, V->dtype, L->n, &variant, &skip);
    a.skip = skip == RAYPC_SKIP_OFF ? 0 : 1;
    a.variant = variant;
    a.out = reinterpret_cast<float4*>(out_rgba_dev);
    a.counts = o.counts_dev;
    a.depth = o.depth_dev;
    a.stats = stats_dev;
    *out = a;
    return RAYPC_OK;
}

BrushItem brush_item(const Volume* V, const Level& L, const BrushArgs& brush) {
    BrushItem it{};
    it.sbmin = L.sbmin;
    it.sbmax = L.sbmax;
    it.cells = L.cells;
    it.stats = L.stats;
    it.n = L.n;
    it.nsb = L.nsb;
    it.nvars = V->nvars;
    it.rin2 = V->r_in * V->r_in;
    it.rout2 = V->r_out * V->r_out;
    it.brush = brush;
    return it;
}

raypc_status ensure_cell_classes(raypc_ctx* ctx, Volume* V, Level& L, cudaStream_t s) {
    if (L.cls_valid) return RAYPC_OK;
    if (!L.classified && !V->brush_set) return fail(RAYPC_ERR_INVALID_ARG, "raypc_set_brush must run first");
    raypc_status st = alloc_cell_classes(ctx, V, L, s);
    if (st) return st;
    if (!L.classified) return classify_all(V, &L, s);
    BrushLaunch P{};                                         // this level's bits again, and its classes
    P.nitems = 1;
    P.items[0] = brush_item(V, L, V->brush);
    P.items[0].active = L.sactive;
    P.items[0].cls = L.cls;
    CK(launch_brush(P, V->dtype, s), "cell class kernel");
    L.cls_valid = true;
    return RAYPC_OK;
}

raypc_status brush_from_host(const Volume* V, const float* lo, const float* hi, uint32_t active_mask, BrushArgs* out) {
    if (!lo || !hi) return fail(RAYPC_ERR_INVALID_ARG, "NULL brush bounds");
    if (active_mask >> V->nvars) return fail(RAYPC_ERR_INVALID_ARG, "active_mask 0x%x names variables >= nvars %d", active_mask, V->nvars);
    BrushArgs b{};
    for (int v = 0; v < kMaxVars; ++v) { b.lo[v] = -INFINITY; b.hi[v] = INFINITY; }
    for (int v = 0; v < V->nvars; ++v) {
        if (isnan(lo[v]) || isnan(hi[v])) return fail(RAYPC_ERR_INVALID_ARG, "NaN brush bound for variable %d", v);
        b.lo[v] = lo[v];
        b.hi[v] = hi[v];
    }
    b.mask = active_mask;
    for (int a = 0; a < kNumPos; ++a) { b.plo[a] = -INFINITY; b.phi[a] = INFINITY; }
    b.pmask = 0u;
    *out = b;
    return RAYPC_OK;
}

raypc_status pos_from_host(const float* lo, const float* hi, uint32_t pos_mask, BrushArgs* b) {
    if (pos_mask >> kNumPos) return fail(RAYPC_ERR_INVALID_ARG, "pos_mask 0x%x names axes >= %d", pos_mask, kNumPos);
    for (int a = 0; a < kNumPos; ++a) { b->plo[a] = -INFINITY; b->phi[a] = INFINITY; }
    b->pmask = pos_mask;
    if (!pos_mask) return RAYPC_OK;
    if (!lo || !hi) return fail(RAYPC_ERR_INVALID_ARG, "NULL position bounds");
    for (int a = 0; a < kNumPos; ++a) {
        if (!((pos_mask >> a) & 1u)) continue;
        if (isnan(lo[a]) || isnan(hi[a])) return fail(RAYPC_ERR_INVALID_ARG, "NaN bound for position axis %d", a);
        b->plo[a] = lo[a];
        b->phi[a] = hi[a];
    }
    return RAYPC_OK;
}

}  // namespace raypc

extern "C" {

const char* raypc_last_error(void) { return g_err.c_str(); }

raypc_status raypc_kernel_launches(unsigned long long* out) {
    if (!out) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    *out = g_launches.load();
    return RAYPC_OK;
}

raypc_status raypc_create(raypc_ctx** out, int device, size_t hbm_budget_bytes) {
    if (!out) return fail(RAYPC_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    int ndev = 0;
    CK(cudaGetDeviceCount(&ndev), "cudaGetDeviceCount");
    if (device < 0 || device >= ndev) return fail(RAYPC_ERR_INVALID_ARG, "device %d out of range (%d devices)", device, ndev);
    raypc_ctx* c = new raypc_ctx();
    c->device = device;
    c->budget = hbm_budget_bytes;
    {
        DeviceGuard g(device);
        if (g.ok) c->open_pool();
    }
    *out = c;
    g_err.clear();
    return RAYPC_OK;
}

raypc_status raypc_destroy(raypc_ctx* ctx) {
    if (!ctx) return RAYPC_OK;
    {
        std::lock_guard<std::mutex> lk(ctx->mu);
        DeviceGuard g(ctx->device);
        for (auto& kv : ctx->vols) free_volume(ctx, kv.second);
        ctx->vols.clear();
        if (ctx->pool) {
            pool_closed(ctx->pool);
            cudaMemPoolDestroy(ctx->pool);                 // released once its last frees have run
        }
    }
    delete ctx;
    return RAYPC_OK;
}

raypc_status raypc_memory_used(raypc_ctx* ctx, size_t* out_bytes) {
    if (!ctx || !out_bytes) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(ctx->mu);
    *out_bytes = ctx->used + ctx->pool_held();
    return RAYPC_OK;
}

raypc_status raypc_load_volume(raypc_ctx* ctx, const void* src, int src_is_device, int src_dtype,
                               int store_dtype, int nx, int ny, int nz, int nvars, float r_in,
                               float r_out, void* stream, int* out_vol) {
    if (!ctx || !src || !out_vol) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    if ((src_dtype != RAYPC_F32 && src_dtype != RAYPC_F16) || (store_dtype != RAYPC_F32 && store_dtype != RAYPC_F16))
        return fail(RAYPC_ERR_INVALID_ARG, "dtype must be RAYPC_F32 or RAYPC_F16");
    if (nvars < 1 || nvars > RAYPC_MAX_VARS) return fail(RAYPC_ERR_INVALID_ARG, "nvars %d not in 1..%d", nvars, RAYPC_MAX_VARS);
    if (nx < 2 || ny < 2 || nz < 2) return fail(RAYPC_ERR_INVALID_ARG, "grid must be at least 2 cells per axis");
    if (nx != ny || ny != nz) return fail(RAYPC_ERR_UNSUPPORTED, "only cubic grids are supported (%d x %d x %d)", nx, ny, nz);
    if (nx > kMaxRowsEdge) return fail(RAYPC_ERR_UNSUPPORTED, "grid edge %d > %d", nx, kMaxRowsEdge);
    if (!(r_in >= 0.f) || !(r_out > r_in) || !isfinite(r_out))
        return fail(RAYPC_ERR_INVALID_ARG, "need 0 <= r_in < r_out (got %g, %g)", r_in, r_out);
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    if (!g.ok) return fail(RAYPC_ERR_CUDA, "cannot select device %d", ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    const int n = nx;
    const size_t nvox = (size_t)n * n * n;
    Volume* V = new Volume();
    V->nvars = nvars;
    V->dtype = store_dtype;
    V->r_in = r_in;
    V->r_out = r_out;
    Level& L = V->lv[0];
    L.set_edge(n);
    L.cells_bytes = nvox * nvars * elem_size(store_dtype);
    L.pairs_bytes = 2 * L.cells_bytes;
    raypc_status st = ctx->alloc(&L.cells, L.cells_bytes, &V->bytes);
    if (st == RAYPC_OK) st = ctx->alloc(&L.pairs, L.pairs_bytes, &V->bytes);
    if (st == RAYPC_OK) st = alloc_bricks(ctx, V, L);
    if (st == RAYPC_OK) st = ctx->alloc((void**)&V->mags, kLevelStatsBytes * (1 + RAYPC_MAX_LOD), &V->bytes);
    if (st != RAYPC_OK) { free_volume(ctx, V); return st; }
    for (int l = 0; l <= RAYPC_MAX_LOD; ++l) V->lv[l].stats.mag = V->mags + l * (kMaxVars + 1);
    st = ingest(ctx, V, src, src_is_device, src_dtype, s);
    if (st != RAYPC_OK) { free_volume(ctx, V); return st; }
    if (!src_is_device) {
        // keep the simple contract of this entry point: the host source is consumed on return
        cudaError_t e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) { free_volume(ctx, V); return cuda_fail(e, "ingest"); }
    }
    V->nlev = 1;
    int id = ctx->next_id++;
    ctx->vols[id] = V;
    *out_vol = id;
    return RAYPC_OK;
}

raypc_status raypc_update_volume(raypc_ctx* ctx, int vol, const void* src, int src_is_device,
                                 int src_dtype, void* stream) {
    if (!ctx || !src) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    if (src_dtype != RAYPC_F32 && src_dtype != RAYPC_F16) return fail(RAYPC_ERR_INVALID_ARG, "bad src_dtype");
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    if ((st = ingest(ctx, V, src, src_is_device, src_dtype, (cudaStream_t)stream, true))) return st;
    V->stale = true;
    for (int l = 1; l <= RAYPC_MAX_LOD; ++l) V->lv[l].bricks = false;
    return RAYPC_OK;
}

raypc_status raypc_free_volume(raypc_ctx* ctx, int vol) {
    if (!ctx) return fail(RAYPC_ERR_INVALID_ARG, "NULL context");
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    ctx->vols.erase(vol);
    cudaDeviceSynchronize();
    free_volume(ctx, V);
    return RAYPC_OK;
}

raypc_status raypc_build_bricks(raypc_ctx* ctx, int vol, int brick_dim, int n_lod, void* stream) {
    if (!ctx) return fail(RAYPC_ERR_INVALID_ARG, "NULL context");
    if (brick_dim != RAYPC_BRICK) return fail(RAYPC_ERR_UNSUPPORTED, "brick_dim must be %d", RAYPC_BRICK);
    if (n_lod < 0 || n_lod > RAYPC_MAX_LOD) return fail(RAYPC_ERR_INVALID_ARG, "n_lod %d not in 0..%d", n_lod, RAYPC_MAX_LOD);
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    cudaStream_t s = (cudaStream_t)stream;
    // Level 0 brick min/max come out of every ingest; build the coarser levels,
    // each fused with its own brick min/max.
    for (int l = 1; l <= n_lod; ++l) {
        Level& P = V->lv[l - 1];
        Level& L = V->lv[l];
        int m = (P.n + 1) / 2;
        if (m < 2) return fail(RAYPC_ERR_INVALID_ARG, "level %d would have fewer than 2 cells per axis", l);
        if (!L.cells) {
            L.set_edge(m);
            L.cells_bytes = (size_t)m * m * m * V->nvars * elem_size(V->dtype);
            L.pairs_bytes = 2 * L.cells_bytes;
            st = ctx->alloc(&L.cells, L.cells_bytes, &V->bytes);
            if (st == RAYPC_OK) st = ctx->alloc(&L.pairs, L.pairs_bytes, &V->bytes);
            if (st) return st;
        }
        if ((st = alloc_bricks(ctx, V, L))) return st;
        if (L.fresh) {           // the ingest or the pass before already wrote this level's cells: its bricks,
                                 // and the next level's cells in the same pass where that is allocated too
            Level* C = l < n_lod && V->lv[l + 1].cells && V->lv[l + 1].n * 2 == L.n &&
                       ingest_next_level_fits(L.cells, L.n) ? &V->lv[l + 1] : nullptr;
            CK(launch_level_bricks(L.cells, V->dtype, L.n, V->nvars, L.bmin, L.bmax, L.sbmin, L.sbmax,
                                   C ? C->cells : nullptr, C ? C->pairs : nullptr, L.stats, s),
               "level bricks kernel");
            if (C) C->fresh = true;
        } else {
            CK(launch_lod(P.cells, P.n, L.cells, L.pairs, V->dtype, V->nvars, L.bmin, L.bmax, L.sbmin, L.sbmax,
                          L.stats, s),
               "LOD kernel");
            if (l < RAYPC_MAX_LOD) V->lv[l + 1].fresh = false;
        }
        L.fresh = false;
        L.bricks = true;
    }
    if (V->stale || 1 + n_lod > V->nlev) V->nlev = 1 + n_lod;   // stale coarser levels drop out
    V->stale = false;
    unclassify(V);
    return RAYPC_OK;
}

// Re-classify every built level under the volume's (new) brush and compute the
// cell classes of level 0, so that a render runs its kernel alone (coarser levels get
// their classes when first rendered).
static raypc_status reclassify(raypc_ctx* ctx, Volume* V, cudaStream_t s) {
    unclassify(V);
    if (V->stale) return RAYPC_OK;   // coarser levels are rebuilt by raypc_build_bricks, which classifies lazily
    const raypc_status st = alloc_cell_classes(ctx, V, V->lv[0], s);
    const raypc_status cl = classify_all(V, st ? nullptr : &V->lv[0], s);
    return cl ? cl : st;
}

raypc_status raypc_set_brush(raypc_ctx* ctx, int vol, const float* lo, const float* hi,
                             uint32_t active_mask, void* stream) {
    if (!ctx || !lo || !hi) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    BrushArgs b{};
    if ((st = brush_from_host(V, lo, hi, active_mask, &b))) return st;
    // the position brush stays as raypc_set_position_brush left it
    for (int a = 0; a < kNumPos; ++a) { b.plo[a] = V->brush.plo[a]; b.phi[a] = V->brush.phi[a]; }
    b.pmask = V->brush.pmask;
    V->brush = b;
    V->brush_set = true;
    return reclassify(ctx, V, (cudaStream_t)stream);
}

raypc_status raypc_set_position_brush(raypc_ctx* ctx, int vol, const float* lo, const float* hi,
                                      uint32_t pos_mask, void* stream) {
    if (!ctx) return fail(RAYPC_ERR_INVALID_ARG, "NULL context");
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    BrushArgs b = V->brush;
    if (!V->brush_set) {           // no variable brush yet: nothing restricted
        for (int v = 0; v < kMaxVars; ++v) { b.lo[v] = -INFINITY; b.hi[v] = INFINITY; }
        b.mask = 0u;
    }
    if ((st = pos_from_host(lo, hi, pos_mask, &b))) return st;
    V->brush = b;
    V->brush_set = true;
    return reclassify(ctx, V, (cudaStream_t)stream);
}

raypc_status raypc_set_tf(raypc_ctx* ctx, int vol, const float* rgbs, int color_var, float v_lo,
                          float v_hi, void* stream) {
    if (!ctx || !rgbs) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    if (!(v_lo < v_hi) || !isfinite(v_lo) || !isfinite(v_hi)) return fail(RAYPC_ERR_INVALID_ARG, "need finite v_lo < v_hi");
    for (int i = 0; i < 4 * RAYPC_TF_ENTRIES; ++i)
        if (!isfinite(rgbs[i])) return fail(RAYPC_ERR_INVALID_ARG, "non-finite transfer function entry %d", i);
    for (int i = 0; i < RAYPC_TF_ENTRIES; ++i)
        if (rgbs[4 * i + 3] < 0.f) return fail(RAYPC_ERR_INVALID_ARG, "negative extinction at entry %d", i);
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    if (color_var < 0 || color_var >= V->nvars) return fail(RAYPC_ERR_INVALID_ARG, "color_var %d out of range", color_var);
    if (!V->tf) {
        size_t dummy = 0;
        if ((st = ctx->alloc((void**)&V->tf, sizeof(float4) * RAYPC_TF_ENTRIES, &dummy))) return st;
        V->bytes += dummy;
    }
    if (!V->tf_prefix) {
        size_t dummy = 0;
        if ((st = ctx->alloc((void**)&V->tf_prefix, sizeof(int) * (RAYPC_TF_ENTRIES + 1), &dummy))) return st;
        V->bytes += dummy;
    }
    int prefix[RAYPC_TF_ENTRIES + 1];
    prefix[0] = 0;
    for (int i = 0; i < RAYPC_TF_ENTRIES; ++i) prefix[i + 1] = prefix[i] + (rgbs[4 * i + 3] > 0.f ? 1 : 0);
    CK(cudaMemcpyAsync(V->tf_prefix, prefix, sizeof(prefix), cudaMemcpyHostToDevice, (cudaStream_t)stream),
       "transfer function prefix upload");
    // pageable host source: cudaMemcpyAsync stages it before returning
    CK(cudaMemcpyAsync(V->tf, rgbs, sizeof(float4) * RAYPC_TF_ENTRIES, cudaMemcpyHostToDevice, (cudaStream_t)stream),
       "transfer function upload");
    V->color_var = color_var;
    V->tf_lo = v_lo;
    V->tf_hi = v_hi;
    V->tf_set = true;
    return RAYPC_OK;
}

// Empty-space distance of the sub-bricks under the activity bits the render reads (the
// brush's, or the TF-visible ones with tf_skip, in a grid of their own): the grid the march
// searches. It is kept until the brush or the values change, but for tf_skip and for renders
// asked to go without skipping: these only need the activity (they read the bits where the grid
// cannot be had, and nothing when nothing is restricted), so what they see is that of their own
// stream's order, also when a graph replays them.
static raypc_status ensure_distance(raypc_ctx* ctx, Volume* V, Level& L, RenderArgs& a, const raypc_render_opts* opts,
                                    cudaStream_t s) {
    if (a.open && !a.skip) return RAYPC_OK;
    const bool tf = opts && opts->tf_skip, off = opts && opts->skip == RAYPC_SKIP_OFF;
    uint8_t** grid = tf ? &L.tf_sdist : &L.sdist;
    if (!*grid) {
        const raypc_status st = ctx->alloc((void**)grid, padded_bytes(L.n), &V->bytes);
        if (st) *grid = nullptr;
        else if (!tf) L.sdist_of = nullptr;
        if (st && tf && L.sdist) grid = &L.sdist;            // no room for two: the other one is stale then
        else if (st) return a.skip ? st : RAYPC_OK;
    }
    if (tf || off || L.sdist_of != a.lv.sactive) {
        CK(launch_subbrick_distance(a.lv.sactive, L.n, *grid, false, s), "empty-space distance");
        if (grid == &L.sdist && (tf || !off)) L.sdist_of = tf ? nullptr : a.lv.sactive;
    }
    a.lv.sdist = *grid;
    return RAYPC_OK;
}

// With tf_skip, the render reads the activity bits ANDed with the TF visibility of
// the level's sub-bricks (computed for this render on its stream).
static raypc_status apply_tf_skip(Volume* V, Level& L, const raypc_render_opts* opts, RenderArgs& a, cudaStream_t s) {
    if (!opts || !opts->tf_skip) return RAYPC_OK;
    TfVisArgs t{};
    t.nsb = L.nsb;
    t.nvars = V->nvars;
    t.color_var = V->color_var;
    t.sbmin = L.sbmin;
    t.sbmax = L.sbmax;
    t.sactive = L.sactive;
    t.tf_prefix = V->tf_prefix;
    t.tf_lo = a.tf_lo;
    t.tf_scale = a.tf_scale;
    t.out_sactive = L.tf_sactive;
    CK(launch_tf_visibility(t, s), "TF visibility kernel");
    a.lv.sactive = L.tf_sactive;
    a.open = 0;
    return RAYPC_OK;
}

raypc_status raypc_render(raypc_ctx* ctx, int vol, int lod, const raypc_camera* cam, int w, int h,
                          const raypc_render_opts* opts, float* out_rgba_dev,
                          unsigned long long* stats_dev, void* stream) {
    if (!ctx) return fail(RAYPC_ERR_INVALID_ARG, "NULL context");
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    Level* L = nullptr;
    if ((st = get_level(V, lod, &L))) return st;
    RenderArgs a{};
    if ((st = make_render_args(V, L, cam, w, h, opts, out_rgba_dev, stats_dev, &a))) return st;
    if ((st = ensure_classified(V, *L, (cudaStream_t)stream))) return st;
    if ((st = ensure_cell_classes(ctx, V, *L, (cudaStream_t)stream))) return st;
    a.cls = L->cls;
    if ((st = apply_tf_skip(V, *L, opts, a, (cudaStream_t)stream))) return st;
    if ((st = ensure_distance(ctx, V, *L, a, opts, (cudaStream_t)stream))) return st;
    CK(launch_render(a, V->dtype, (cudaStream_t)stream), "render kernel");
    return RAYPC_OK;
}

raypc_status raypc_render_progressive(raypc_ctx* ctx, int vol, int lod, const raypc_camera* cam, int w, int h,
                                      const raypc_render_opts* opts, uint32_t seed, uint32_t pass,
                                      float* accum_rgba_dev, float* out_rgba_dev,
                                      unsigned long long* stats_dev, void* stream) {
    if (!ctx) return fail(RAYPC_ERR_INVALID_ARG, "NULL context");
    if (pass == 0xFFFFFFFFu) return fail(RAYPC_ERR_INVALID_ARG, "pass index 2^32 - 1 out of range");
    if (((uintptr_t)accum_rgba_dev) & 15u) return fail(RAYPC_ERR_INVALID_ARG, "accum_rgba_dev must be 16-byte aligned");
    if (accum_rgba_dev && accum_rgba_dev == out_rgba_dev) return fail(RAYPC_ERR_INVALID_ARG, "accum_rgba_dev and out_rgba_dev alias");
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    Level* L = nullptr;
    if ((st = get_level(V, lod, &L))) return st;
    RenderArgs a{};
    if ((st = make_render_args(V, L, cam, w, h, opts, out_rgba_dev, stats_dev, &a))) return st;
    if ((st = ensure_classified(V, *L, (cudaStream_t)stream))) return st;
    if ((st = ensure_cell_classes(ctx, V, *L, (cudaStream_t)stream))) return st;
    a.cls = L->cls;
    a.jit_seed = seed;
    a.jit_pass = pass;
    a.accum = reinterpret_cast<float4*>(accum_rgba_dev);
    a.accum_w = 1.0f / (float)((double)pass + 1.0);
    if ((st = apply_tf_skip(V, *L, opts, a, (cudaStream_t)stream))) return st;
    if ((st = ensure_distance(ctx, V, *L, a, opts, (cudaStream_t)stream))) return st;
    CK(launch_render(a, V->dtype, (cudaStream_t)stream), "render kernel");
    return RAYPC_OK;
}

// PC axis ids: stored variables 0..nvars-1 and position axes RAYPC_AXIS_POS(0..3).
static raypc_status check_axes(const Volume* V, const int* axis_order, int naxes) {
    for (int a = 0; a < naxes; ++a) {
        const int id = axis_order[a];
        const bool ok = (id >= 0 && id < V->nvars) || (id >= kPosAxisBase && id < kPosAxisBase + kNumPos);
        if (!ok) return fail(RAYPC_ERR_INVALID_ARG, "axis %d names variable %d", a, id);
    }
    return RAYPC_OK;
}

raypc_status raypc_pc_histogram(raypc_ctx* ctx, int vol, int lod, const int* axis_order, int naxes,
                                int bins, const float* edges, int use_brush, uint32_t* out_counts_dev,
                                void* stream) {
    if (!ctx || !axis_order || !edges || !out_counts_dev) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    if (naxes < 2 || naxes > RAYPC_MAX_VARS) return fail(RAYPC_ERR_INVALID_ARG, "naxes %d not in 2..%d", naxes, RAYPC_MAX_VARS);
    if (bins < 2 || bins > 1024) return fail(RAYPC_ERR_INVALID_ARG, "bins %d not in 2..1024", bins);
    for (int a = 0; a < naxes; ++a)
        for (int k = 0; k <= bins; ++k) {
            float e = edges[(size_t)a * (bins + 1) + k];
            if (isnan(e)) return fail(RAYPC_ERR_INVALID_ARG, "NaN edge (axis %d, edge %d)", a, k);
            if (k && e < edges[(size_t)a * (bins + 1) + k - 1]) return fail(RAYPC_ERR_INVALID_ARG, "edges of axis %d decrease at %d", a, k);
        }
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    Level* L = nullptr;
    if ((st = get_level(V, lod, &L))) return st;
    if ((st = check_axes(V, axis_order, naxes))) return st;
    if (use_brush && !V->brush_set) return fail(RAYPC_ERR_INVALID_ARG, "use_brush needs raypc_set_brush");
    if (V->stale && lod > 0) return fail(RAYPC_ERR_INVALID_ARG, "level %d is stale after raypc_update_volume", lod);
    cudaStream_t s = (cudaStream_t)stream;
    // with the volume's brush, its sub-brick classification lets the kernel skip inactive sub-bricks
    const bool use_activity = use_brush && !V->stale;
    if (use_activity && (st = ensure_classified(V, *L, s))) return st;
    HistArgs h{};
    h.cells = L->cells;
    h.n = L->n;
    h.nvars = V->nvars;
    h.brush = V->brush;
    h.use_brush = use_brush ? 1 : 0;
    h.naxes = naxes;
    h.bins = bins;
    for (int a = 0; a < kMaxVars; ++a) h.axis[a] = a < naxes ? axis_order[a] : 0;
    for (int a = 0; a < naxes; ++a) {
        const float e0 = edges[(size_t)a * (bins + 1)], eN = edges[(size_t)a * (bins + 1) + bins];
        h.guess_e0[a] = e0;
        h.guess_scale[a] = (eN > e0 && isfinite(eN - e0)) ? (float)bins / (eN - e0) : 0.0f;
    }
    h.need_mask = use_brush ? V->brush.mask : 0u;
    for (int a = 0; a < naxes; ++a)
        if (axis_order[a] < kPosAxisBase) h.need_mask |= 1u << axis_order[a];
    double ri = (double)V->r_in * (double)L->n, ro = (double)V->r_out * (double)L->n;
    h.s_in = (int64_t)ceil(ri * ri);
    h.s_out = (int64_t)floor(ro * ro);
    // edges: in the launch parameters when the table is small, else a device copy owned by
    // this call (freed in stream order)
    const size_t ne = (size_t)naxes * (bins + 1);
    float* dedges = nullptr;
    cudaError_t e = cudaSuccess;
    h.edges_host = edges;
    if (ne > (size_t)kHistInlineEdges) {
        CK(ctx->scratch((void**)&dedges, sizeof(float) * ne, s), "edge buffer");
        e = cudaMemcpyAsync(dedges, edges, sizeof(float) * ne, cudaMemcpyHostToDevice, s);
    }
    // large grids list the cells' bins in stream-ordered scratch and count them in shared memory;
    // without room for that (or with more bins than fit there) the blocks spread their atomics over
    // zeroed copies, summed into the output afterwards (which then needs no clearing), and the
    // same scratch holds the row counter that balances the warps
    const size_t count = (size_t)(naxes - 1) * bins * bins;
    h.edges = dedges;
    h.out = out_counts_dev;
    h.sactive = use_activity ? L->sactive : nullptr;
    h.nsb = L->nsb;
    if (e == cudaSuccess && hist_by_list(h)) h.list = ctx->spare_scratch(hist_list(h).bytes, s);
    const int ncopies = h.list || ((uintptr_t)out_counts_dev & 15u) ? 1 : hist_copies(L->n, naxes, bins);
    const size_t copy_bytes = sizeof(uint32_t) * (count * ncopies + 4);
    uint32_t* copies = nullptr;
    if (e == cudaSuccess && ncopies > 1) {
        e = ctx->scratch((void**)&copies, copy_bytes, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(copies, 0, copy_bytes, s);
    } else if (e == cudaSuccess) {
        e = cudaMemsetAsync(out_counts_dev, 0, sizeof(uint32_t) * count, s);
    }
    if (e == cudaSuccess) {
        h.copies = copies;
        h.ncopies = copies ? ncopies : 1;
        h.rowctr = copies ? copies + count * ncopies : nullptr;
        e = launch_histogram(h, V->dtype, s);
        if (e == cudaSuccess && copies) e = launch_histogram_reduce(copies, ncopies, count, out_counts_dev, s);
    }
    if (h.list) cudaFreeAsync(h.list, s);
    if (copies) cudaFreeAsync(copies, s);
    if (dedges) cudaFreeAsync(dedges, s);
    if (e != cudaSuccess) return cuda_fail(e, "histogram");
    return RAYPC_OK;
}

raypc_status raypc_pc_subsample(raypc_ctx* ctx, int vol, int lod, uint32_t seed, long long k,
                                const int* axis_order, int naxes, long long* out_cells_dev,
                                float* out_values_dev, uint8_t* out_in_brush_dev, long long* out_count,
                                void* stream) {
    if (!ctx || !out_count) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    if (k < 0 || k > 0x7fffffffLL) return fail(RAYPC_ERR_INVALID_ARG, "k %lld not in 0..2^31-1", k);
    if (naxes < 0 || naxes > RAYPC_MAX_VARS) return fail(RAYPC_ERR_INVALID_ARG, "naxes %d not in 0..%d", naxes, RAYPC_MAX_VARS);
    if (naxes > 0 && !axis_order) return fail(RAYPC_ERR_INVALID_ARG, "NULL axis_order");
    if (k > 0 && (!out_cells_dev || !out_in_brush_dev || (naxes > 0 && !out_values_dev)))
        return fail(RAYPC_ERR_INVALID_ARG, "NULL output");
    if (((uintptr_t)out_cells_dev) & 7u) return fail(RAYPC_ERR_INVALID_ARG, "out_cells_dev must be 8-byte aligned");
    if (((uintptr_t)out_values_dev) & 3u) return fail(RAYPC_ERR_INVALID_ARG, "out_values_dev must be 4-byte aligned");
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    Level* L = nullptr;
    if ((st = get_level(V, lod, &L))) return st;
    if ((st = check_axes(V, axis_order, naxes))) return st;
    if (V->stale && lod > 0) return fail(RAYPC_ERR_INVALID_ARG, "level %d is stale after raypc_update_volume", lod);
    const double ri = (double)V->r_in * (double)L->n, ro = (double)V->r_out * (double)L->n;
    const int64_t s_in = (int64_t)ceil(ri * ri), s_out = (int64_t)floor(ro * ro);
    const unsigned long long N = s_out < 0 ? 0ull : count_in_shell(L->n, s_in, s_out);
    const unsigned long long m = std::min<unsigned long long>((unsigned long long)k, N);
    *out_count = (long long)m;
    if (m == 0) return RAYPC_OK;
    SubsampleArgs a{};
    a.cells = L->cells;
    a.n = L->n;
    a.nvars = V->nvars;
    const int64_t imax = 0x7fffffff;
    a.s_in = (int)std::min<int64_t>(std::max<int64_t>(s_in, 0), imax);
    a.s_out = (int)std::min<int64_t>(s_out, imax);
    a.key = ((unsigned long long)seed << 32) | 0xFFFFFFFFull;
    if (V->brush_set) {
        a.brush = V->brush;
    } else {
        for (int v = 0; v < kMaxVars; ++v) { a.brush.lo[v] = -INFINITY; a.brush.hi[v] = INFINITY; }
        for (int p = 0; p < kNumPos; ++p) { a.brush.plo[p] = -INFINITY; a.brush.phi[p] = INFINITY; }
    }
    a.naxes = naxes;
    for (int i = 0; i < naxes; ++i) {
        a.axis[i] = axis_order[i];
        if (axis_order[i] >= kPosAxisBase) a.use_pos = 1;
    }
    if (a.brush.pmask) a.use_pos = 1;
    a.m = m;
    a.out_cells = out_cells_dev;
    a.out_values = out_values_dev;
    a.out_flags = out_in_brush_dev;
    cudaStream_t s = (cudaStream_t)stream;
    // select state and per-block counts: a small device buffer owned by this call (freed in stream order)
    void* scratch = nullptr;
    CK(ctx->scratch(&scratch, pc_subsample_scratch_bytes(), s), "subsample scratch");
    cudaError_t e = launch_pc_subsample(a, V->dtype, m, N, scratch, s);
    cudaFreeAsync(scratch, s);
    if (e != cudaSuccess) return cuda_fail(e, "pc subsample");
    return RAYPC_OK;
}

raypc_status raypc_filter_points(raypc_ctx* ctx, int vol, int lod, const float* points_dev, long long npts,
                                 uint8_t* out_pass_dev, void* stream) {
    if (!ctx) return fail(RAYPC_ERR_INVALID_ARG, "NULL context");
    if (npts < 0) return fail(RAYPC_ERR_INVALID_ARG, "npts %lld < 0", npts);
    if (npts > 0 && (!points_dev || !out_pass_dev)) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    if (((uintptr_t)points_dev) & 3u) return fail(RAYPC_ERR_INVALID_ARG, "points_dev must be 4-byte aligned");
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    Level* L = nullptr;
    if ((st = get_level(V, lod, &L))) return st;
    if (V->stale && lod > 0) return fail(RAYPC_ERR_INVALID_ARG, "level %d is stale after raypc_update_volume", lod);
    RenderArgs r{};                       // the brush and the per-sample |p|^2 range of a render
    if (V->brush_set) {
        r.brush = V->brush;
    } else {
        for (int v = 0; v < kMaxVars; ++v) { r.brush.lo[v] = -INFINITY; r.brush.hi[v] = INFINITY; }
        for (int p = 0; p < kNumPos; ++p) { r.brush.plo[p] = -INFINITY; r.brush.phi[p] = INFINITY; }
    }
    r.rin2 = V->r_in * V->r_in;
    r.rout2 = V->r_out * V->r_out;
    finish_position_brush(r);
    PointFilterArgs a{};
    a.pairs = L->pairs;
    a.n = L->n;
    a.nvars = V->nvars;
    a.brush = r.brush;
    a.keep_lo2 = r.keep_lo2;
    a.keep_hi2 = r.keep_hi2;
    a.pts = points_dev;
    a.npts = npts;
    a.out = out_pass_dev;
    CK(launch_filter_points(a, V->dtype, (cudaStream_t)stream), "point filter kernel");
    return RAYPC_OK;
}

static raypc_status check_camera(const raypc_camera* cam) {
    if (!cam) return fail(RAYPC_ERR_INVALID_ARG, "NULL camera");
    for (int i = 0; i < 3; ++i)
        if (!isfinite(cam->eye[i]) || !isfinite(cam->target[i]) || !isfinite(cam->up[i]))
            return fail(RAYPC_ERR_INVALID_ARG, "non-finite camera");
    if (!(cam->tan_half_vfov > 0.f) || !isfinite(cam->tan_half_vfov)) return fail(RAYPC_ERR_INVALID_ARG, "tan_half_vfov must be > 0");
    float fx = cam->target[0] - cam->eye[0], fy = cam->target[1] - cam->eye[1], fz = cam->target[2] - cam->eye[2];
    if (fx == 0.f && fy == 0.f && fz == 0.f) return fail(RAYPC_ERR_INVALID_ARG, "eye == target");
    float cx = fy * cam->up[2] - fz * cam->up[1], cy = fz * cam->up[0] - fx * cam->up[2], cz = fx * cam->up[1] - fy * cam->up[0];
    if (cx == 0.f && cy == 0.f && cz == 0.f) return fail(RAYPC_ERR_INVALID_ARG, "up is parallel to the view direction");
    return RAYPC_OK;
}

raypc_status raypc_warp_image(raypc_ctx* ctx, const raypc_camera* from, const raypc_camera* to, int w, int h,
                              const float* src_rgba_dev, const float* src_depth_dev, const float* bg,
                              int fill_holes, float* out_rgba_dev, int32_t* out_src_dev, void* stream) {
    if (!ctx || !src_rgba_dev || !src_depth_dev || !out_rgba_dev) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    raypc_status st;
    if ((st = check_camera(from)) || (st = check_camera(to))) return st;
    if (w < 1 || h < 1 || w > 32768 || h > 32768) return fail(RAYPC_ERR_INVALID_ARG, "image size %d x %d out of range", w, h);
    if ((((uintptr_t)src_rgba_dev) | ((uintptr_t)out_rgba_dev)) & 15u)
        return fail(RAYPC_ERR_INVALID_ARG, "src_rgba_dev and out_rgba_dev must be 16-byte aligned");
    if (((uintptr_t)src_depth_dev) & 3u || ((uintptr_t)out_src_dev) & 3u) return fail(RAYPC_ERR_INVALID_ARG, "misaligned depth or source index buffer");
    if (src_rgba_dev == out_rgba_dev) return fail(RAYPC_ERR_INVALID_ARG, "out_rgba_dev must not alias src_rgba_dev");
    WarpArgs a{};
    for (int i = 0; i < 3; ++i) {
        a.from_eye[i] = from->eye[i]; a.from_target[i] = from->target[i]; a.from_up[i] = from->up[i];
        a.to_eye[i] = to->eye[i]; a.to_target[i] = to->target[i]; a.to_up[i] = to->up[i];
    }
    a.from_tan_half = from->tan_half_vfov;
    a.to_tan_half = to->tan_half_vfov;
    a.w = w;
    a.h = h;
    a.src_rgba = reinterpret_cast<const float4*>(src_rgba_dev);
    a.src_depth = src_depth_dev;
    for (int c = 0; c < 4; ++c) {
        a.bg[c] = bg ? bg[c] : 0.0f;
        if (!isfinite(a.bg[c])) return fail(RAYPC_ERR_INVALID_ARG, "non-finite background");
    }
    a.out = reinterpret_cast<float4*>(out_rgba_dev);
    a.out_src = out_src_dev;
    a.fill_holes = fill_holes ? 1 : 0;
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    // per-pixel selection keys: a device buffer owned by this call (freed in stream order)
    CK(ctx->scratch((void**)&a.keys, sizeof(unsigned long long) * (size_t)w * h, s), "warp keys");
    cudaError_t e = launch_warp(a, s);
    cudaFreeAsync(a.keys, s);
    if (e != cudaSuccess) return cuda_fail(e, "warp kernels");
    return RAYPC_OK;
}

raypc_status raypc_volume_info(raypc_ctx* ctx, int vol, int lod, int* out_n, int* out_nvars,
                               int* out_dtype, int* out_bricks_per_axis) {
    if (!ctx) return fail(RAYPC_ERR_INVALID_ARG, "NULL context");
    std::lock_guard<std::mutex> lk(ctx->mu);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    Level* L = nullptr;
    if ((st = get_level(V, lod, &L))) return st;
    if (out_n) *out_n = L->n;
    if (out_nvars) *out_nvars = V->nvars;
    if (out_dtype) *out_dtype = V->dtype;
    if (out_bricks_per_axis) *out_bricks_per_axis = L->nb;
    return RAYPC_OK;
}

raypc_status raypc_export_volume(raypc_ctx* ctx, int vol, int lod, void* out_dev, void* stream) {
    if (!ctx || !out_dev) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    Level* L = nullptr;
    if ((st = get_level(V, lod, &L))) return st;
    CK(cudaMemcpyAsync(out_dev, L->cells, L->cells_bytes, cudaMemcpyDeviceToDevice, (cudaStream_t)stream),
       "export copy");
    return RAYPC_OK;
}

raypc_status raypc_get_bricks(raypc_ctx* ctx, int vol, int lod, float* out_min_dev, float* out_max_dev,
                              void* stream) {
    if (!ctx || !out_min_dev || !out_max_dev) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    Level* L = nullptr;
    if ((st = get_level(V, lod, &L))) return st;
    if (!L->bricks) return fail(RAYPC_ERR_INVALID_ARG, "bricks of level %d not built", lod);
    size_t bytes = L->nbricks() * V->nvars * sizeof(float);
    cudaStream_t s = (cudaStream_t)stream;
    CK(cudaMemcpyAsync(out_min_dev, L->bmin, bytes, cudaMemcpyDeviceToDevice, s), "copy brick min");
    CK(cudaMemcpyAsync(out_max_dev, L->bmax, bytes, cudaMemcpyDeviceToDevice, s), "copy brick max");
    return RAYPC_OK;
}

raypc_status raypc_get_skip_list(raypc_ctx* ctx, int vol, int lod, uint32_t* active_bits_dev,
                                 uint32_t* skippable_bits_dev, uint32_t* active_list_dev,
                                 uint32_t* n_active_dev, void* stream) {
    if (!ctx) return fail(RAYPC_ERR_INVALID_ARG, "NULL context");
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    Level* L = nullptr;
    if ((st = get_level(V, lod, &L))) return st;
    cudaStream_t s = (cudaStream_t)stream;
    if (V->stale) return fail(RAYPC_ERR_INVALID_ARG, "volume updated: raypc_build_bricks must run first");
    if ((st = ensure_classified(V, *L, s))) return st;
    // by every call, in its own stream's order: a list kept from one call could be read before the
    // stream that computes it gets there
    BrickListArgs b{};
    b.bmin = L->bmin;
    b.bmax = L->bmax;
    b.n = L->n;
    b.nb = L->nb;
    b.nvars = V->nvars;
    b.rin2 = V->r_in * V->r_in;
    b.rout2 = V->r_out * V->r_out;
    b.brush = V->brush;
    b.active = L->active;
    b.skippable = L->skippable;
    b.list = L->list;
    b.n_active = L->n_active;
    CK(launch_brick_list(b, s), "brick list kernels");
    size_t wb = L->nwords() * sizeof(uint32_t);
    if (active_bits_dev) CK(cudaMemcpyAsync(active_bits_dev, L->active, wb, cudaMemcpyDeviceToDevice, s), "copy active bits");
    if (skippable_bits_dev) CK(cudaMemcpyAsync(skippable_bits_dev, L->skippable, wb, cudaMemcpyDeviceToDevice, s), "copy skippable bits");
    if (active_list_dev) CK(cudaMemcpyAsync(active_list_dev, L->list, L->nbricks() * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s), "copy active list");
    if (n_active_dev) CK(cudaMemcpyAsync(n_active_dev, L->n_active, sizeof(uint32_t), cudaMemcpyDeviceToDevice, s), "copy active count");
    return RAYPC_OK;
}

raypc_status raypc_get_cell_classes(raypc_ctx* ctx, int vol, int lod, uint16_t* out_dev, void* stream) {
    if (!ctx || !out_dev) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    Level* L = nullptr;
    if ((st = get_level(V, lod, &L))) return st;
    if (V->stale) return fail(RAYPC_ERR_INVALID_ARG, "volume updated: raypc_build_bricks must run first");
    cudaStream_t s = (cudaStream_t)stream;
    if ((st = ensure_cell_classes(ctx, V, *L, s))) return st;
    CK(cudaMemcpyAsync(out_dev, L->cls, (size_t)L->n * L->n * L->n * sizeof(uint16_t), cudaMemcpyDeviceToDevice, s),
       "copy cell classes");
    return RAYPC_OK;
}

raypc_status raypc_get_skip_distance(raypc_ctx* ctx, int vol, int lod, uint8_t* out_dev, void* stream) {
    if (!ctx || !out_dev) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    Level* L = nullptr;
    if ((st = get_level(V, lod, &L))) return st;
    if (V->stale) return fail(RAYPC_ERR_INVALID_ARG, "volume updated: raypc_build_bricks must run first");
    cudaStream_t s = (cudaStream_t)stream;
    if ((st = ensure_classified(V, *L, s))) return st;
    CK(launch_subbrick_distance(L->sactive, L->n, out_dev, true, s), "empty-space distance");
    return RAYPC_OK;
}

raypc_status raypc_get_sub_bricks(raypc_ctx* ctx, int vol, int lod, float* out_min_dev, float* out_max_dev,
                                  uint32_t* active_bits_dev, void* stream) {
    if (!ctx) return fail(RAYPC_ERR_INVALID_ARG, "NULL context");
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    Volume* V = nullptr;
    raypc_status st = get_volume(ctx, vol, &V);
    if (st) return st;
    Level* L = nullptr;
    if ((st = get_level(V, lod, &L))) return st;
    if (!L->bricks) return fail(RAYPC_ERR_INVALID_ARG, "bricks of level %d not built", lod);
    cudaStream_t s = (cudaStream_t)stream;
    const size_t bytes = L->nsbricks() * V->nvars * sizeof(float);
    if (out_min_dev) CK(cudaMemcpyAsync(out_min_dev, L->sbmin, bytes, cudaMemcpyDeviceToDevice, s), "copy sub-brick min");
    if (out_max_dev) CK(cudaMemcpyAsync(out_max_dev, L->sbmax, bytes, cudaMemcpyDeviceToDevice, s), "copy sub-brick max");
    if (active_bits_dev) {
        if (V->stale) return fail(RAYPC_ERR_INVALID_ARG, "volume updated: raypc_build_bricks must run first");
        if ((st = ensure_classified(V, *L, s))) return st;
        CK(cudaMemcpyAsync(active_bits_dev, L->sactive, L->nswords() * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s),
           "copy sub-brick active bits");
    }
    return RAYPC_OK;
}

}  // extern "C"
