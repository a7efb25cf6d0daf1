// Internal host-runtime types shared by the C-ABI translation units
// (contexts, resident volumes and their levels, error reporting). Not part of
// the public interface; include/raypc.h is.
#pragma once

#include <stdarg.h>
#include <stdio.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <string>

#include "common.cuh"
#include "raypc.h"

namespace raypc {

// Error reporting: the message of the last failing call on this thread.
raypc_status fail(raypc_status code, const char* fmt, ...);
raypc_status cuda_fail(cudaError_t e, const char* what);
void set_last_error(const char* msg);

#define CK(call, what)                                       \
    do {                                                     \
        cudaError_t e_ = (call);                             \
        if (e_ != cudaSuccess) return raypc::cuda_fail(e_, what); \
    } while (0)

// Selects a device for the lifetime of the guard and restores the previous one.
struct DeviceGuard {
    int prev = -1;
    bool ok = false;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) return;
        if (prev != dev && cudaSetDevice(dev) != cudaSuccess) return;
        ok = true;
    }
    ~DeviceGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

struct Level {
    int n = 0, nb = 0, nsb = 0;   // edge, 8^3 bricks per axis, 4^3 sub-bricks per axis
    void* cells = nullptr;     // planar values, storage dtype
    void* pairs = nullptr;     // per-variable x-pairs (render layout)
    size_t cells_bytes = 0, pairs_bytes = 0;
    float* bmin = nullptr;
    float* bmax = nullptr;
    uint32_t* active = nullptr;
    uint32_t* skippable = nullptr;
    uint32_t* list = nullptr;
    uint32_t* n_active = nullptr;
    LevelStats stats{};           // of the stored values; mag is the volume's
    float* sbmin = nullptr;       // [nsb^3][nvars]
    float* sbmax = nullptr;
    uint32_t* sactive = nullptr;  // sub-brick activity bits under the current brush
    uint16_t* cls = nullptr;      // cell classes under the current brush (n^3), computed on demand
    uint32_t* tf_sactive = nullptr;  // activity AND TF visibility (renders with tf_skip)
    uint8_t* sdist = nullptr;        // padded empty-space distance of the sub-bricks (renders)
    uint8_t* tf_sdist = nullptr;     // the same under tf_sactive
    const uint32_t* sdist_of = nullptr;   // activity bits that sdist was computed from (null: stale)
    bool cls_valid = false;
    bool bricks = false;
    bool classified = false;      // sactive is current
    bool fresh = false;           // cells and pairs written by the last ingest of the finer level,
                                  // brick min/max not yet (raypc_build_bricks computes them)
    size_t nbricks() const { return (size_t)nb * nb * nb; }
    size_t nwords() const { return (nbricks() + 31) / 32; }
    size_t nsbricks() const { return (size_t)nsb * nsb * nsb; }
    size_t nswords() const { return (nsbricks() + 31) / 32; }
    void set_edge(int edge) {
        n = edge;
        nb = (edge + kBrick - 1) / kBrick;
        nsb = (edge + kSub - 1) / kSub;
    }
};

struct Volume {
    int nvars = 0, dtype = 0;
    bool stale = false;       // level 0 updated since the last build_bricks
    float r_in = 0.f, r_out = 1.f;
    int nlev = 0;             // built levels (1 + coarser)
    Level lv[1 + RAYPC_MAX_LOD];
    unsigned* mags = nullptr;     // the levels' magnitudes, one after another
    bool brush_set = false;
    BrushArgs brush{};
    float4* tf = nullptr;
    int* tf_prefix = nullptr;     // [257]: TF entries < j with sigma > 0 (TF-aware skipping)
    bool tf_set = false;
    int color_var = 0;
    float tf_lo = 0.f, tf_hi = 1.f;
    size_t bytes = 0;
    // host-source updates: two staging buffers of the source's size used in turn, filled on a
    // copy stream of the volume's own; ev_consumed[i] marks the last ingest that read buffer i
    void* staging[2] = {nullptr, nullptr};
    size_t staging_bytes = 0;
    int stage_next = 0;
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t ev_copied = nullptr, ev_consumed[2] = {nullptr, nullptr};
    bool consumed_pending[2] = {false, false};
};

inline size_t elem_size(int dtype) { return dtype == RAYPC_F16 ? 2 : 4; }

raypc_status get_volume(raypc_ctx* ctx, int vol, Volume** out);
raypc_status get_level(Volume* V, int lod, Level** out);

// The contexts' scratch pools. trim_pools gives back what those of a device keep (with wait,
// after the work in flight); false when they keep nothing.
void pool_opened(int device, cudaMemPool_t pool);
void pool_closed(cudaMemPool_t pool);
bool trim_pools(int device, bool wait);

// An allocation (f() -> cudaError_t) that the idle memory of the device's scratch pools must not
// make fail: tried again without it.
template <typename F>
cudaError_t allocate(int device, F f) {
    cudaError_t e = f();
    for (int wait = 0; e == cudaErrorMemoryAllocation && wait < 2; ++wait) {
        cudaGetLastError();
        if (!trim_pools(device, wait != 0)) break;
        e = f();
    }
    return e;
}

// Fill the march arguments of one render of level L of volume V (brush and
// classification taken from V / L; callers may override them).
raypc_status make_render_args(Volume* V, Level* L, const raypc_camera* cam, int w, int h,
                              const raypc_render_opts* opts, float* out_rgba_dev,
                              unsigned long long* stats_dev, RenderArgs* a);

// The classification of level L of volume V under a brush, without outputs.
BrushItem brush_item(const Volume* V, const Level& L, const BrushArgs& brush);

// Resolve RAYPC_AUTO launch choices from the tuning table (tune.cu).
void resolve_launch(int device, int dtype, int n, int* variant, int* skip);

// Completion records of a batch's most recent launch: *records points at the
// mapped host array indexed like the launch's views, *seq is the value a
// record's seq field takes when that view is finished (see ViewDone).
void batch_last_records(raypc_batch* b, const ViewDone** records, unsigned* seq);

// Compute the cell classes of level L under the volume's brush if they are
// not current (allocates them on first use).
raypc_status ensure_cell_classes(raypc_ctx* ctx, Volume* V, Level& L, cudaStream_t s);

// Validated brush box of a volume from host arrays (nvars entries each); no position brush.
raypc_status brush_from_host(const Volume* V, const float* lo, const float* hi, uint32_t active_mask, BrushArgs* out);

// Validated position brush (axes x, y, z, radius; bounds read only for axes in pos_mask) into b.
raypc_status pos_from_host(const float* lo, const float* hi, uint32_t pos_mask, BrushArgs* b);

// Per-sample |p|^2 range of a render (keep_lo2, keep_hi2) from its shell radii and the radius
// brush; call after the brush is final.
void finish_position_brush(RenderArgs& a);

}  // namespace raypc

struct raypc_ctx {
    int device = 0;
    size_t budget = 0;
    size_t used = 0;
    std::mutex mu;
    std::map<int, raypc::Volume*> vols;
    int next_id = 1;

    // Stream-ordered scratch of single calls, from a pool of the context's own that keeps up to
    // kScratchKept bytes between calls (the device's default pool gives everything back at each
    // synchronisation, and the next call maps its scratch anew). Safe on any stream; freed with
    // cudaFreeAsync on the stream that used it. Without a pool it comes from the default one.
    // What the pool holds counts as memory used, and is given back when any context of the device
    // needs it. At 512^3 FP16 a listed whole-shell histogram takes 1.20 ms when it maps its 540 MB
    // and 0.53 ms when the pool holds them.
    cudaMemPool_t pool = nullptr;
    static constexpr unsigned long long kScratchKept = 640ull << 20;
    void open_pool() {
        cudaMemPoolProps props{};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = device;
        unsigned long long keep = kScratchKept;
        if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
            pool = nullptr;
            cudaGetLastError();
            return;
        }
        raypc::pool_opened(device, pool);
        if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) cudaGetLastError();
    }
    size_t pool_bytes(cudaMemPoolAttr what) const {
        unsigned long long v = 0;
        if (pool && cudaMemPoolGetAttribute(pool, what, &v) != cudaSuccess) cudaGetLastError();
        return (size_t)v;
    }
    size_t pool_held() const { return pool_bytes(cudaMemPoolAttrReservedMemCurrent); }
    cudaError_t scratch(void** p, size_t bytes, cudaStream_t s) {
        return raypc::allocate(device, [&] { return pool ? cudaMallocFromPoolAsync(p, bytes, pool, s) : cudaMallocAsync(p, bytes, s); });
    }
    // Scratch that a call can do without (null: none), within the budget when there is one.
    void* spare_scratch(size_t bytes, cudaStream_t s) {
        void* p = nullptr;
        if (budget && used + std::max(pool_held(), pool_bytes(cudaMemPoolAttrUsedMemCurrent) + bytes) > budget) return nullptr;
        if ((pool ? cudaMallocFromPoolAsync(&p, bytes, pool, s) : cudaMallocAsync(&p, bytes, s)) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        if (budget && used + pool_held() > budget) {        // other streams' scratch is not free yet
            cudaFreeAsync(p, s);
            return nullptr;
        }
        return p;
    }

    // Device allocation charged against the budget.
    raypc_status alloc(void** p, size_t bytes, size_t* charged) {
        if (budget && used + bytes > budget)
            return raypc::fail(RAYPC_ERR_OOM, "HBM budget exceeded: %zu used + %zu requested > %zu", used, bytes, budget);
        if (budget && used + pool_held() + bytes > budget) cudaMemPoolTrimTo(pool, 0);   // idle scratch makes way
        const cudaError_t e = raypc::allocate(device, [&] { return cudaMalloc(p, bytes ? bytes : 16); });
        if (e != cudaSuccess) return raypc::cuda_fail(e, "cudaMalloc");
        used += bytes;
        *charged += bytes;
        return RAYPC_OK;
    }
};
