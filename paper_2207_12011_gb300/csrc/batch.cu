// Batched rendering: many views (each with its own camera, image size and
// brush box) in one CUDA graph, captured once and replayed with new view
// tables and render parameters.
//
// Per batch the host fills a view table (double-buffered in pinned memory);
// the graph uploads it, zeroes the per-view counters, classifies every view's
// sub-bricks and cells under that view's brush into the view's own buffers, and
// renders the views in nodes side by side, so that the blocks of the next views
// fill the GPU while the last blocks of one finish. The table's address never
// changes; the render nodes' kernels, grids and parameters are set on the
// instantiated graph before each replay, and the nodes beyond the batch's views
// are switched off. A graph is captured per table buffer and storage dtype, with
// a power of two of render nodes.
#include <vector>

#include "runtime.h"

using namespace raypc;

struct raypc_batch {
    raypc_ctx* ctx = nullptr;
    int max_views = 0;
    size_t table_bytes = 0;
    char* d_table = nullptr;          // BatchHeader, then max_views BrushItem (device)
    unsigned* d_tiles = nullptr;      // max_views finished-tile counters
    ViewDone* h_done[2] = {nullptr, nullptr};   // mapped pinned completion records per table slot
    ViewDone* d_done[2] = {nullptr, nullptr};   // their device aliases
    unsigned seq = 0;                 // launch sequence number
    int last_slot = 0;
    char* h_table[2] = {nullptr, nullptr};   // pinned host copies of the table
    cudaEvent_t done[2] = {nullptr, nullptr};
    bool used[2] = {false, false};
    int cur = 0;
    std::vector<uint32_t*> bits;      // per view slot: sub-brick active words, padded distance grid
    std::vector<size_t> bits_words;   // capacity (words) per slot
    std::vector<uint16_t*> cls;       // per view slot: cell classes under the view's brush (n^3 words)
    std::vector<size_t> cls_cells;    // capacity (cells) per slot
    cudaStream_t cap_stream = nullptr;
    cudaGraphExec_t exec[2] = {nullptr, nullptr};
    int exec_dtype[2] = {-1, -1};     // storage dtype of the captured graph
    cudaGraph_t graph[2] = {nullptr, nullptr};   // the captured graph (kept: it owns the node handles)
    std::vector<cudaGraphNode_t> nodes[2];   // its render nodes, the first `enabled` of them switched on
    int enabled[2] = {0, 0};
    std::vector<ViewLaunch> launch;   // their parameters, as filled for a call
    size_t charged = 0;
};

namespace {

constexpr size_t kHeaderBytes = 256;   // BatchHeader padded so the views start aligned

BatchHeader* hdr_of(char* table) { return reinterpret_cast<BatchHeader*>(table); }
BrushItem* views_of(char* table) { return reinterpret_cast<BrushItem*>(table + kHeaderBytes); }

void wait_idle(raypc_batch* b) {
    for (int i = 0; i < 2; ++i)
        if (b->used[i]) cudaEventSynchronize(b->done[i]);
}

void release(raypc_batch* b) {
    wait_idle(b);
    for (int i = 0; i < 2; ++i) {
        if (b->exec[i]) cudaGraphExecDestroy(b->exec[i]);
        if (b->graph[i]) cudaGraphDestroy(b->graph[i]);
        if (b->h_table[i]) cudaFreeHost(b->h_table[i]);
        if (b->h_done[i]) cudaFreeHost(b->h_done[i]);
        if (b->done[i]) cudaEventDestroy(b->done[i]);
    }
    for (uint32_t* p : b->bits)
        if (p) cudaFree(p);
    for (uint16_t* p : b->cls)
        if (p) cudaFree(p);
    if (b->d_table) cudaFree(b->d_table);
    if (b->d_tiles) cudaFree(b->d_tiles);
    if (b->cap_stream) cudaStreamDestroy(b->cap_stream);
    if (b->ctx) b->ctx->used -= b->charged < b->ctx->used ? b->charged : b->ctx->used;
}

raypc_status capture(raypc_batch* b, int slot, int dtype) {
    int dev = 0, sms = 0;
    CK(cudaGetDevice(&dev), "cudaGetDevice");
    CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "SM count");
    const unsigned blocks = (unsigned)sms * 8u;
    if (b->exec[slot]) {
        cudaGraphExecDestroy(b->exec[slot]);
        b->exec[slot] = nullptr;
    }
    if (b->graph[slot]) {
        cudaGraphDestroy(b->graph[slot]);
        b->graph[slot] = nullptr;
    }
    b->nodes[slot].clear();
    cudaStream_t s = b->cap_stream;
    CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal), "begin graph capture");
    cudaError_t e = cudaMemcpyAsync(b->d_table, b->h_table[slot], b->table_bytes, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(b->d_tiles, 0, sizeof(unsigned) * b->max_views, s);
    if (e == cudaSuccess) e = launch_brush_views(hdr_of(b->d_table), views_of(b->d_table), dtype, s);
    if (e == cudaSuccess) e = launch_subbrick_distance_views(hdr_of(b->d_table), views_of(b->d_table), blocks, s);
    cudaGraph_t graph = nullptr;
    cudaError_t e2 = cudaStreamEndCapture(s, &graph);
    if (e == cudaSuccess) e = e2;
    // the render nodes follow the last captured launch, side by side
    cudaGraphNode_t last = nullptr;
    if (e == cudaSuccess) {
        size_t n = 0;
        e = cudaGraphGetNodes(graph, nullptr, &n);
        std::vector<cudaGraphNode_t> all(n);
        if (e == cudaSuccess) e = cudaGraphGetNodes(graph, all.data(), &n);
        for (size_t i = 0; i < n && e == cudaSuccess && !last; ++i) {
            size_t after = 0;
            e = cudaGraphNodeGetDependentNodes(all[i], nullptr, nullptr, &after);
            if (e == cudaSuccess && after == 0) last = all[i];
        }
    }
    size_t count = 1;
    while (count < b->launch.size()) count *= 2;
    for (size_t i = 0; i < count && e == cudaSuccess; ++i) {
        const cudaKernelNodeParams p = render_view_node(b->launch[i < b->launch.size() ? i : 0], dtype);
        cudaGraphNode_t node = nullptr;
        e = cudaGraphAddKernelNode(&node, graph, &last, 1, &p);
        b->nodes[slot].push_back(node);
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec[slot], graph, 0);
    b->graph[slot] = graph;
    if (e != cudaSuccess) return cuda_fail(e, "batch graph capture");
    b->exec_dtype[slot] = dtype;
    b->enabled[slot] = (int)count;
    return RAYPC_OK;
}

}  // namespace

void raypc::batch_last_records(raypc_batch* b, const ViewDone** records, unsigned* seq) {
    *records = b->h_done[b->last_slot];
    *seq = b->seq;
}

extern "C" {

raypc_status raypc_batch_create(raypc_ctx* ctx, int max_views, raypc_batch** out) {
    if (!ctx || !out) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    if (max_views < 1 || max_views > 4096) return fail(RAYPC_ERR_INVALID_ARG, "max_views %d not in 1..4096", max_views);
    *out = nullptr;
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    raypc_batch* b = new raypc_batch();
    b->ctx = ctx;
    b->max_views = max_views;
    b->table_bytes = kHeaderBytes + sizeof(BrushItem) * (size_t)max_views;
    b->bits.assign(max_views, nullptr);
    b->bits_words.assign(max_views, 0);
    b->cls.assign(max_views, nullptr);
    b->cls_cells.assign(max_views, 0);
    raypc_status st = ctx->alloc((void**)&b->d_table, b->table_bytes, &b->charged);
    if (st == RAYPC_OK) st = ctx->alloc((void**)&b->d_tiles, sizeof(unsigned) * max_views, &b->charged);
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 2 && st == RAYPC_OK && e == cudaSuccess; ++i) {
        e = cudaHostAlloc((void**)&b->h_table[i], b->table_bytes, cudaHostAllocDefault);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->done[i], cudaEventDisableTiming);
        if (e == cudaSuccess) memset(b->h_table[i], 0, b->table_bytes);
        if (e == cudaSuccess) e = cudaHostAlloc((void**)&b->h_done[i], sizeof(ViewDone) * max_views, cudaHostAllocMapped);
        if (e == cudaSuccess) {
            memset((void*)b->h_done[i], 0, sizeof(ViewDone) * max_views);
            e = cudaHostGetDevicePointer((void**)&b->d_done[i], b->h_done[i], 0);
        }
    }
    if (st == RAYPC_OK && e == cudaSuccess) e = cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking);
    if (st == RAYPC_OK && e != cudaSuccess) st = cuda_fail(e, "batch resources");
    if (st != RAYPC_OK) {
        release(b);
        delete b;
        return st;
    }
    *out = b;
    return RAYPC_OK;
}

raypc_status raypc_batch_destroy(raypc_batch* b) {
    if (!b) return RAYPC_OK;
    {
        std::lock_guard<std::mutex> lk(b->ctx->mu);
        DeviceGuard g(b->ctx->device);
        release(b);
    }
    delete b;
    return RAYPC_OK;
}

raypc_status raypc_render_batch(raypc_batch* b, const raypc_view* views, int nviews, void* stream) {
    if (!b || !views) return fail(RAYPC_ERR_INVALID_ARG, "NULL argument");
    if (nviews < 1 || nviews > b->max_views) return fail(RAYPC_ERR_INVALID_ARG, "nviews %d not in 1..%d", nviews, b->max_views);
    raypc_ctx* ctx = b->ctx;
    std::lock_guard<std::mutex> lk(ctx->mu);
    DeviceGuard g(ctx->device);
    const int slot = b->cur;
    // the table buffer of this slot was last read by the batch two calls ago
    if (b->used[slot]) CK(cudaEventSynchronize(b->done[slot]), "wait for the previous use of the view table");
    BatchHeader* H = hdr_of(b->h_table[slot]);
    BrushItem* T = views_of(b->h_table[slot]);
    b->launch.resize(nviews);
    int dtype = -1, variant = 0;
    unsigned chunks = 0;
    int dist = 0;
    long long tiles = 0;
    raypc_status st;
    for (int i = 0; i < nviews; ++i) {
        const raypc_view& q = views[i];
        Volume* V = nullptr;
        if ((st = get_volume(ctx, q.vol, &V))) return st;
        Level* L = nullptr;
        if ((st = get_level(V, q.lod, &L))) return st;
        if (dtype < 0) dtype = V->dtype;
        if (V->dtype != dtype) return fail(RAYPC_ERR_INVALID_ARG, "view %d: all views of a batch need one storage dtype", i);
        RenderArgs& a = b->launch[i].a;
        if ((st = make_render_args(V, L, &q.cam, q.w, q.h, &q.opts, q.out_rgba_dev, q.stats_dev, &a))) return st;
        if ((st = brush_from_host(V, q.lo, q.hi, q.active_mask, &a.brush))) return st;
        if ((st = pos_from_host(q.pos_lo, q.pos_hi, q.pos_mask, &a.brush))) return st;
        finish_position_brush(a);
        if (i == 0) variant = a.variant;
        a.variant = variant;
        tiles += (long long)((q.w + block_tile_w(variant) - 1) / block_tile_w(variant)) *
                 ((q.h + block_tile_h(variant) - 1) / block_tile_h(variant));
        if (tiles > 0x7fffffffLL) return fail(RAYPC_ERR_INVALID_ARG, "batch has more than 2^31 tiles");
        // per view: sub-brick activity bits and the sub-bricks' padded empty-space distance (bytes)
        const size_t words = L->nswords(), need = words + (padded_bytes(L->n) + 3) / 4;
        if (b->bits_words[i] < need) {
            // growing a slot's masks: no batch may still be reading the old ones
            wait_idle(b);
            if (b->bits[i]) cudaFree(b->bits[i]);
            b->bits[i] = nullptr;
            b->bits_words[i] = 0;
            size_t ch = 0;
            if ((st = ctx->alloc((void**)&b->bits[i], need * sizeof(uint32_t), &ch))) return st;
            b->charged += ch;
            b->bits_words[i] = need;
        }
        const size_t cells = (size_t)L->n * L->n * L->n;
        if (b->cls_cells[i] < cells) {
            // growing a slot's cell classes: no batch may still be reading the old ones
            wait_idle(b);
            if (b->cls[i]) cudaFree(b->cls[i]);
            b->cls[i] = nullptr;
            b->cls_cells[i] = 0;
            size_t ch = 0;
            if ((st = ctx->alloc((void**)&b->cls[i], cells * sizeof(uint16_t), &ch))) return st;
            b->charged += ch;
            b->cls_cells[i] = cells;
        }
        BrushItem it = brush_item(V, *L, a.brush);
        it.active = b->bits[i];
        it.cls = b->cls[i];
        it.sdist = reinterpret_cast<uint8_t*>(b->bits[i] + words);
        if (q.opts.tf_skip) {
            a.open = 0;
            it.tf_prefix = V->tf_prefix;
            it.color_var = V->color_var;
            it.tf_lo = a.tf_lo;
            it.tf_scale = a.tf_scale;
        }
        it.chunk_begin = chunks;
        chunks += brush_chunks(L->n);
        it.dist_begin = dist;
        dist += subbrick_distance_tiles(L->n);
        T[i] = it;
        a.lv.sactive = it.active;
        a.lv.sdist = it.sdist;
        a.cls = it.cls;
        b->launch[i].t = ViewTiles{b->d_tiles + i, b->d_done[slot] + i, b->seq + 1};
    }
    H->nviews = nviews;
    H->chunks = chunks;
    H->dist_total = dist;
    if (!b->exec[slot] || b->exec_dtype[slot] != dtype || b->nodes[slot].size() < (size_t)nviews)
        if ((st = capture(b, slot, dtype))) return st;
    for (int i = 0; i < nviews; ++i) {
        const cudaKernelNodeParams p = render_view_node(b->launch[i], dtype);
        CK(cudaGraphExecKernelNodeSetParams(b->exec[slot], b->nodes[slot][i], &p), "batch render parameters");
    }
    for (; b->enabled[slot] < nviews; ++b->enabled[slot])
        CK(cudaGraphNodeSetEnabled(b->exec[slot], b->nodes[slot][b->enabled[slot]], 1), "batch render node");
    for (; b->enabled[slot] > nviews; --b->enabled[slot])
        CK(cudaGraphNodeSetEnabled(b->exec[slot], b->nodes[slot][b->enabled[slot] - 1], 0), "batch render node");
    CK(cudaGraphLaunch(b->exec[slot], (cudaStream_t)stream), "batch graph launch");
    CK(cudaEventRecord(b->done[slot], (cudaStream_t)stream), "batch completion event");
    b->used[slot] = true;
    b->last_slot = slot;
    b->seq += 1;
    b->cur ^= 1;
    count_launches(2 + nviews);
    return RAYPC_OK;
}

}  // extern "C"
