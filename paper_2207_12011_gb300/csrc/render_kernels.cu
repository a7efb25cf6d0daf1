// Brushed emission-absorption ray marching (Section 2.2 of the paper).
//
// One thread per ray; a warp covers a small pixel tile (8x4, 16x2 or 4x8: the
// launch variant) so that neighbouring rays fetch neighbouring vertices, and a
// 128-thread block covers 2x2 warp tiles (64-thread blocks measured 500-510 us
// against 472 at 256^3 FP32, 1024^2, 256-thread ones 485: neighbouring warps
// share cache lines, and a block holds its registers until its last warp ends).
// The per-pixel march is one device function shared by the single-frame kernel
// and the batch's, so a view renders bit-identically alone and inside a batch.
//
// The march alternates a search and an evaluation, because instruction issue
// bounds it (not memory: 62 MB of DRAM traffic per 256^3 frame) and most
// lattice samples lie in sub-bricks that no brushed sample can lie in:
//  - search: the sub-bricks of the next kSearch lattice samples of the ray are
//    looked up together in a byte grid of empty-space distances (0: active),
//    whose index takes three FMAs and three rounded-down additions per sample;
//  - evaluation: the samples found in active sub-bricks, in order, each lane
//    its own: position, shell and radius test, interpolation cell (exactly
//    rounded FP32), the cell's class, then the restricted variables that the
//    class does not decide and last the colour variable, each an FP32 trilinear
//    interpolation from four x-pair loads, with exit on the first failure. Kept
//    samples are coloured by the transfer function (from shared memory) and
//    composited front to back with early ray termination.
// Against one sample per pass (position, exact cell, distance, evaluation) this
// executes 398 M instead of 555 M warp instructions at 256^3 FP32, 1024^2 (705 ->
// 472 us) and renders 512^3 FP16 at 1920x1080 in 1.41 instead of 2.20 ms. Every
// decision is taken on the same values in the same order as before.
//
// Where nothing is restricted every sample of the shell is in an active sub-brick, and the
// search, which could only cost, is left out: 256^3 FP32, 1024^2, unbrushed 951 us (1075 with
// it, as with one sample per pass), in the wide form 1239 (1517; 1260 with one sample per pass),
// 512^3 FP16 at 1920x1080 2237 (2483; 2553).
//
// The samples inside the inner core are jumped over analytically (exactly: see
// the march), and lanes that are all far from any active sub-brick skip samples
// together. The lattice itself (t_k = t0 + (k + j) dt, j = 1/2 except in
// jittered progressive passes) is never shifted by a skip.
#include "common.cuh"

namespace raypc {

namespace {

constexpr int kThreads = kRenderThreads;

__device__ __forceinline__ bool bit_of(const uint32_t* bits, uint32_t id) {
    return (__ldg(bits + (id >> 5)) >> (id & 31)) & 1u;
}

// Byte offsets inside one variable's x-pair plane: 32 bits when the plane is
// smaller than 4 GB (WIDE = false), else 64.
template <bool WIDE> struct Offset { using type = uint32_t; };
template <> struct Offset<true> { using type = size_t; };

// FP32 trilinear value of one variable: four pair loads give the 8 corners
// (x0, x0+1) at (y0,z0), (y1,z0), (y0,z1), (y1,z1).
template <int DT, typename OFF>
__device__ __forceinline__ float interp_var(const char* plane, OFF base, OFF sy, OFF sz, float fx, float fy, float fz) {
    const float2 a = Pair<DT>::load(plane + base, 0);
    const float2 b = Pair<DT>::load(plane + (OFF)(base + sy), 0);
    const float2 c = Pair<DT>::load(plane + (OFF)(base + sz), 0);
    const float2 d = Pair<DT>::load(plane + (OFF)(base + sz + sy), 0);
    return trilerp_rn(a.x, a.y, b.x, b.y, c.x, c.y, d.x, d.y, fx, fy, fz);
}

// Per-view block state: the transfer function (staged in shared memory as
// entries and differences to the next entry) and the brush bounds.
struct ViewShared {
    float4 tf[kTF - 1][2];        // (entry j, entry j+1 - entry j)
    float lo[kMaxVars], hi[kMaxVars];
};

// Fill S for view A (all threads of the block call it; the caller syncs).
__device__ __forceinline__ void load_view_shared(const RenderArgs& A, ViewShared& S) {
    for (int i = threadIdx.x; i < kTF - 1; i += blockDim.x) {
        const float4 e0 = A.tf[i], e1 = A.tf[i + 1];
        S.tf[i][0] = e0;
        S.tf[i][1] = make_float4(e1.x - e0.x, e1.y - e0.y, e1.z - e0.z, e1.w - e0.w);
    }
    if (threadIdx.x < kMaxVars) {
        S.lo[threadIdx.x] = A.brush.lo[threadIdx.x];
        S.hi[threadIdx.x] = A.brush.hi[threadIdx.x];
    }
}

// Lattice samples whose sub-bricks are looked up together: 8 loads in flight, and
// the loop's bounds, votes and jumps once per 8 samples. 256^3 FP32, 1024^2:
// 513 us with 4, 507 with 6, 502 with 8, 475 against 472 with 16 in the present
// form (532 with 2; 64^3, 256^2: 59 us with 8, 67 with 16).
constexpr int kSearch = 8;

// Empty-space distance of the sub-brick that holds the sample at (x, y, z).
// The narrow form reads the padded grid (see subbrick_pad): floor(u / 4) of the
// unclamped grid coordinate u comes from the mantissa of u + 1.5 * 2^25 rounded
// down (one unit there is 4), and the pad holds the clamped entries, so the
// index takes no conversion and no clamp. Its callers guarantee -1 <= u < n
// (RenderArgs::narrow); the final min keeps any other input inside the grid.
template <bool WIDE>
__device__ __forceinline__ int sample_distance(const RenderArgs& A, float x, float y, float z, float hn, float off) {
    const int n = A.lv.n, pd = A.lv.pd;
    if (!WIDE) {
        const uint32_t bx = __float_as_uint(__fadd_rd(__fmaf_rn(x, hn, off), 0x1.8p25f));
        const uint32_t by = __float_as_uint(__fadd_rd(__fmaf_rn(y, hn, off), 0x1.8p25f));
        const uint32_t bz = __float_as_uint(__fadd_rd(__fmaf_rn(z, hn, off), 0x1.8p25f));
        const uint32_t id = (bz * pd + by) * pd + bx + A.lv.pbias;
        return __ldg(A.lv.sdist + min(id, A.lv.plast));
    }
    float u;
    const uint32_t ix = (uint32_t)grid_index_rn(x, n, hn, off, u) >> 2;
    const uint32_t iy = (uint32_t)grid_index_rn(y, n, hn, off, u) >> 2;
    const uint32_t iz = (uint32_t)grid_index_rn(z, n, hn, off, u) >> 2;
    if (A.lv.sdist) return __ldg(A.lv.sdist + ((size_t)((iz + 1) * pd + iy + 1) * pd + ix + 1));
    return bit_of(A.lv.sactive, (iz * A.lv.nsb + iy) * A.lv.nsb + ix) ? 0 : 1;
}

// March the ray of this thread's pixel in warp tile `warp` of block tile (tile_x, tile_y) of view A
// and write its pixel, optional counts and (warp-aggregated) statistics. All
// 32 lanes of every warp must call it. DEPTH: the depth output may be requested
// (A.depth); without it the march keeps no trace of the first kept sample. WIDE:
// no bound on the volume's size or the sample positions (see RenderArgs::narrow).
template <int DT, int VAR, bool DEPTH, bool WIDE>
__device__ __forceinline__ void march_pixel(const RenderArgs& A, const ViewShared& S, int tile_x, int tile_y, int warp) {
    using OFF = typename Offset<WIDE>::type;
    const int lane = threadIdx.x & 31;
    constexpr int WTW = warp_tile_w(VAR), WTH = 32 / WTW;
    const int px = tile_x * block_tile_w(VAR) + (warp & 1) * WTW + (lane % WTW);
    const int py = tile_y * block_tile_h(VAR) + (warp >> 1) * WTH + (lane / WTW);
    const bool inside = px < A.w && py < A.h;

    unsigned marched = 0, kept = 0, evald = 0, skipped = 0, hit = 0, ert_hit = 0;
    float Cr = 0.f, Cg = 0.f, Cb = 0.f, Aa = 0.f;
    float depth = __int_as_float(0x7f800000);       // t of the first kept sample; +inf if none

    if (inside) {
        // Camera basis and pixel direction (exactly rounded, fixed order; the same
        // arithmetic as camera_ray_rn, written out here for the register allocation).
        float Fx = __fsub_rn(A.target[0], A.eye[0]);
        float Fy = __fsub_rn(A.target[1], A.eye[1]);
        float Fz = __fsub_rn(A.target[2], A.eye[2]);
        normalize_rn(Fx, Fy, Fz);
        float Rx, Ry, Rz, Ux, Uy, Uz;
        cross_rn(Fx, Fy, Fz, A.up[0], A.up[1], A.up[2], Rx, Ry, Rz);
        normalize_rn(Rx, Ry, Rz);
        cross_rn(Rx, Ry, Rz, Fx, Fy, Fz, Ux, Uy, Uz);
        const float aspect = __fdiv_rn((float)A.w, (float)A.h);
        const float sxs = __fmul_rn(A.tan_half, aspect);
        const float qx = __fdiv_rn((float)(2 * px + 1), (float)A.w);
        const float qy = __fdiv_rn((float)(2 * py + 1), (float)A.h);
        const float sx = __fmul_rn(__fsub_rn(qx, 1.0f), sxs);
        const float sy = __fmul_rn(__fsub_rn(1.0f, qy), A.tan_half);
        float dx = __fmaf_rn(sy, Ux, __fmaf_rn(sx, Rx, Fx));
        float dy = __fmaf_rn(sy, Uy, __fmaf_rn(sx, Ry, Fy));
        float dz = __fmaf_rn(sy, Uz, __fmaf_rn(sx, Rz, Fz));
        normalize_rn(dx, dy, dz);
        const float ox = A.eye[0], oy = A.eye[1], oz = A.eye[2];
        // Outer-sphere interval through the point closest to the centre.
        const float b = dot3_rn(ox, oy, oz, dx, dy, dz);
        const float hx = __fmaf_rn(-b, dx, ox), hy = __fmaf_rn(-b, dy, oy), hz = __fmaf_rn(-b, dz, oz);
        const float disc = __fsub_rn(A.rout2, dot3_rn(hx, hy, hz, hx, hy, hz));
        if (disc > 0.0f) {
            hit = 1;
            const float sq = __fsqrt_rn(disc);
            const float t0 = fmaxf(__fsub_rn(-b, sq), 0.0f);
            const float t1 = __fadd_rn(-b, sq);
            const int n = A.lv.n;
            const float hn = 0.5f * (float)n, off = hn - 0.5f;
            const float dt = A.dt;
            // Lattice end: the first k with t_k >= t1, found once per ray from an
            // estimate corrected with the exact predicate (t_k is non-decreasing in k).
            const float inv_dt = 1.0f / dt;
            // lattice offset of this pixel (1/2 unless this is a jittered progressive pass)
            const float jo = lattice_offset(A.jit_seed, A.jit_pass, (unsigned long long)py * A.w + px);
            int n_lat = max(0, (int)floorf((t1 - t0) * inv_dt - jo));
            while (n_lat > 0 && !(__fmaf_rn(__fadd_rn((float)(n_lat - 1), jo), dt, t0) < t1)) --n_lat;
            while (__fmaf_rn(__fadd_rn((float)n_lat, jo), dt, t0) < t1) ++n_lat;
            // Inner core: the samples core_a..core_b lie inside r_in and fail the shell
            // test, so the march jumps over them. The range comes from the core chord of
            // a slightly smaller sphere and is then verified with the per-sample FP32
            // arithmetic at both ends: t_k grows with k and the exact |o + t d|^2 is
            // convex in t, so no sample in between exceeds the larger end value, and the
            // FP32 |p|^2 of a sample differs from the exact value by at most ~5 * 2^-24
            // relative; ends below r_in^2 (1 - 2^-10) therefore prove every sample in
            // between fails the shell test.
            int core_a = n_lat, core_b = n_lat - 1;               // empty unless verified
            {
                const float hh = dot3_rn(hx, hy, hz, hx, hy, hz);
                const float shrink = __fmul_rn(A.keep_lo2, 1.0f - 0x1p-9f);
                if (hh < shrink) {
                    const float sc = __fsqrt_rn(__fsub_rn(shrink, hh));
                    const float tc0 = __fsub_rn(-b, sc), tc1 = __fadd_rn(-b, sc);
                    const int ka = max(0, (int)ceilf(fminf((tc0 - t0) * inv_dt - jo, 1.0e9f)));
                    const int kb = min(n_lat - 1, (int)floorf(fminf((tc1 - t0) * inv_dt - jo, 1.0e9f)));
                    if (ka < kb) {
                        const float lim = __fmul_rn(A.keep_lo2, 1.0f - 0x1p-10f);
                        const float ta = __fmaf_rn(__fadd_rn((float)ka, jo), dt, t0);
                        const float tb = __fmaf_rn(__fadd_rn((float)kb, jo), dt, t0);
                        const float ax = __fmaf_rn(ta, dx, ox), ay = __fmaf_rn(ta, dy, oy), az = __fmaf_rn(ta, dz, oz);
                        const float bx = __fmaf_rn(tb, dx, ox), by = __fmaf_rn(tb, dy, oy), bz = __fmaf_rn(tb, dz, oz);
                        if (dot3_rn(ax, ay, az, ax, ay, az) <= lim && dot3_rn(bx, by, bz, bx, by, bz) <= lim) {
                            core_a = ka;
                            core_b = kb;
                        }
                    }
                }
            }
            // Coordinate brushes: along the ray each coordinate fma(t_k, d, o) is
            // monotone in k, so the samples inside every restricted coordinate range
            // form one index range [k_first, k_last); the rest are marched but never kept.
            int k_first = 0, k_last = n_lat;
            if (A.brush.pmask & 7u) {
                const float dd[3] = {dx, dy, dz}, oo[3] = {ox, oy, oz};
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    if (!((A.brush.pmask >> a) & 1u)) continue;
                    const float lo = A.brush.plo[a], hi = A.brush.phi[a];
                    const float d = dd[a], o = oo[a];
                    if (d == 0.0f) {                                   // constant coordinate o
                        if (!(o >= lo && o <= hi)) k_last = 0;
                        continue;
                    }
                    // smallest k in [0, n_lat] whose coordinate has entered (leave = false)
                    // or left (leave = true) the range
                    auto first = [&](bool leave) {
                        int l = 0, h = n_lat;
                        while (l < h) {
                            const int m = (l + h) >> 1;
                            const float c = __fmaf_rn(__fmaf_rn(__fadd_rn((float)m, jo), dt, t0), d, o);
                            const bool p = d > 0.0f ? (leave ? c > hi : c >= lo) : (leave ? c < lo : c <= hi);
                            if (p) h = m; else l = m + 1;
                        }
                        return l;
                    };
                    k_first = max(k_first, first(false));
                    k_last = min(k_last, first(true));
                }
            }
            // n_lat is needed again only for the count after the loop: park it in shared
            // memory rather than in a register across the loop
            __shared__ int s_lat[kThreads];
            reinterpret_cast<volatile int*>(s_lat)[threadIdx.x] = n_lat;
            // sample indices are floats from here on (exact: n_lat < 2^24)
            float k = (float)k_first;
            const float k_end = (float)k_last, k_core = (float)(core_b + 1);
            float stop = fminf((float)core_a, k_end);            // first stretch ends at the core
            for (;;) {
                if (k >= stop) {
                    if (stop >= k_end) break;
                    k = fmaxf(k, k_core);                        // the rest after the core
                    stop = k_end;
                    continue;
                }
                // Search: the distances D of the sub-bricks of the next kSearch samples, all
                // loads in flight together (a stretch's last sample stands in for those behind it).
                unsigned todo = 0u;                              // samples k + q in active sub-bricks
                int D = 0;
                if (A.open) {
                    todo = (1u << (int)fminf(stop - k, (float)kSearch)) - 1u;
                } else {
#pragma unroll
                    for (int q = 0; q < kSearch; ++q) {
                        const float kq = fminf(k + (float)q, stop - 1.0f);
                        const float t = __fmaf_rn(__fadd_rn(kq, jo), dt, t0);
                        D = sample_distance<WIDE>(A, __fmaf_rn(t, dx, ox), __fmaf_rn(t, dy, oy), __fmaf_rn(t, dz, oz), hn, off);
                        if (D == 0 && k + (float)q < stop) todo |= 1u << q;
                    }
                }
                // No lane has an active sample and every lane's last one has D >= 2: every
                // sub-brick within D - 1 of it is inactive, so the cell index stays in that
                // box -- at least 4 (D - 1) cells beyond the sub-brick on every side -- for the
                // next floor((4 (D - 1) - 1/16) / (dt n/2)) samples (dt n/2 bounds the cells per
                // sample on any axis; 1/16 cell covers the FP32 rounding of t, the position and
                // the grid coordinate). The lanes running together skip those samples together
                // (the count for D >= 2, 4 or 8, by vote), so they stay on neighbouring samples.
                const unsigned grp = __activemask();
                if (__all_sync(grp, todo == 0u)) {
                    k = fminf(k + (float)kSearch, stop);         // one behind the sample of D
                    if (A.skip && __all_sync(grp, D >= 2 && k + A.jump[2] < 65536.0f)) {
                        const float m = !__all_sync(grp, D >= 4) ? A.jump[0]
                                      : (__all_sync(grp, D >= kDistCap) ? A.jump[2] : A.jump[1]);
                        skipped += (unsigned)m;
                        k += m;
                    }
                    continue;
                }
                // Evaluate this lane's active samples in order. Structured control flow throughout, so
                // that the lanes meet again after every step.
                while (todo) {
                    const float kq = k + (float)(__ffs(todo) - 1);
                    todo &= todo - 1u;
                    const float t = __fmaf_rn(__fadd_rn(kq, jo), dt, t0);
                    const float pxw = __fmaf_rn(t, dx, ox), pyw = __fmaf_rn(t, dy, oy), pzw = __fmaf_rn(t, dz, oz);
                    const float r2 = dot3_rn(pxw, pyw, pzw, pxw, pyw, pzw);
                    if (r2 >= A.keep_lo2 && r2 <= A.keep_hi2) {
                        ++evald;
                        float ux, uy, uz;
                        const int ix = grid_index_rn(pxw, n, hn, off, ux);
                        const int iy = grid_index_rn(pyw, n, hn, off, uy);
                        const int iz = grid_index_rn(pzw, n, hn, off, uz);
                        const OFF cell = ((OFF)iz * n + iy) * n + ix;
                        // cell class: a variable whose 8 corners all pass needs no interpolation,
                        // one whose corners all fail (or hold a NaN) rejects the sample outright
                        unsigned need = A.cls ? (unsigned)__ldg(A.cls + cell) : A.brush.mask;
                        if (!(need & kCellFail)) {
                            const float nm1 = (float)(n - 1);
                            const float fx = grid_weight_rn(ux, ix, nm1), fy = grid_weight_rn(uy, iy, nm1),
                                        fz = grid_weight_rn(uz, iz, nm1);
                            constexpr OFF kPair = DT == kF16 ? 4 : 8;
                            const OFF base = cell * kPair, sy_ = (OFF)n * kPair, sz_ = sy_ * n;
                            const size_t plane = (size_t)n * n * n * kPair;
                            const char* pairs = static_cast<const char*>(A.lv.pairs);
                            // the variables the brush still has to test, the colour variable last (tested
                            // or not): one loop body for both, so that lanes with nothing to test fetch
                            // their colour while the others test
                            const int cv = A.color_var;
                            const bool test_c = (need >> cv) & 1u;
                            need &= ~(1u << cv);
                            bool pass, more;
                            float vc;
                            do {
                                const bool last = need == 0u;
                                const int v = last ? cv : __ffs(need) - 1;
                                need &= need - 1u;
                                vc = interp_var<DT, OFF>(pairs + plane * v, base, sy_, sz_, fx, fy, fz);
                                pass = (last && !test_c) || (vc >= S.lo[v] && vc <= S.hi[v]);
                                more = pass && !last;
                            } while (more);
                            if (pass) {
                                // index of the first kept sample, parked in the depth output until the end
                                if (DEPTH && kept == 0u && A.depth) A.depth[(size_t)py * A.w + px] = kq;
                                ++kept;
                                // transfer function (continuous; no rounding contract needed)
                                float sp = (vc - A.tf_lo) * A.tf_scale;
                                sp = fminf(fmaxf(sp, 0.0f), 255.0f);
                                const int jj = min((int)sp, kTF - 2);
                                const float w = sp - (float)jj;
                                const float4 e0 = S.tf[jj][0], de = S.tf[jj][1];
                                const float er = fmaf(w, de.x, e0.x);
                                const float eg = fmaf(w, de.y, e0.y);
                                const float eb = fmaf(w, de.z, e0.z);
                                const float es = fmaf(w, de.w, e0.w);
                                const float alpha = 1.0f - __expf(-es * dt);
                                const float ta = (1.0f - Aa) * alpha;
                                Cr = fmaf(ta, er, Cr);
                                Cg = fmaf(ta, eg, Cg);
                                Cb = fmaf(ta, eb, Cb);
                                Aa += ta;
                                if (A.ert && Aa >= kErtThreshold) {
                                    ert_hit = 1;
                                    marched = (unsigned)kq + 1u;
                                    todo = 0u;
                                    k = stop = k_end;            // the ray ends here
                                }
                            }
                        }
                    }
                }
                k = fminf(k + (float)kSearch, stop);
            }
            // every lattice sample up to termination
            if (!ert_hit) marched = (unsigned)reinterpret_cast<volatile int*>(s_lat)[threadIdx.x];
            if (DEPTH && kept && A.depth)                         // t of the first kept sample
                depth = __fmaf_rn(__fadd_rn(A.depth[(size_t)py * A.w + px], jo), dt, t0);
        }
        const float tr = 1.0f - Aa;
        float4 o;
        o.x = fmaf(tr, A.bg[0], Cr);
        o.y = fmaf(tr, A.bg[1], Cg);
        o.z = fmaf(tr, A.bg[2], Cb);
        o.w = fmaf(tr, A.bg[3], Aa);
        const size_t pix = (size_t)py * A.w + px;
        A.out[pix] = o;
        if (A.accum) {
            // running mean of the passes 0..jit_pass
            float4 m = o;
            if (A.jit_pass != 0u) {
                const float4 prev = A.accum[pix];
                m.x = fmaf(A.accum_w, o.x - prev.x, prev.x);
                m.y = fmaf(A.accum_w, o.y - prev.y, prev.y);
                m.z = fmaf(A.accum_w, o.z - prev.z, prev.z);
                m.w = fmaf(A.accum_w, o.w - prev.w, prev.w);
            }
            A.accum[pix] = m;
        }
        if (A.counts) {
            A.counts[2 * pix] = marched;
            A.counts[2 * pix + 1] = kept;
        }
        if (DEPTH && A.depth) A.depth[pix] = depth;
    }
    if (A.stats) {
        unsigned vals[6] = {marched, evald, kept, skipped, hit, ert_hit};
#pragma unroll
        for (int s = 0; s < 6; ++s) {
            unsigned r = __reduce_add_sync(0xffffffffu, vals[s]);
            if (lane == 0 && r) atomicAdd(A.stats + s, (unsigned long long)r);
        }
    }
}

template <int DT, int VAR, bool DEPTH, bool WIDE>
__global__ void __launch_bounds__(kThreads) k_render(RenderArgs A) {
    __shared__ ViewShared S;
    load_view_shared(A, S);
    __syncthreads();
    march_pixel<DT, VAR, DEPTH, WIDE>(A, S, blockIdx.x, blockIdx.y, threadIdx.x >> 5);
}

// One view of a batch: the single-frame kernel (its arguments have to sit at a
// fixed place in the launch parameters: the march reads them as constant
// operands, and a table of views indexed by the block measured 530 against
// 474 us at 256^3 FP32, 1024^2) and the view's completion record.
template <int DT, int VAR, bool DEPTH, bool WIDE>
__global__ void __launch_bounds__(kThreads) k_render_view(RenderArgs A, ViewTiles T) {
    __shared__ ViewShared S;
    load_view_shared(A, S);
    __syncthreads();
    march_pixel<DT, VAR, DEPTH, WIDE>(A, S, blockIdx.x, blockIdx.y, threadIdx.x >> 5);
    __syncthreads();                                          // the tile's pixels and statistics are issued
    if (threadIdx.x == 0) {
        // this block's writes before the count: a release, because a full fence would also drop
        // the cache lines that the SM's other blocks are reading
        unsigned prev;
        asm volatile("atom.add.release.gpu.global.u32 %0, [%1], %2;" : "=r"(prev) : "l"(T.tile_done), "r"(1u) : "memory");
        if (prev + 1 == gridDim.x * gridDim.y) {
            // last tile of the view: every other tile's writes precede their counts
            __threadfence();
            for (int k = 0; k < kNStats; ++k)
                T.done->stats[k] = A.stats ? __ldcg(A.stats + k) : 0ull;
            __threadfence_system();                           // record before the flag, as the host sees it
            T.done->seq = T.seq;
        }
    }
}

template <int DT, int VAR, bool DEPTH, bool WIDE>
cudaError_t launch_t(const RenderArgs& a, cudaStream_t stream) {
    dim3 grid((a.w + block_tile_w(VAR) - 1) / block_tile_w(VAR), (a.h + block_tile_h(VAR) - 1) / block_tile_h(VAR));
    k_render<DT, VAR, DEPTH, WIDE><<<grid, kThreads, 0, stream>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

// The wide form (volumes or cameras outside the narrow form's bounds, renders
// that search and have no distance grid) and depth renders use the 8x4 tiles.
template <int DT>
cudaError_t launch_dt(const RenderArgs& a, cudaStream_t stream) {
    if (!a.narrow || (!a.lv.sdist && !a.open)) return launch_t<DT, 1, true, true>(a, stream);
    if (a.depth) return launch_t<DT, 1, true, false>(a, stream);
    switch (a.variant) {
        case 2: return launch_t<DT, 2, false, false>(a, stream);
        case 3: return launch_t<DT, 3, false, false>(a, stream);
        default: return launch_t<DT, 1, false, false>(a, stream);
    }
}

typedef void (*ViewKernel)(RenderArgs, ViewTiles);

template <int DT>
ViewKernel view_kernel(int variant, bool depth, bool wide) {
    if (wide) return k_render_view<DT, 1, true, true>;
    if (depth) return k_render_view<DT, 1, true, false>;
    return variant == 2 ? k_render_view<DT, 2, false, false>
                        : variant == 3 ? k_render_view<DT, 3, false, false> : k_render_view<DT, 1, false, false>;
}

}  // namespace

cudaError_t launch_render(const RenderArgs& a, int dtype, cudaStream_t stream) {
    if (dtype == kF16) return launch_dt<kF16>(a, stream);
    return launch_dt<kF32>(a, stream);
}

// Views with a depth output, and wide ones, run those instances, with 8x4 tiles.
cudaKernelNodeParams render_view_node(ViewLaunch& v, int dtype) {
    const bool wide = !v.a.narrow, depth = v.a.depth != nullptr;
    const int variant = wide || depth ? 1 : v.a.variant;
    v.arg[0] = &v.a;
    v.arg[1] = &v.t;
    cudaKernelNodeParams p{};
    p.func = (void*)(dtype == kF16 ? view_kernel<kF16>(variant, depth, wide) : view_kernel<kF32>(variant, depth, wide));
    p.gridDim = dim3((v.a.w + block_tile_w(variant) - 1) / block_tile_w(variant),
                     (v.a.h + block_tile_h(variant) - 1) / block_tile_h(variant));
    p.blockDim = dim3(kThreads);
    p.kernelParams = v.arg;
    return p;
}

}  // namespace raypc
