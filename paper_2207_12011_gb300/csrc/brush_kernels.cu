// What a brush edit computes (Section 2.2: the data is not modified, so only
// the classification of the sub-bricks and of the interpolation cells changes):
// one launch gives the activity bits of the sub-bricks of any number of levels
// and, for the levels that ask for them, the cell classes of the active ones.
//
// A warp takes 32 consecutive sub-bricks: a lane classifies one (shell, position
// brush, min/max against the brush), a ballot is the word of activity bits, and
// the warp then computes the classes of the active ones in groups of 8 that are
// neighbours in x (32 x 4 x 4 cells). Lanes run along x, so every load is one or
// two whole 64-byte segments; each cell's corners are folded along x in the lane,
// then along y and z from row to row in registers. A variable whose range over
// every active sub-brick of the group lies inside the brush by its margin is not
// read at all (most of a brush's variables, in most groups). FP16 volumes fold
// two cells per instruction as binary16 pairs (exact) and decide them with four
// comparisons against binary16 bounds (see half_bounds).
//
// Bound by instruction issue and load latency: 512^3 FP16 with a 6-variable brush
// reads about a third of the field.
#include <algorithm>

#include "common.cuh"

namespace raypc {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kBrushWarps = 8;

__device__ __forceinline__ float margin(float m) { return __fmaf_rn(m, 0x1p-20f, 0x1p-120f); }

// Class of one cell for one restricted variable from its corner range (mx NaN when
// a corner is): kCellFail, 0 (inside) or `need`.
__device__ __forceinline__ unsigned cell_class(float mn, float mx, float lo, float hi, unsigned need) {
    const float m = fmaxf(fabsf(mn), fabsf(mx));
    const float d = margin(m);
    const float up = __fadd_rn(mx, d), dn = __fsub_rn(mn, d);
    unsigned w = need;
    if (dn >= lo && up <= hi) w = 0u;
    if (up < lo || dn > hi) w = kCellFail;
    if (m > 0x1p126f) w = need;
    if (mx != mx) w = kCellFail;
    return w;
}

// binary16 neighbours (bits of non-NaN values; the infinities are their own outer neighbours).
__device__ __forceinline__ unsigned half_next(unsigned h) {
    if (h == 0x7c00u) return h;
    if (h == 0x8000u) h = 0u;
    return h & 0x8000u ? h - 1u : h + 1u;
}
__device__ __forceinline__ unsigned half_prev(unsigned h) { return half_next(h ^ 0x8000u) ^ 0x8000u; }
__device__ __forceinline__ float half_val(unsigned h) { return __half2float(__ushort_as_half((unsigned short)h)); }

// binary16 bounds of a lower bound lo for corner values of at most M: a cell with
// maximum mx fails (RN(mx + d) < lo) iff mx <= F, and one with minimum mn is inside
// (RN(mn - d) >= lo) iff mn >= I. d is the margin of the cell's own largest
// magnitude m, between that of |h| and that of M for the value h tested; false when
// some binary16 value's class depends on where in that range m lies.
__device__ __forceinline__ bool half_bounds(float lo, float M, unsigned& F, unsigned& I) {
    auto fails = [&](unsigned h, float m) { return __fadd_rn(half_val(h), margin(m)) < lo; };
    auto inside = [&](unsigned h, float m) { return __fsub_rn(half_val(h), margin(m)) >= lo; };
    const unsigned up = __half_as_ushort(__float2half_ru(lo));           // smallest value >= lo
    bool ok = true;
    F = half_prev(up);                                                   // largest value < lo
    if (!fails(F, M)) {
        ok = !fails(F, fabsf(half_val(F)));
        F = half_prev(F);
        ok = ok && (fails(F, M) || F == 0xfc00u);
    }
    I = up;
    if (!inside(I, M)) {
        ok = ok && !inside(I, fabsf(half_val(I)));
        I = half_next(I);
        ok = ok && (inside(I, M) || I == 0x7c00u);
    }
    return ok;
}

// The brush of one item in shared memory.
struct BrushShared {
    BrushItem it;
    unsigned fail_lo[kMaxVars], fail_hi[kMaxVars];     // binary16 bounds, twice in a word: fails iff
    unsigned in_lo[kMaxVars], in_hi[kMaxVars];         // mx <= fail_lo or mn >= fail_hi; inside iff
                                                       // mn >= in_lo and mx <= in_hi
    unsigned pairs;                                    // variables decided by them
    unsigned finite;                                   // the level holds finite values only
};

__device__ __forceinline__ __half2 as_half2(unsigned u) { return *reinterpret_cast<const __half2*>(&u); }
__device__ __forceinline__ unsigned as_bits(__half2 h) { return *reinterpret_cast<const unsigned*>(&h); }

// Corner folds of a lane's cells: FP16 two cells in x as a binary16 pair, FP32 one.
template <int DT> struct Corners;
template <> struct Corners<kF16> {
    using V = __half2;
    static constexpr int kX = 2, kZ = 2;               // cells of a lane along x and z
    static __device__ __forceinline__ V lo(V a, V b) { return __hmin2(a, b); }
    static __device__ __forceinline__ V hi(V a, V b) { return __hmax2_nan(a, b); }
    // corners (x, x+1) and (x+1, x+2) of a row, x even; even: rows start at even elements
    static __device__ __forceinline__ void row(const void* cells, size_t r, int x, int n, bool even, V& mn, V& mx) {
        const unsigned short* c = static_cast<const unsigned short*>(cells) + r;
        const int x0 = min(x, (n - 1) & ~1), x1 = min(x + 1, n - 1), x2 = min(x + 2, n - 1);
        const unsigned p = even ? __ldg(reinterpret_cast<const unsigned*>(c + x0))
                                : (unsigned)__ldg(c + x0) | ((unsigned)__ldg(c + x1) << 16);
        const unsigned q = __byte_perm(p, (unsigned)__ldg(c + x2), 0x5432);
        mn = lo(as_half2(p), as_half2(q));
        mx = hi(as_half2(p), as_half2(q));
    }
    static __device__ __forceinline__ unsigned classes(const BrushShared& S, int v, V mn, V mx) {
        const unsigned need = 0x00010001u << v;
        if ((S.pairs >> v) & 1u) {
            const unsigned fail = __hle2_mask(mx, as_half2(S.fail_lo[v])) | __hge2_mask(mn, as_half2(S.fail_hi[v]));
            const unsigned in = __hge2_mask(mn, as_half2(S.in_lo[v])) & __hle2_mask(mx, as_half2(S.in_hi[v]));
            return (fail & 0x80008000u) | (~(fail | in) & need);
        }
        const float2 a = __half22float2(mn), b = __half22float2(mx);
        const float lo = S.it.brush.lo[v], hi = S.it.brush.hi[v];
        return cell_class(a.x, b.x, lo, hi, 1u << v) | (cell_class(a.y, b.y, lo, hi, 1u << v) << 16);
    }
};
template <> struct Corners<kF32> {
    using V = float;
    static constexpr int kX = 1, kZ = 4;
    static __device__ __forceinline__ V lo(V a, V b) { return fminf(a, b); }
    static __device__ __forceinline__ V hi(V a, V b) { return max_nan(a, b); }
    static __device__ __forceinline__ void row(const void* cells, size_t r, int x, int n, bool, V& mn, V& mx) {
        const float* c = static_cast<const float*>(cells) + r;
        const float a = __ldg(c + min(x, n - 1)), b = __ldg(c + min(x + 1, n - 1));
        mn = lo(a, b);
        mx = hi(a, b);
    }
    static __device__ __forceinline__ unsigned classes(const BrushShared& S, int v, V mn, V mx) {
        return cell_class(mn, mx, S.it.brush.lo[v], S.it.brush.hi[v], 1u << v);
    }
};

// Classes of the cells of up to 8 sub-bricks (sx .. sx + 7, sy, sz), sx a multiple
// of 8, over the variables `vars`; written for the sub-bricks in `act` (bit k: sx + k).
template <int DT>
__device__ __forceinline__ void classes_of_group(const BrushShared& S, int sx, int sy, int sz, unsigned act,
                                                 unsigned vars, int lane) {
    using C = Corners<DT>;
    using V = typename C::V;
    constexpr int kLanes = 32 / C::kX;                       // lanes along x; the others take the next z cells
    const int n = S.it.n;
    const int x = sx * kSub + (lane % kLanes) * C::kX, y = sy * kSub, z = sz * kSub + (lane / kLanes) * C::kZ;
    const size_t nn = (size_t)n * n;
    const bool even = (n & 1) == 0;
    unsigned word[C::kZ][kSub];
#pragma unroll
    for (int c = 0; c < C::kZ; ++c)
#pragma unroll
        for (int r = 0; r < kSub; ++r) word[c][r] = 0u;
    while (vars) {                                           // uniform over the warp
        const int v = __ffs(vars) - 1;
        vars &= vars - 1u;
        const char* plane = static_cast<const char*>(S.it.cells) + nn * n * (size_t)v * (DT == kF16 ? 2 : 4);
        V pmn[kSub], pmx[kSub];                              // the previous z plane, folded along x and y
#pragma unroll
        for (int c = 0; c <= C::kZ; ++c) {
            const size_t rz = (size_t)min(z + c, n - 1) * nn;
            V rmn[kSub + 1], rmx[kSub + 1];
#pragma unroll
            for (int r = 0; r <= kSub; ++r)
                C::row(plane, rz + (size_t)min(y + r, n - 1) * n, x, n, even, rmn[r], rmx[r]);
#pragma unroll
            for (int r = 0; r < kSub; ++r) {
                const V mn = C::lo(rmn[r], rmn[r + 1]), mx = C::hi(rmx[r], rmx[r + 1]);
                if (c > 0) word[c - 1][r] |= C::classes(S, v, C::lo(pmn[r], mn), C::hi(pmx[r], mx));
                pmn[r] = mn;
                pmx[r] = mx;
            }
        }
    }
    // cells with an index of n - 1 do not exist
    if (!((act >> ((lane % kLanes) * C::kX / kSub)) & 1u) || x >= n - 1) return;
#pragma unroll
    for (int c = 0; c < C::kZ; ++c)
#pragma unroll
        for (int r = 0; r < kSub; ++r) {
            if (z + c >= n - 1 || y + r >= n - 1) continue;
            uint16_t* out = S.it.cls + ((size_t)(z + c) * n + (y + r)) * n + x;
            if (C::kX == 2 && even) {
                *reinterpret_cast<unsigned*>(out) = word[c][r];
            } else {
                out[0] = (uint16_t)word[c][r];
                if (C::kX == 2 && x + 1 < n - 1) out[1] = (uint16_t)(word[c][r] >> 16);
            }
        }
}

// Word w (32 sub-bricks) of the item; of its groups, this warp computes those with
// number % split == part.
template <int DT>
__device__ __forceinline__ void classify_word(const BrushShared& S, unsigned w, int part, int split, int lane) {
    const int nsb = S.it.nsb;
    const unsigned total = (unsigned)nsb * nsb * nsb;
    const unsigned b = w * 32u + lane;
    unsigned inside = 0u;
    bool act = b < total && classify_brick(b, nsb, kSub, 2.0f / (float)S.it.n, S.it.rin2, S.it.rout2, S.it.brush,
                                           S.it.nvars, S.it.sbmin, S.it.sbmax, inside);
    if (act && S.it.tf_prefix) {                             // TF-aware skipping of a batched view
        const size_t o = (size_t)b * S.it.nvars + S.it.color_var;
        act = tf_range_visible(S.it.sbmin[o], S.it.sbmax[o], S.it.tf_prefix, S.it.tf_lo, S.it.tf_scale);
    }
    unsigned rem = __ballot_sync(kFull, act);
    if (lane == 0 && part == 0) S.it.active[w] = rem;
    if (!S.it.cls) return;
    // a NaN corner fails its cell whatever the range says: ranges decide finite levels only
    const unsigned mine = S.it.brush.mask & ~(S.finite ? inside : 0u);
    int group = 0;
    while (rem) {
        const int j = __ffs(rem) - 1;
        const unsigned id = w * 32u + j;
        const int sx = (int)(id % nsb), sy = (int)((id / nsb) % nsb), sz = (int)(id / ((unsigned)nsb * nsb));
        const int first = j - (sx & 7);                      // lane of sub-brick sx & ~7 (may be < 0)
        const int end = min(min(first + 8, j + nsb - sx), 32);
        const unsigned lanes = (end < 32 ? (1u << end) - 1u : kFull) & ~((1u << j) - 1u);
        const unsigned here = rem & lanes;
        rem &= ~lanes;
        if (group++ % split != part) continue;
        const unsigned vars = __reduce_or_sync(kFull, (here >> lane) & 1u ? mine : 0u);
        classes_of_group<DT>(S, sx & ~7, sy, sz, first >= 0 ? here >> first : here << -first, vars, lane);
    }
}

// Blocks walk the chunks (kBrushWarps * per_warp / split words) of all items.
template <int DT>
__global__ void __launch_bounds__(32 * kBrushWarps) k_brush(const __grid_constant__ BrushLaunch P) {
    __shared__ BrushShared S;
    const BrushItem* items = P.table ? P.table : P.items;
    const int nitems = P.table ? P.header->nviews : P.nitems;
    const unsigned total = P.table ? P.header->chunks : P.chunks;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int cur = -1;
    for (unsigned c = blockIdx.x; c < total; c += gridDim.x) {
        int vi = 0, hi = nitems - 1;
        while (vi < hi) {
            const int mid = (vi + hi + 1) >> 1;
            if (items[mid].chunk_begin <= c) vi = mid; else hi = mid - 1;
        }
        if (vi != cur) {                                     // uniform over the block
            __syncthreads();
            static_assert(sizeof(BrushItem) % 4 == 0, "copied by words");
            for (int i = threadIdx.x; i < (int)(sizeof(BrushItem) / 4); i += blockDim.x)
                reinterpret_cast<unsigned*>(&S.it)[i] = reinterpret_cast<const unsigned*>(items + vi)[i];
            if (threadIdx.x == 0) S.pairs = 0u;
            __syncthreads();
            if (threadIdx.x <= kMaxVars) {
                // magnitudes of the level: keys of another generation hold nothing of this one
                const unsigned long long key = S.it.stats[threadIdx.x];
                const unsigned bits = (unsigned)(key >> 32) == S.it.gen ? (unsigned)key : 0u;
                const int v = threadIdx.x;
                if (v == kMaxVars) {
                    S.finite = bits == 0u;
                } else if (DT == kF16 && v < S.it.nvars) {
                    unsigned f0, i0, f1, i1;
                    const float M = __uint_as_float(bits);
                    const bool ok0 = half_bounds(S.it.brush.lo[v], M, f0, i0);
                    const bool ok1 = half_bounds(-S.it.brush.hi[v], M, f1, i1);
                    S.fail_lo[v] = f0 * 0x10001u;
                    S.in_lo[v] = i0 * 0x10001u;
                    S.fail_hi[v] = (f1 ^ 0x8000u) * 0x10001u;
                    S.in_hi[v] = (i1 ^ 0x8000u) * 0x10001u;
                    if (ok0 && ok1) atomicOr(&S.pairs, 1u << v);
                }
            }
            __syncthreads();
            if (threadIdx.x == 0 && !S.finite) S.pairs = 0u;  // NaN and infinite corners: cell_class
            __syncthreads();
            cur = vi;
        }
        const unsigned words = ((unsigned)S.it.nsb * S.it.nsb * S.it.nsb + 31u) / 32u;
        for (int i = 0; i < P.per_warp; ++i) {
            const unsigned unit = ((c - S.it.chunk_begin) * P.per_warp + i) * kBrushWarps + warp;
            const unsigned w = unit / P.split;
            if (w < words) classify_word<DT>(S, w, (int)(unit % P.split), P.split, lane);
        }
    }
}

// Activity of the 8^3 bricks of one level and its dilation (inspection only: the
// renders and histograms use the sub-bricks).
__global__ void k_brick_bits(BrickListArgs A) {
    const size_t b = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t nbricks = (size_t)A.nb * A.nb * A.nb;
    unsigned inside = 0;
    const bool act = b < nbricks && classify_brick(b, A.nb, kBrick, 2.0f / (float)A.n, A.rin2, A.rout2, A.brush, A.nvars,
                                                   A.bmin, A.bmax, inside);
    const unsigned word = __ballot_sync(kFull, act);
    if ((threadIdx.x & 31) == 0 && b < nbricks) A.active[b >> 5] = word;
}

__global__ void k_skippable(BrickListArgs A) {
    const size_t b = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t nbricks = (size_t)A.nb * A.nb * A.nb;
    const bool s = b < nbricks && skippable_brick(b, A.nb, A.active);
    const unsigned word = __ballot_sync(kFull, s);
    if ((threadIdx.x & 31) == 0 && b < nbricks) A.skippable[b >> 5] = word;
}

// Ordered compaction of the active 8^3 brick ids, one block of 1024 threads:
// each thread owns a contiguous run of bitmask words; a block-wide exclusive
// scan of the per-thread popcounts gives every thread its offset.
__global__ void __launch_bounds__(1024) k_compact(BrickListArgs A) {
    __shared__ unsigned s_sum[1024];
    const size_t nbricks = (size_t)A.nb * A.nb * A.nb;
    const size_t nwords = (nbricks + 31) / 32;
    const size_t per = (nwords + blockDim.x - 1) / blockDim.x;
    const size_t w0 = min(nwords, threadIdx.x * per), w1 = min(nwords, w0 + per);
    unsigned cnt = 0;
    for (size_t w = w0; w < w1; ++w) cnt += __popc(A.active[w]);
    s_sum[threadIdx.x] = cnt;
    __syncthreads();
    for (int off = 1; off < (int)blockDim.x; off <<= 1) {
        const unsigned add = threadIdx.x >= (unsigned)off ? s_sum[threadIdx.x - off] : 0u;
        __syncthreads();
        s_sum[threadIdx.x] += add;
        __syncthreads();
    }
    unsigned pos = s_sum[threadIdx.x] - cnt;
    for (size_t w = w0; w < w1; ++w) {
        uint32_t bits = A.active[w];
        while (bits) {
            const int j = __ffs(bits) - 1;
            bits &= bits - 1;
            const size_t id = w * 32 + j;
            if (id < nbricks) A.list[pos++] = (uint32_t)id;
        }
    }
    if (threadIdx.x == blockDim.x - 1) *A.n_active = s_sum[threadIdx.x];
}

unsigned words_of(int n) {
    const unsigned nsb = (unsigned)((n + kSub - 1) / kSub);
    return (nsb * nsb * nsb + 31u) / 32u;
}

constexpr int kPerWarp = 2;          // units a warp takes before its block looks for the next chunk

}  // namespace

unsigned brush_chunks(int n) {
    const unsigned unit = (unsigned)(kBrushWarps * kPerWarp);
    return (words_of(n) + unit - 1) / unit;
}

// Grids of fewer words than the GPU has warps give each word's groups to four warps.
cudaError_t launch_brush(BrushLaunch& P, int dtype, cudaStream_t stream) {
    unsigned words = 0;
    for (int i = 0; i < P.nitems; ++i) words += words_of(P.items[i].n);
    P.table = nullptr;
    P.header = nullptr;
    P.split = words < 4096 ? 4 : 1;
    P.per_warp = words < 4096 ? 1 : kPerWarp;
    P.chunks = 0;
    const unsigned unit = (unsigned)(kBrushWarps * P.per_warp / (P.split > kBrushWarps ? 1 : 1));
    for (int i = 0; i < P.nitems; ++i) {
        P.items[i].chunk_begin = P.chunks;
        P.chunks += (words_of(P.items[i].n) * (unsigned)P.split + unit - 1) / unit;
    }
    if (dtype == kF16) k_brush<kF16><<<P.chunks, 32 * kBrushWarps, 0, stream>>>(P);
    else k_brush<kF32><<<P.chunks, 32 * kBrushWarps, 0, stream>>>(P);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_brush_views(const BatchHeader* hdr, const BrushItem* table, int dtype, unsigned blocks,
                               cudaStream_t stream) {
    BrushLaunch P{};
    P.table = table;
    P.header = hdr;
    P.split = 1;
    P.per_warp = kPerWarp;
    if (dtype == kF16) k_brush<kF16><<<blocks, 32 * kBrushWarps, 0, stream>>>(P);
    else k_brush<kF32><<<blocks, 32 * kBrushWarps, 0, stream>>>(P);
    return cudaGetLastError();
}

cudaError_t launch_brick_list(const BrickListArgs& a, cudaStream_t stream) {
    const size_t nbricks = (size_t)a.nb * a.nb * a.nb;
    const unsigned blocks = (unsigned)((nbricks + 255) / 256);
    k_brick_bits<<<blocks, 256, 0, stream>>>(a);
    k_skippable<<<blocks, 256, 0, stream>>>(a);
    k_compact<<<1, 1024, 0, stream>>>(a);
    count_launches(3);
    return cudaGetLastError();
}

}  // namespace raypc
