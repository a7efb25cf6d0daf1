// What a brush edit computes (Section 2.2: the data is not modified, so only
// the classification of the sub-bricks and of the interpolation cells changes):
// one launch gives the activity bits of the sub-bricks of any number of levels
// and, for the levels that ask for them, the cell classes of the active ones.
//
// A block takes a chunk of 32-bit words of activity: its warps first classify the
// words (a lane per sub-brick: shell, position brush, min/max against the
// brush), then compute the cell classes of the active sub-bricks in groups of 4
// that are neighbours in x (16 x 4 x 4 cells), taken one by one from a list in
// shared memory because some words have none and some 8 of them. A lane takes two
// cells in x and walks z: each cell's corners are folded along x and y in the
// lane, along z from plane to plane in registers. A variable whose range over every
// active sub-brick of the group lies inside the brush by its margin is not read
// at all (of a 6-variable brush's variables 4 of 6, on average, at 256^3). FP16
// volumes fold two cells per instruction as binary16 pairs (exact) and decide them
// with four comparisons against binary16 bounds (see half_bounds). Both hold for
// sub-bricks without NaN or infinite values, which the ingest marks; others read every
// variable that has some and are decided value by value (512^3 FP16 with NaN outside the
// shell: 242 us; 568 where one NaN took both from the whole level, 545 before either).
//
// Bound by load latency. One launch against the former four and their counters'
// clears, which read every restricted variable's x-pairs a sub-brick at a time:
// 532 -> 205 us at 512^3 FP16 with a 6-variable brush, 109 -> 58 us at 256^3 FP16,
// 68 -> 44 us at 256^3 FP32 with 4 variables (of 205 us the classification takes
// 44, the stores 29). Groups of 8 with whole cells' rows in registers measured 250-
// 390, one warp per word 216, the x-pair layout 204 with twice the bytes.
#include <algorithm>

#include "common.cuh"

namespace raypc {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kBrushWarps = 8;
constexpr int kBrushBlocks = 6;                       // resident blocks per SM: load latency wants the warps
constexpr unsigned kChunkWords = 16;                  // words a block classifies before it takes their groups

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

// Corner folds of a lane's two cells (x, x + 1), x even, as a pair of values.
template <int DT> struct Corners;
template <> struct Corners<kF16> {
    using V = __half2;
    static __device__ __forceinline__ V lo(V a, V b) { return __hmin2(a, b); }
    static __device__ __forceinline__ V hi(V a, V b) { return __hmax2_nan(a, b); }
    // corners (x, x+1) and (x+1, x+2) of row c; EVEN: rows start at even elements and x+1 < n
    template <bool EVEN>
    static __device__ __forceinline__ void row(const void* c, size_t r, int x0, int x1, int x2, V& mn, V& mx) {
        const unsigned short* p = static_cast<const unsigned short*>(c) + r;
        const unsigned a = EVEN ? __ldg(reinterpret_cast<const unsigned*>(p + x0))
                                : (unsigned)__ldg(p + x0) | ((unsigned)__ldg(p + x1) << 16);
        const unsigned b = __byte_perm(a, (unsigned)__ldg(p + x2), 0x5432);
        mn = lo(as_half2(a), as_half2(b));
        mx = hi(as_half2(a), as_half2(b));
    }
    template <bool ODD>
    static __device__ __forceinline__ unsigned classes(const BrushShared& S, int v, V mn, V mx) {
        const unsigned need = 0x00010001u << v;
        if (!ODD && ((S.pairs >> v) & 1u)) {
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
    using V = float2;
    static __device__ __forceinline__ V lo(V a, V b) { return make_float2(fminf(a.x, b.x), fminf(a.y, b.y)); }
    static __device__ __forceinline__ V hi(V a, V b) { return make_float2(max_nan(a.x, b.x), max_nan(a.y, b.y)); }
    template <bool EVEN>
    static __device__ __forceinline__ void row(const void* c, size_t r, int x0, int x1, int x2, V& mn, V& mx) {
        const float* p = static_cast<const float*>(c) + r;
        const float2 a = EVEN ? __ldg(reinterpret_cast<const float2*>(p + x0)) : make_float2(__ldg(p + x0), __ldg(p + x1));
        const float2 b = make_float2(a.y, __ldg(p + x2));
        mn = lo(a, b);
        mx = hi(a, b);
    }
    template <bool>
    static __device__ __forceinline__ unsigned classes(const BrushShared& S, int v, V mn, V mx) {
        const float lo = S.it.brush.lo[v], hi = S.it.brush.hi[v];
        return cell_class(mn.x, mx.x, lo, hi, 1u << v) | (cell_class(mn.y, mx.y, lo, hi, 1u << v) << 16);
    }
};

constexpr unsigned kOdd = 1u << 16;  // in a list entry: NaN or infinite values
constexpr int kGroup = 4;            // sub-bricks of a group: 8 lanes of two cells in x, 4 lanes in y

// Classes of the cells of up to kGroup sub-bricks (sx .. sx + 3, sy, sz), sx a multiple
// of kGroup, over the variables `vars`; written for the sub-bricks in `act` (bit k: sx + k). ODD: one
// of them may hold NaN or infinite values, which the binary16 bounds do not decide.
template <int DT, bool EVEN, bool ODD>
__device__ __forceinline__ void classes_of_group(const BrushShared& S, int sx, int sy, int sz, unsigned act,
                                                 unsigned vars, int lane) {
    using C = Corners<DT>;
    using V = typename C::V;
    const int n = S.it.n;
    const int x = sx * kSub + 2 * (lane & 7), y = sy * kSub + (lane >> 3), z = sz * kSub;
    const size_t nn = (size_t)n * n;
    const int x0 = EVEN ? min(x, n - 2) : min(x, n - 1), x1 = min(x + 1, n - 1), x2 = min(x + 2, n - 1);
    const size_t r0 = (size_t)min(y, n - 1) * n, r1 = (size_t)min(y + 1, n - 1) * n;
    unsigned word[kSub] = {0u, 0u, 0u, 0u};
    while (vars) {                                           // uniform over the warp
        const int v = __ffs(vars) - 1;
        vars &= vars - 1u;
        const char* plane = static_cast<const char*>(S.it.cells) + nn * n * (size_t)v * (DT == kF16 ? 2 : 4);
        V pmn{}, pmx{};                                      // the previous z plane, folded along x and y
#pragma unroll
        for (int c = 0; c <= kSub; ++c) {
            const size_t rz = (size_t)min(z + c, n - 1) * nn;
            V amn, amx, bmn, bmx;
            C::template row<EVEN>(plane, rz + r0, x0, x1, x2, amn, amx);
            C::template row<EVEN>(plane, rz + r1, x0, x1, x2, bmn, bmx);
            const V mn = C::lo(amn, bmn), mx = C::hi(amx, bmx);
            if (c > 0) word[c > 0 ? c - 1 : 0] |= C::template classes<ODD>(S, v, C::lo(pmn, mn), C::hi(pmx, mx));
            pmn = mn;
            pmx = mx;
        }
    }
    // cells with an index of n - 1 do not exist
    if (!((act >> ((lane & 7) >> 1)) & 1u) || x >= n - 1 || y >= n - 1) return;
#pragma unroll
    for (int c = 0; c < kSub; ++c) {
        if (z + c >= n - 1) break;
        uint16_t* out = S.it.cls + ((size_t)(z + c) * n + y) * n + x;
        if (EVEN) {
            *reinterpret_cast<unsigned*>(out) = word[c];
        } else {
            out[0] = (uint16_t)word[c];
            if (x + 1 < n - 1) out[1] = (uint16_t)(word[c] >> 16);
        }
    }
}

// Classify word w (32 sub-bricks) of the item, store its activity bits and append the
// groups with active sub-bricks to the block's list.
__device__ __forceinline__ void classify_word(const BrushShared& S, unsigned w, int lane, uint2* list, unsigned* count) {
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
    const unsigned word = __ballot_sync(kFull, act);
    if (lane == 0) S.it.active[w] = word;
    if (!S.it.cls || word == 0u) return;
    // a NaN corner fails its cell whatever the range says: ranges do not decide variables that may
    // have one. Such a variable sets kOdd beside the variables to read.
    unsigned mine = act ? S.it.brush.mask & ~inside : 0u;
    if (act && !S.finite) {
        for (unsigned m = S.it.brush.mask; m; m &= m - 1u) {
            const int v = __ffs(m) - 1;
            const uint8_t* odd = S.it.stats.odd + (size_t)v * total + b;
            if (odd[0] || (b % (unsigned)nsb + 1u < (unsigned)nsb && odd[1])) mine |= (1u << v) | kOdd;
        }
    }
    // the lanes of this lane's group: kGroup neighbours in x, cut at the word's and the row's ends
    const int sx = (int)(b % (unsigned)nsb), k = sx & (kGroup - 1);
    const int first = lane - k, end = min(min(first + kGroup, lane + nsb - sx), 32);
    const unsigned lanes = (end < 32 ? (1u << end) - 1u : kFull) & ~((1u << max(first, 0)) - 1u);
    unsigned vars = 0u;
#pragma unroll
    for (int q = 0; q < kGroup; ++q) {                       // the group's lanes are consecutive
        const int l = max(first, 0) + q;
        const unsigned m = __shfl_sync(kFull, mine, l & 31);
        if (l < end) vars |= m;
    }
    const unsigned here = word & lanes;
    const bool head = lane == max(first, 0) && here != 0u;   // one lane per group
    const unsigned heads = __ballot_sync(kFull, head);
    unsigned at = 0u;
    if (lane == 0) at = atomicAdd(count, (unsigned)__popc(heads));
    at = __shfl_sync(kFull, at, 0) + __popc(heads & ((1u << lane) - 1u));
    // sub-brick id of the group's first place (its row's, in front of this word too), which of
    // the group are active, the variables to read
    if (head) list[at] = make_uint2(b - k, (first >= 0 ? here >> first : here << -first) << 8 | vars);
}

// The warps take the groups of a block's list one by one. ODD: those with NaN or infinite values
// of FP16 levels, in a pass of their own, because a branch in the other groups' loop cost them
// registers (256^3 FP16, 8 variables of noise: 12 % of the edit; the passes 7 %).
template <int DT, bool ODD>
__device__ __forceinline__ void take_groups(const BrushShared& S, const uint2* list, unsigned groups, unsigned* next, int lane) {
    const int nsb = S.it.nsb;
    for (;;) {
        unsigned g = 0u;
        if (lane == 0) g = atomicAdd(next, 1u);
        g = __shfl_sync(kFull, g, 0);
        if (g >= groups) break;
        const uint2 e = list[g];
        if (DT == kF16 && ((e.y & kOdd) != 0u) != ODD) continue;
        const int sx = (int)(e.x % (unsigned)nsb), sy = (int)((e.x / nsb) % nsb), sz = (int)(e.x / ((unsigned)nsb * nsb));
        if ((S.it.n & 1) == 0) classes_of_group<DT, true, ODD>(S, sx, sy, sz, e.y >> 8, e.y & 0xffu, lane);
        else classes_of_group<DT, false, ODD>(S, sx, sy, sz, e.y >> 8, e.y & 0xffu, lane);
    }
}

// Blocks walk the chunks (P.words words each) of all items: the warps first
// classify the chunk's words, then take its groups from the block's list one by one
// (a word has between none and 32, and each takes a load latency per variable).
template <int DT>
__global__ void __launch_bounds__(32 * kBrushWarps, kBrushBlocks) k_brush(const __grid_constant__ BrushLaunch P) {
    __shared__ BrushShared S;
    __shared__ uint2 s_list[32 * kChunkWords];
    __shared__ unsigned s_count, s_next;
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
        __syncthreads();                                     // the previous chunk's state is no longer read
        if (threadIdx.x == 0) s_count = s_next = 0u;
        if (vi != cur) {                                     // uniform over the block
            static_assert(sizeof(BrushItem) % 4 == 0, "copied by words");
            for (int i = threadIdx.x; i < (int)(sizeof(BrushItem) / 4); i += blockDim.x)
                reinterpret_cast<unsigned*>(&S.it)[i] = reinterpret_cast<const unsigned*>(items + vi)[i];
            if (threadIdx.x == 0) S.pairs = 0u;
            __syncthreads();
            if (threadIdx.x <= kMaxVars) {
                const unsigned bits = S.it.stats.mag[threadIdx.x];   // magnitude of the variable
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
            cur = vi;
        }
        __syncthreads();
        const int nsb = S.it.nsb;
        const unsigned words = ((unsigned)nsb * nsb * nsb + 31u) / 32u;
        const unsigned w0 = (c - S.it.chunk_begin) * P.words;
        for (unsigned w = w0 + warp; w < min(words, w0 + P.words); w += kBrushWarps)
            classify_word(S, w, lane, s_list, &s_count);
        __syncthreads();
        take_groups<DT, false>(S, s_list, s_count, &s_next, lane);
        if (DT == kF16 && !S.finite) {                       // uniform over the block
            __syncthreads();
            if (threadIdx.x == 0) s_next = 0u;
            __syncthreads();
            take_groups<DT, DT == kF16>(S, s_list, s_count, &s_next, lane);
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

int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

}  // namespace

unsigned brush_chunks(int n) { return (words_of(n) + kChunkWords - 1) / kChunkWords; }

// Chunks of kChunkWords words, or on grids with fewer chunks than SMs have room for,
// fewer words, so that every SM has some.
cudaError_t launch_brush(BrushLaunch& P, int dtype, cudaStream_t stream) {
    unsigned words = 0;
    for (int i = 0; i < P.nitems; ++i) words += words_of(P.items[i].n);
    const unsigned blocks = (unsigned)sm_count() * kBrushBlocks;
    P.table = nullptr;
    P.header = nullptr;
    P.words = std::min<unsigned>(kChunkWords, std::max(1u, (words + blocks - 1) / blocks));
    P.chunks = 0;
    for (int i = 0; i < P.nitems; ++i) {
        P.items[i].chunk_begin = P.chunks;
        P.chunks += (words_of(P.items[i].n) + P.words - 1) / P.words;
    }
    if (dtype == kF16) k_brush<kF16><<<std::min(P.chunks, blocks), 32 * kBrushWarps, 0, stream>>>(P);
    else k_brush<kF32><<<std::min(P.chunks, blocks), 32 * kBrushWarps, 0, stream>>>(P);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_brush_views(const BatchHeader* hdr, const BrushItem* table, int dtype, cudaStream_t stream) {
    BrushLaunch P{};
    P.table = table;
    P.header = hdr;
    P.words = kChunkWords;
    const unsigned blocks = (unsigned)sm_count() * kBrushBlocks;
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
