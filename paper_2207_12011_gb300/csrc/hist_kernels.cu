// Adjacent-axis parallel-coordinates density histograms (Section 2.1 PC data,
// Fig. 2): for every in-shell (and, optionally, in-brush) cell and every pair
// of adjacent axes (a, a+1), H[a][bin_a][bin_{a+1}] += 1.
//
// A scan over HBM, the binning of the kept cells, and the counting. Rows whose cells
// all lie outside the shell are skipped without touching memory. The vector kernels
// (even grid edge, 16-byte aligned fields) stream 16-byte chunks per variable (8 FP16
// or 4 FP32 cells per lane): through a cp.async double buffer in shared memory and a
// compact list of the kept cells when something is brushed, straight into
// registers when every in-shell cell counts. The scalar kernel (odd grid edges,
// unaligned fields) takes one cell per lane. Position axes and the position
// brush use the cell centre, coordinate RN((2i + 1 - n) / n). With the
// volume's own brush the cells of inactive 4^3 sub-bricks are skipped without loads:
// every vertex of such a sub-brick fails the brush (its values lie between the
// sub-brick's min and max) or lies outside the shell (the sub-brick's widened
// box, which holds the vertex centres, misses the shell). The in-shell test is
// integer-exact. Bins come from the FP32 edges: an affine guess, checked against every
// edge when the table is staged, and corrected by comparisons where that finds it inexact.
//
// What bounds a large call is the counting: five L2 atomics per cell of six axes, of
// which few can be merged (neighbouring cells of a 256-bin table rarely share a bin
// pair) and many meet at hot bins. Large grids therefore list the cells' bins in HBM and
// count them one pair at a time in shared memory (k_hist_count): 512^3 FP16, 6
// axes, 256 bins, whole shell 1438 -> 537 us; 4 brushed variables 422 -> 313 us;
// 250^3 264 -> 115 us. Smaller grids, tables that do not fit and calls without scratch
// add runs of equal bins straight to L2 (see by_pair), on large grids spread over
// partial histograms that a reduction sums.
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "host_math.h"

namespace raypc {

namespace {

constexpr int kHistThreads = 256;                    // scalar kernel
constexpr int kHistVecThreads = 512;                 // vector kernel (two resident blocks per SM)
constexpr int kHistVecWarps = kHistVecThreads / 32;
constexpr unsigned kFull = 0xffffffffu;

// Affine guess of the bin of v, 0 .. bins - 1, non-decreasing in v (a NaN v gives 0): the place of v
// among the bins as a fraction, saturated to [0, 1], times top = the float below bins, rounded
// down to an integer in the low mantissa bits of the result.
__device__ __forceinline__ unsigned bin_guess_raw(float top, float v, float scale, float off) {
    return __float_as_uint(__fmaf_rd(__saturatef(fmaf(v, scale, off)), top, 0x1p23f));
}
__device__ __forceinline__ int bin_guess(float top, float v, float scale, float off) {
    return (int)(bin_guess_raw(top, v, scale, off) - 0x4b000000u);
}
__device__ __forceinline__ float guess_top(int bins) { return __uint_as_float(__float_as_uint((float)bins) - 1u); }

// How the bins of a call's axes are found from the guess (stage_edges picks one).
enum BinMode : int {
    kBinWalk = 0,                  // the guess is walked to the bin, comparing edges
    kBinNear = 1,                  // the guess is at most one bin off for every v
    kBinExact = 2,                 // the guess is the bin of every binary16 v
};

// From a guess to the bin. Out of line: rare, and an inlined copy per axis made the kernels too large
// to come from HBM in time when their first launch finds the caches full of other data.
__device__ __noinline__ int walk_bin(const float* e, int bins, float v, int j) {
    while (j > 0 && !(v >= e[j])) --j;
    while (j < bins - 1 && v >= e[j + 1]) ++j;
    return j;
}

// Number of interior edges e_1..e_{bins-1} that are <= v, for non-decreasing edges:
// the guess corrected with comparisons of edges only, so exact for any edges. The
// staged table holds NaN for e_0 and e_bins, on which no count depends. NaN values
// compare false everywhere and land in bin 0.
template <int MODE>
__device__ __forceinline__ int bin_of(const float* e, int bins, float top, float v, float scale, float off) {
    int j = bin_guess(top, v, scale, off);
    if constexpr (MODE == kBinNear) {
        j += (v >= e[j + 1] ? 1 : 0) - (v < e[j] ? 1 : 0);
    } else if constexpr (MODE == kBinWalk) {
        j = walk_bin(e, bins, v, j);
    }
    return j;
}

// Adds one count per kept lane to hist[key] (all 32 lanes call it, in x order of
// their cells; km = ballot of kept): a lane whose key differs from its left neighbour's, or whose left
// neighbour is not kept, starts a run and adds the run's length once. Neighbouring
// cells of a smooth field mostly share their bin pair, so few atomics remain.
__device__ __forceinline__ void add_runs(uint32_t* hist, unsigned key, bool kept, unsigned km, int lane) {
    const unsigned left = __shfl_up_sync(kFull, key, 1);
    const bool head = kept && (lane == 0 || !((km >> (lane - 1)) & 1u) || left != key);
    const unsigned hm = __ballot_sync(kFull, head);
    if (head) {
        const unsigned after = lane == 31 ? 0u : (kFull << (lane + 1));
        const unsigned stop = (hm | ~km) & after;            // next run start or next lane not kept
        const int end = stop ? __ffs(stop) - 1 : 32;
        atomicAdd(hist + key, (unsigned)(end - lane));
    }
}

// Largest integer m >= 0 with m * m <= a (0 <= a < 2^31; m + 1 <= 46341, so the squares fit 32 bits).
__device__ __forceinline__ int isqrt_floor(int a) {
    unsigned m = (unsigned)__fsqrt_rn((float)a);           // at most one off
    if (m * m > (unsigned)a) --m;
    if ((m + 1u) * (m + 1u) <= (unsigned)a) ++m;
    return (int)m;
}

// Kernel view of a histogram call: the brushed variables and the axes as
// compact lists (the host builds it from HistArgs). Edge tables of up to
// kInlineEdges floats travel in the launch parameters (no device copy);
// larger ones are read from `edges`.
constexpr int kInlineEdges = kHistInlineEdges;
struct HistLaunch {
    const void* cells;
    int n, bins;
    int nbr;                       // brushed variables tested per cell
    int bvar[kMaxVars];
    float blo[kMaxVars], bhi[kMaxVars];
    int naxes;
    int avar[kMaxVars];            // variable of each axis, or kPosAxisBase + position axis
    float plo[kNumPos], phi[kNumPos];
    uint32_t pmask;                // position brush at the cell centre (0: none)
    int use_pos;                   // the position brush or a position axis is in use
    // load slots of the vector kernel: slot a < naxes is axis a (loaded when it names a
    // stored variable), slots naxes..nslot-1 hold brushed variables that are no axis
    int nslot;
    int svar[kMaxVars];            // variable of each slot (-1: position axis, nothing to load)
    uint32_t sbr;                  // bit s: slot s is tested against the brush
    float slo[kMaxVars], shi[kMaxVars];
    uint32_t slo_h2[kMaxVars], shi_h2[kMaxVars];   // FP16 fields: the same bounds as binary16 pairs
    float guess_scale[kMaxVars], guess_off[kMaxVars];   // bin guess: fma(v, scale, off) of the bins
    long long soff[kMaxVars];      // byte offset of each load slot's plane (vector kernel)
    int item0, items;              // rows (or segments) of this launch: item0 .. items - 1
    int rot;                       // row order: plane z is rotated in y by z * rot (mod n)
    int batch;                     // segments a warp of the group walk takes at a time (1 .. 32)
    // list mode: bins of the counted cells instead of counts (see ListSlots)
    unsigned char* list;
    unsigned char* list_mask;      // one byte per 8 cells of the list: the ones that count
    unsigned* list_next;           // zeroed: chunks taken
    unsigned list_chunks, list_batch;   // chunks that fit, chunks a warp takes at a time
    uint32_t* rowctr;              // zeroed row counter, or null: rows by warp stride
    int s_in, s_out;               // shell test on 2x+1-n etc., clamped to int
    int by_pair;                   // direct counts by add_pairs (else add_tuples)
    uint32_t* out;                 // nout histograms; block b adds to copy b % nout
    int nout;
    const uint32_t* sactive;       // optional sub-brick activity (see HistArgs)
    int nsb;
    const float* edges;            // naxes x (bins + 1) on the device, or null: edges_inl
    float edges_inl[kInlineEdges];
};

// The bin edges of a call in shared memory, and how its bins are found.
struct BinTable {
    float off[kMaxVars];           // guess offsets
    int ok[kMaxVars];              // bit c < kOffsets: the guess with offset c is exact; bit kOffsets: near
};
constexpr int kOffsets = 4;
__device__ __forceinline__ float offset_of(float off, int c, float bin) {
    return off + bin * (c == 0 ? 0.0f : c == 1 ? 0x1p-15f : c == 2 ? -0x1p-15f : 0x1p-14f);
}

// Copy the edges of axes a0 .. a0 + naxes - 1 into shared memory (all threads), with
// each axis's outer edges e_0 and e_bins replaced by NaN (see bin_of), and choose the
// mode; syncs. The guess and the bin are both non-decreasing in v, so the guess is
// at most one off everywhere if at every interior edge e_k it is k - 1 or more and
// just below it k or less, and it is the bin of every binary16 value if it is k or
// more at the smallest one >= e_k and k - 1 or less at the one before. A guess
// that misses that by its rounding at some edge is tried with its offset moved by
// a few 2^-15 of a bin.
template <int DT>
__device__ __forceinline__ int stage_edges(const HistLaunch& A, int a0, int naxes, float* s_edges, BinTable& T) {
    const int bins = A.bins, ne = naxes * (bins + 1);
    const float top = guess_top(bins), bin = 1.0f / (float)bins;
    const int all = DT == kF16 ? (2 << kOffsets) - 1 : 1 << kOffsets;
    if (threadIdx.x < kMaxVars) T.ok[threadIdx.x] = all;
    __syncthreads();
    for (int i = threadIdx.x; i < ne; i += blockDim.x) {
        const int a = i / (bins + 1), k = i - a * (bins + 1), src = a0 * (bins + 1) + i;
        float e = __int_as_float(0x7fffffff);
        if (k != 0 && k != bins) {
            e = A.edges ? __ldg(A.edges + src) : A.edges_inl[src];
            const float scale = A.guess_scale[a0 + a], off = A.guess_off[a0 + a];
            int ok = bin_guess(top, e, scale, off) >= k - 1 &&
                     bin_guess(top, nextafterf(e, -INFINITY), scale, off) <= k ? 1 << kOffsets : 0;
            if (DT == kF16) {
                const unsigned up = __half_as_ushort(__float2half_ru(e)), dn = half_prev(up);
                const float vu = __half2float(__ushort_as_half((unsigned short)up));
                const float vd = __half2float(__ushort_as_half((unsigned short)dn));
#pragma unroll 1
                for (int c = 0; c < kOffsets; ++c)
                    if (bin_guess(top, vu, scale, offset_of(off, c, bin)) >= k && bin_guess(top, vd, scale, offset_of(off, c, bin)) < k)
                        ok |= 1 << c;
            }
            if (ok != all) atomicAnd(&T.ok[a], ok);
        }
        s_edges[i] = e;
    }
    __syncthreads();
    bool near = true, exact = DT == kF16;
    for (int a = 0; a < naxes; ++a) {
        const int av = A.avar[a0 + a];
        near = near && (T.ok[a] >> kOffsets);
        exact = exact && av < kPosAxisBase && (T.ok[a] & ((1 << kOffsets) - 1));
    }
    if (threadIdx.x < naxes) {
        const int c = exact ? __ffs(T.ok[threadIdx.x]) - 1 : 0;
        T.off[threadIdx.x] = offset_of(A.guess_off[a0 + threadIdx.x], c, bin);
    }
    __syncthreads();
    return exact ? kBinExact : near ? kBinNear : kBinWalk;
}

// Row geometry shared by both kernels: the x range of the r-th row (y, z) inside the
// outer sphere, |2x + 1 - n| <= m, and the range [ca, cb] of its cells inside the
// inner sphere (empty when ca > cb); false when the whole row lies outside.
// Rows are taken in z-planes whose y order is rotated by z * rot. With a row
// counter the vector kernel's warps take the next untaken rows whenever they
// finish (rot = 0): they finish together whatever the brush leaves in each row.
// Without one they take rows by warp stride, and rot is a golden-ratio fraction
// of n: a stride that is a multiple of n would otherwise give every warp one y
// -- all its rows long chords through the shell or all short ones near the
// outer sphere. The scalar kernel keeps the plain order (rot = 0).
struct RowSpan {
    int y, z, syz, xa, xb, ca, cb;
    float cy, cz;
    size_t base;                   // (z n + y) n
    uint32_t srow;                 // first sub-brick id of the row's sub-brick row
};

__device__ __forceinline__ bool row_span(const HistLaunch& A, int r, RowSpan& R) {
    const int n = A.n;
    R.z = r / n;
    R.y = r - R.z * n;
    if (A.rot) R.y += (R.z * A.rot) % n;                    // z * rot < 2^24 for n <= 4096
    if (R.y >= n) R.y -= n;
    const int dy = 2 * R.y + 1 - n, dz = 2 * R.z + 1 - n;
    R.syz = dy * dy + dz * dz;                              // < 2^31 for n <= 4096
    if (R.syz > A.s_out) return false;
    const int m = isqrt_floor(A.s_out - R.syz);
    R.xa = max(0, (n - m) / 2);
    R.xb = min(n - 1, (n - 1 + m) / 2);
    R.ca = 1;
    R.cb = 0;
    const int din = A.s_in - R.syz;                         // cells with dx^2 < din fail the shell test
    if (din > 0) {
        const int mi = isqrt_floor(din - 1);                // |2x + 1 - n| <= mi
        R.ca = max(0, (n - mi) / 2);
        R.cb = min(n - 1, (n - 1 + mi) / 2);
    }
    R.cy = A.use_pos ? cell_centre_rn(R.y, n) : 0.0f;
    R.cz = A.use_pos ? cell_centre_rn(R.z, n) : 0.0f;
    R.base = ((size_t)R.z * n + R.y) * n;
    R.srow = ((uint32_t)(R.z >> 2) * A.nsb + (uint32_t)(R.y >> 2)) * A.nsb;
    return true;
}

// The warp's row after r (r = its warp index - nwarps: its first row). With a
// row counter, warps take batches of kRowBatch neighbouring rows: warp w starts
// with batch w, and every later batch is nwarps + the counter's next value,
// taken one batch ahead in lane 0's rq (first_batch gives its initial value) so
// that the atomic's latency hides behind a batch's work, and few enough atomics
// meet at the one address. Without one, rows go by warp stride. Every lane calls
// it; the result is the same in all of them.
constexpr int kRowBatch = 2;

__device__ __forceinline__ unsigned first_batch(const HistLaunch& A, int gwarp) {
    return A.rowctr ? (unsigned)gwarp : 0u;
}

__device__ __forceinline__ int take_row(const HistLaunch& A, int r, int rows, int nwarps, int lane, unsigned& rq) {
    if (!A.rowctr) return r + nwarps;
    if (r >= A.item0 && (r - A.item0 + 1) % kRowBatch != 0) return r + 1;
    const int t = A.item0 + (int)__shfl_sync(kFull, rq, 0) * kRowBatch;
    if (t < rows && lane == 0) rq = (unsigned)nwarps + atomicAdd(A.rowctr, 1u);
    return t;
}

// Whether cell x of row R is counted before any brushed value is read: in the
// shell (integers), in an active sub-brick when the activity is given (a vertex
// of an inactive sub-brick fails the brush or lies outside the shell), and
// inside the position brush at the cell centre.
__device__ __forceinline__ bool cell_geometry_passes(const HistLaunch& A, const RowSpan& R, int x) {
    const int dx = 2 * x + 1 - A.n;
    const int sh = dx * dx + R.syz;
    if (!(sh >= A.s_in && sh <= A.s_out)) return false;
    if (A.sactive) {
        const uint32_t sid = R.srow + (uint32_t)(x >> 2);
        if (!((__ldg(A.sactive + (sid >> 5)) >> (sid & 31)) & 1u)) return false;
    }
    if (A.pmask) {
        BrushArgs pb;
#pragma unroll
        for (int a = 0; a < kNumPos; ++a) { pb.plo[a] = A.plo[a]; pb.phi[a] = A.phi[a]; }
        pb.pmask = A.pmask;
        const float cx = cell_centre_rn(x, A.n);
        if (!pos_pass(cx, R.cy, R.cz, dot3_rn(cx, R.cy, R.cz, cx, R.cy, R.cz), pb)) return false;
    }
    return true;
}

// Scalar kernel: any grid edge, any alignment, any number of axes. A warp walks
// one x-row of cells (lanes over x, two cells per lane in flight); persistent
// grid, rows by warp stride in their plain order (the launch gives it rot = 0 and
// no row counter: either costs this latency-bound kernel registers and time).
template <int DT>
__global__ void __launch_bounds__(kHistThreads) k_hist_scalar(const __grid_constant__ HistLaunch A) {
    extern __shared__ float s_edges[];
    __shared__ BinTable T;
    // (without the check against binary16 values, which the near form here does not need: the table's
    // staging is a third of a small call, 65^3 FP16 24.5 -> 19.0 us)
    const int mode = stage_edges<kF32>(A, 0, A.naxes, s_edges, T);
    const float top = guess_top(A.bins);

    const int lane = threadIdx.x & 31;
    const int n = A.n;
    const int rows = n * n;
    const int gwarp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int nwarps = (int)((gridDim.x * blockDim.x) >> 5);
    const int bins = A.bins;
    const size_t plane = (size_t)n * n * n;
    uint32_t* const out = A.out + (size_t)(blockIdx.x % (unsigned)A.nout) * (A.naxes - 1) * bins * bins;

    for (int r = gwarp; r < rows; r += nwarps) {
        RowSpan R;
        if (!row_span(A, r, R)) continue;
        for (int x0 = R.xa; x0 <= R.xb; x0 += 64) {
            bool keep[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int x = x0 + lane + 32 * j;
                keep[j] = x <= R.xb && cell_geometry_passes(A, R, x);
            }
            // brushed variables first, all loads in flight together
            float bv[2][kMaxVars];
#pragma unroll
            for (int k = 0; k < kMaxVars; ++k) {
                if (k >= A.nbr) break;
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    bv[j][k] = keep[j] ? load_cell<DT>(A.cells, A.bvar[k] * plane + R.base + x0 + lane + 32 * j) : 0.0f;
            }
#pragma unroll
            for (int k = 0; k < kMaxVars; ++k) {
                if (k >= A.nbr) break;
#pragma unroll
                for (int j = 0; j < 2; ++j) keep[j] = keep[j] && bv[j][k] >= A.blo[k] && bv[j][k] <= A.bhi[k];
            }
            if (__ballot_sync(kFull, keep[0] || keep[1]) == 0u) continue;
            // axis values of the cells that pass (brushed ones come back from L1), binned and
            // added in x order
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const unsigned km = __ballot_sync(kFull, keep[j]);
                if (km == 0u) continue;
                const int x = x0 + lane + 32 * j;
                float cx = 0.0f, cr2 = 0.0f;
                if (A.use_pos && keep[j]) {
                    cx = cell_centre_rn(x, n);
                    cr2 = dot3_rn(cx, R.cy, R.cz, cx, R.cy, R.cz);
                }
                unsigned prev = 0u;
#pragma unroll
                for (int a = 0; a < kMaxVars; ++a) {
                    if (a >= A.naxes) break;
                    const int av = A.avar[a];
                    unsigned b = 0u;
                    if (keep[j]) {
                        const float v = av >= kPosAxisBase ? pos_axis(cx, R.cy, R.cz, cr2, av - kPosAxisBase)
                                                           : load_cell<DT>(A.cells, av * plane + R.base + x);
                        const float* e = s_edges + a * (bins + 1);
                        b = (unsigned)(mode != kBinWalk ? bin_of<kBinNear>(e, bins, top, v, A.guess_scale[a], T.off[a])
                                                        : bin_of<kBinWalk>(e, bins, top, v, A.guess_scale[a], T.off[a]));
                    }
                    if (a > 0) add_runs(out + (size_t)(a - 1) * bins * bins, prev * (unsigned)bins + b, keep[j], km, lane);
                    prev = b;
                }
            }
        }
    }
}

__device__ __forceinline__ __half2 u32_as_half2(unsigned u) {
    __half2 h;
    memcpy(&h, &u, sizeof(h));
    return h;
}

// Element j of a 16-byte chunk of FP32 values.
template <int DT> __device__ __forceinline__ float chunk_elem(const uint4& c, int j);
template <> __device__ __forceinline__ float chunk_elem<kF32>(const uint4& c, int j) {
    return __uint_as_float(j == 0 ? c.x : j == 1 ? c.y : j == 2 ? c.z : c.w);
}

// Asynchronous 16-byte global -> shared copies (no registers held while in
// flight); a group is waited for with cp.async.wait_group, a hardware wait.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_prev() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }

// One chunk row of the vector kernel: 32 lanes x VEC consecutive cells of row r
// starting at xw, and this lane's cells that pass the geometric tests.
struct ChunkRow {
    int r, xw;                     // r = -1: none
    RowSpan R;
    unsigned kb;
    unsigned rq;                   // with a row counter, lane 0: the row to take after this one
};


// Bits j of [0, VEC) with lo <= j <= hi.
template <int VEC>
__device__ __forceinline__ unsigned span_bits(int lo, int hi) {
    const int l = max(lo, 0), h = min(hi, VEC - 1);
    return l > h ? 0u : (2u << h) - (1u << l);
}

// Geometric keep bits of this lane's chunk (cells x0 .. x0 + VEC - 1, x0 any): in the
// shell (the row's ranges), in an active sub-brick when the activity is given, inside
// the position brush.
template <int VEC>
__device__ __forceinline__ unsigned chunk_geometry(const HistLaunch& A, const RowSpan& R, int x0) {
    unsigned kb = span_bits<VEC>(R.xa - x0, R.xb - x0) & ~span_bits<VEC>(R.ca - x0, R.cb - x0);
    if (kb && A.sactive) {
        // the activity of the sub-bricks that the chunk's cells lie in, from the first kept cell's on
        const int xs = x0 + __ffs(kb) - 1, s0 = xs >> 2;
        const uint32_t sid = R.srow + (uint32_t)s0;
        unsigned act = __ldg(A.sactive + (sid >> 5)) >> (sid & 31);
        const int more = min((x0 + 31 - __clz(kb)) >> 2, A.nsb - 1) - s0;   // to the last kept cell's
        if ((int)(sid & 31) + more > 31) act |= __ldg(A.sactive + (sid >> 5) + 1) << (32 - (sid & 31));
#pragma unroll
        for (int q = 0; q < VEC / 4 + 1; ++q)
            if (!((act >> q) & 1u)) kb &= ~span_bits<VEC>(4 * (s0 + q) - x0, 4 * (s0 + q) + 3 - x0);
    }
    if (kb && A.pmask) {
        BrushArgs pb;
#pragma unroll
        for (int a = 0; a < kNumPos; ++a) { pb.plo[a] = A.plo[a]; pb.phi[a] = A.phi[a]; }
        pb.pmask = A.pmask;
#pragma unroll
        for (int j = 0; j < VEC; ++j) {
            const float cx = cell_centre_rn(x0 + j, A.n);
            if (((kb >> j) & 1u) && !pos_pass(cx, R.cy, R.cz, dot3_rn(cx, R.cy, R.cz, cx, R.cy, R.cz), pb))
                kb &= ~(1u << j);
        }
    }
    return kb;
}

// The warp's next chunk row after (r, xw): the next chunk of the same row, else the
// first chunk of the next row (by warp stride) that meets the outer sphere and holds
// a cell passing the geometric tests in some lane.
template <int VEC>
__device__ __forceinline__ void next_chunk_row(const HistLaunch& A, int nwarps, int lane, ChunkRow& C) {
    constexpr int CH = 32 * VEC;
    const int rows = A.items;
    int r = C.r, xw = C.xw + CH;
    bool have_row = r >= A.item0;
    for (;;) {
        if (!have_row || xw > C.R.xb) {
            r = take_row(A, r, rows, nwarps, lane, C.rq);
            if (r >= rows) { C.r = -1; C.kb = 0u; return; }
            if (!row_span(A, r, C.R)) { have_row = false; continue; }
            have_row = true;
            // chunks start on 16-byte boundaries of the plane: before x = 0 of the row when the edge is
            // no multiple of VEC (the cells in front are another row's)
            const int lead = (int)(C.R.base & (VEC - 1));
            xw = ((C.R.xa + lead) & ~(VEC - 1)) - lead;
        }
        const unsigned kb = chunk_geometry<VEC>(A, C.R, xw + lane * VEC);
        if (__ballot_sync(kFull, kb != 0u) != 0u) {
            C.r = r;
            C.xw = xw;
            C.kb = kb;
            return;
        }
        xw += CH;
    }
}

// How a warp of the vector kernel walks the cells: chunk rows of whole x-rows, or
// groups of active sub-bricks. Both hold the current chunk's geometric keep bits kb,
// this lane's element offset off (its VEC consecutive cells) and, for position
// axes, the centre of listed cell c (lane c / VEC, cell c % VEC).
template <int VEC>
struct RowWalk {
    ChunkRow C;
    int nwarps;
    unsigned kb;
    size_t off;
    __device__ __forceinline__ void start(const HistLaunch& A, int gwarp, int nw) {
        nwarps = nw;
        C.r = A.item0 + gwarp - nw;
        C.xw = 0;
        C.rq = first_batch(A, gwarp);
    }
    __device__ __forceinline__ bool more() const { return C.r >= 0; }
    __device__ __forceinline__ void next(const HistLaunch& A, int lane) {
        next_chunk_row<VEC>(A, nwarps, lane, C);
        kb = C.kb;
        off = C.R.base + C.xw + lane * VEC;
    }
    __device__ __forceinline__ void centre(const HistLaunch& A, int c, float& cx, float& cy, float& cz) const {
        cx = cell_centre_rn(C.xw + c, A.n);
        cy = C.R.cy;
        cz = C.R.cz;
    }
};

// For listed calls: groups of 2 VEC / 4 sub-bricks that are neighbours in x, with an active one among
// them: 2 VEC x 4 x 4 cells, lane 2 r + h the h-th half of row r (y = r % 4, z =
// r / 4), taken from segments of 8 sub-bricks of a sub-brick row. Under a brush the
// active sub-bricks are few and short in x: a chunk row of 32 VEC cells of one
// x-row has a third of its lanes at work, a group two thirds, and no row needs its
// sphere's chord (256^3 FP16, 3 brushed variables: 42 -> 25 M warp instructions). The
// segments come in batches, their bits loaded at once (512^3: 352 -> 214 us).
template <int VEC>
struct GroupWalk {
    static constexpr int kSubs = VEC / 2;              // sub-bricks of a group
    int nwarps, base;                                  // first segment of the batch (-1: no more)
    unsigned rq, segs, mine, bits, kb;                 // segments left in the batch, lane j's: the bits of segment j
    int sx, sy, sz;                                    // first sub-brick of the segment's bits, and its row
    int gx;                                            // first sub-brick of the current group
    size_t off;
    __device__ __forceinline__ void start(const HistLaunch& A, int gwarp, int nw) {
        nwarps = nw;
        base = 0;
        rq = (unsigned)gwarp;
        segs = bits = 0u;
    }
    __device__ __forceinline__ bool more() const { return base >= 0; }
    // The activity bits of the warp's next batch of segments, one segment per lane: the batch's
    // number was taken from the row counter a batch ahead, and
    // empty segments cost a bit each instead of a load's latency.
    __device__ __forceinline__ bool next_batch(const HistLaunch& A, int lane) {
        const unsigned b = __shfl_sync(kFull, rq, 0);
        const long long first = A.item0 + (long long)b * A.batch;
        if (first >= A.items) {
            base = -1;
            return false;
        }
        base = (int)first;
        if (lane == 0) rq = (unsigned)nwarps + atomicAdd(A.rowctr, 1u);
        mine = 0u;
        const int seg = base + lane, per_row = (A.nsb + 7) >> 3;
        if (lane < A.batch && seg < A.items) {
            const int row = seg / per_row, x = (seg - row * per_row) << 3;
            const uint32_t id = (uint32_t)row * A.nsb + x;
            const int here = min(8, A.nsb - x);        // sub-bricks of the segment
            mine = __ldg(A.sactive + (id >> 5)) >> (id & 31);
            if ((int)(id & 31) + here > 32) mine |= __ldg(A.sactive + (id >> 5) + 1) << (32 - (id & 31));
            mine &= (1u << here) - 1u;
        }
        segs = __ballot_sync(kFull, mine != 0u);
        return true;
    }
    __device__ __forceinline__ void next(const HistLaunch& A, int lane) {
        const int n = A.n, nsb = A.nsb, per_row = (nsb + 7) >> 3;
        kb = 0u;
        for (;;) {
            if (bits == 0u) {                          // uniform over the warp
                while (segs == 0u)
                    if (!next_batch(A, lane)) return;
                const int j = __ffs(segs) - 1;
                segs &= segs - 1u;
                bits = __shfl_sync(kFull, mine, j);
                const int row = (base + j) / per_row;
                sx = (base + j - row * per_row) << 3;
                sz = row / nsb;
                sy = row - sz * nsb;
            }
            const int g = (__ffs(bits) - 1) & ~(kSubs - 1);
            const unsigned act = (bits >> g) & ((1u << kSubs) - 1u);
            bits &= ~(((1u << kSubs) - 1u) << g);
            gx = sx + g;
            const int half = lane & 1, row = lane >> 1;
            const int x = gx * 4 + half * VEC, y = sy * 4 + (row & 3), z = sz * 4 + (row >> 2);
            if (x < n) {                               // n is a multiple of VEC and of 4
#pragma unroll
                for (int q = 0; q < VEC / 4; ++q)
                    if ((act >> (half * (VEC / 4) + q)) & 1u) kb |= 0xfu << (4 * q);
            }
            const int dy = 2 * y + 1 - n, dz = 2 * z + 1 - n, syz = dy * dy + dz * dz;
            if (kb) {
                // |2x + 1 - n| over the run: all of it in the shell, or cell by cell
                const int d0 = 2 * x + 1 - n, d1 = d0 + 2 * (VEC - 1);
                const int far = max(abs(d0), abs(d1)), near = d0 > 0 ? d0 : (d1 < 0 ? -d1 : 0);
                if (!(near * near + syz >= A.s_in && far * far + syz <= A.s_out)) {
#pragma unroll
                    for (int q = 0; q < VEC; ++q) {
                        const int d = d0 + 2 * q, sh = d * d + syz;
                        if (!(sh >= A.s_in && sh <= A.s_out)) kb &= ~(1u << q);
                    }
                }
            }
            if (kb && A.pmask) {
                BrushArgs pb;
#pragma unroll
                for (int a = 0; a < kNumPos; ++a) { pb.plo[a] = A.plo[a]; pb.phi[a] = A.phi[a]; }
                pb.pmask = A.pmask;
                const float cy = cell_centre_rn(y, n), cz = cell_centre_rn(z, n);
#pragma unroll
                for (int q = 0; q < VEC; ++q) {
                    const float cx = cell_centre_rn(x + q, n);
                    if (((kb >> q) & 1u) && !pos_pass(cx, cy, cz, dot3_rn(cx, cy, cz, cx, cy, cz), pb)) kb &= ~(1u << q);
                }
            }
            if (__ballot_sync(kFull, kb != 0u) != 0u) {
                off = ((size_t)z * n + y) * n + x;
                return;
            }
        }
    }
    __device__ __forceinline__ void centre(const HistLaunch& A, int c, float& cx, float& cy, float& cz) const {
        const int l = c / VEC, row = l >> 1;
        cx = cell_centre_rn(gx * 4 + (l & 1) * VEC + c % VEC, A.n);
        cy = cell_centre_rn(sy * 4 + (row & 3), A.n);
        cz = cell_centre_rn(sz * 4 + (row >> 2), A.n);
    }
};

// One binning round of the vector kernel: lane l holds a cell iff kept (the kept lanes
// are a prefix) with its axis values val[a]; bn[a] receives their bins. NAX: the number of
// axes, 0: A.naxes.
template <int NAX, int MODE>
__device__ __forceinline__ void bins_of(const HistLaunch& A, const float* s_edges, const BinTable& T,
                                        const float (&val)[kMaxVars], unsigned (&bn)[kMaxVars]) {
    const float top = guess_top(A.bins);
#pragma unroll
    for (int a = 0; a < (NAX ? NAX : kMaxVars); ++a) {
        bn[a] = 0u;
        if (!NAX && a >= A.naxes) continue;
        bn[a] = (unsigned)bin_of<MODE>(s_edges + a * (A.bins + 1), A.bins, top, val[a], A.guess_scale[a], T.off[a]);
    }
}

// Direct counts by tuple: a lane whose bin tuple differs from its left neighbour's starts a run
// and adds the run's length to each adjacent-axis pair (one L2 atomic per pair and
// run; km: mask of the kept lanes).
__device__ __forceinline__ void add_tuples(const HistLaunch& A, uint32_t* out, const unsigned (&bn)[kMaxVars], bool kept,
                                           unsigned km, int lane) {
    const int naxes = A.naxes, bins = A.bins;
    bool same = lane > 0;
#pragma unroll
    for (int w = 0; w < 3; ++w) {
        if (3 * w >= naxes) break;
        unsigned packed = 0u;                               // three bins, 10 bits each
#pragma unroll
        for (int a = 3 * w; a < 3 * w + 3 && a < kMaxVars; ++a) packed |= bn[a] << (10 * (a % 3));
        const unsigned left = __shfl_up_sync(kFull, packed, 1);   // by every lane: outside the condition
        same = same && left == packed;
    }
    const bool head = kept && !same;
    const unsigned hm = __ballot_sync(kFull, head);
    if (head) {
        const unsigned after = lane == 31 ? 0u : (kFull << (lane + 1));
        const unsigned stop = (hm | ~km) & after;            // next run start or the last kept lane
        const unsigned len = (unsigned)((stop ? __ffs(stop) - 1 : 32) - lane);
        const unsigned bb = (unsigned)(bins * bins);
#pragma unroll
        for (int a = 1; a < kMaxVars; ++a) {
            if (a >= naxes) break;
            atomicAdd(out + ((a - 1) * bb + bn[a - 1] * (unsigned)bins + bn[a]), len);
        }
    }
}

// The same by pair: runs of each adjacent-axis pair on its own.
__device__ __forceinline__ void add_pairs(const HistLaunch& A, uint32_t* out, const unsigned (&bn)[kMaxVars], bool kept,
                                          unsigned km, int lane) {
    const unsigned bins = (unsigned)A.bins;
#pragma unroll
    for (int a = 1; a < kMaxVars; ++a) {
        if (a >= A.naxes) break;
        add_runs(out + (size_t)(a - 1) * bins * bins, bn[a - 1] * bins + bn[a], kept, km, lane);
    }
}

// A warp's place in the list of binned cells. The list is made of chunks of 32 units of
// 8 cells, each axis's bins contiguous within a chunk (bytes up to 256 bins, else 16
// bits), with one mask byte per unit. A warp takes list_batch chunks at a time from a
// counter, the first ones when it has a cell to list.
constexpr int kListCells = 256;
constexpr unsigned kListBatch = 4;                           // most chunks taken at a time
struct ListSlots {
    unsigned chunk, left;                                    // current chunk, chunks of its batch after it
    unsigned fill;                                           // used cells (k_hist_bins: used units) of the chunk
    unsigned after;                                          // the next batch (lane 0), taken with the last
    bool early;                                              // chunk of its batch, when batches have several
    __device__ __forceinline__ void start(unsigned full) {
        chunk = ~0u;
        left = after = 0u;
        fill = full;
        early = false;
    }
    __device__ __forceinline__ void advance(const HistLaunch& A, int lane) {
        if (left) {
            --left;
            ++chunk;
        } else {
            if (!early && lane == 0) after = atomicAdd(A.list_next, A.list_batch);
            chunk = __shfl_sync(kFull, after, 0);
            left = A.list_batch - 1u;
            early = false;
            if (left) return;
        }
        if (left == 0u && A.list_batch > 1u) {
            early = true;
            if (lane == 0) after = atomicAdd(A.list_next, A.list_batch);
        }
    }
    __device__ __forceinline__ void mask(const HistLaunch& A, unsigned c, unsigned unit, unsigned bits) const {
        if (c < A.list_chunks) A.list_mask[(size_t)c * 32 + unit] = (unsigned char)bits;
    }
    // masks of the chunk's units: the first fill cells
    __device__ __forceinline__ void close(const HistLaunch& A, int lane) {
        mask(A, chunk, lane, (1u << min(8, max(0, (int)fill - 8 * lane))) - 1u);
    }
    // the rest of the chunk from unit u on, the rest of its batch and the batch taken early are empty
    __device__ __forceinline__ void finish(const HistLaunch& A, unsigned u, int lane) {
        if (lane >= (int)u) mask(A, chunk, lane, 0u);
        for (unsigned i = 1; i <= left; ++i) mask(A, chunk + i, lane, 0u);
        const unsigned next = __shfl_sync(kFull, after, 0);
        for (unsigned i = 0; early && i < A.list_batch; ++i) mask(A, next + i, lane, 0u);
    }
    // a round of up to 32 cells, take of them kept (a prefix of the lanes)
    template <int NAX>
    __device__ __forceinline__ void put(const HistLaunch& A, const unsigned (&bn)[kMaxVars], bool kept, int take, int lane) {
        const int naxes = NAX ? NAX : A.naxes;
        if (fill + 32 > kListCells) {
            close(A, lane);
            advance(A, lane);
            fill = 0u;
        }
        if (kept && chunk < A.list_chunks) {                 // the list is sized for every in-shell cell
            const size_t at = (size_t)chunk * (size_t)(naxes * kListCells) + fill + lane;
#pragma unroll
            for (int a = 0; a < (NAX ? NAX : kMaxVars); ++a) {
                if (!NAX && a >= naxes) break;
                if (A.bins <= 256) A.list[at + a * kListCells] = (unsigned char)bn[a];
                else reinterpret_cast<unsigned short*>(A.list)[at + a * kListCells] = (unsigned short)bn[a];
            }
        }
        fill += (unsigned)take;
    }
};

// Vector kernel (even grid edge, 16-byte aligned planes, at most kMaxVars load slots). While a warp tests and bins one chunk of its walk (32 lanes x
// 16 bytes, 8 FP16 or 4 FP32 cells per lane) it has the next one's slots copied
// into its other shared buffer with cp.async (only chunks with a cell that passes
// the shell, sub-brick and position tests), so HBM latency hides behind the
// binning and no registers wait on loads. All brushed slots are tested (FP16: two
// cells at a time against exact binary16 bounds); the surviving cells go into a
// compact list (warp prefix sum) from which the warp bins 32 cells per round,
// reading the axis values from the buffer. LIST: the bins go into a list that
// k_hist_count turns into counts; else straight into L2 atomics. Persistent grid;
// rows or segments from the row counter or by warp stride; the edge table is staged
// once per resident block. NAX: 0 with a position axis or a position brush, else the
// number of axes, or -1 for any (fixed loops have no checks and immediate offsets: 89 -> 82
// us at 250^3 FP16 by groups).
template <int DT, typename Walk, int NAX, bool LIST>
__global__ void __launch_bounds__(kHistVecThreads, 2) k_hist(const __grid_constant__ HistLaunch A) {
    constexpr int VEC = DT == kF16 ? 8 : 4;
    constexpr int kMost = NAX > 0 ? NAX : kMaxVars;
    constexpr bool kCarry = DT == kF16 && NAX != 0;            // FP16: a remainder waits for the next chunk
    extern __shared__ __align__(16) unsigned char s_raw[];
    __shared__ BinTable T;
    float* s_edges = reinterpret_cast<float*>(s_raw);
    const int ne16 = (A.naxes * (A.bins + 1) + 3) & ~3;
    const int nslot = A.nslot, naxes = NAX > 0 ? NAX : A.naxes;
    const int buf_bytes = nslot * 512;                          // one chunk of every slot
    unsigned char* s_warp = s_raw + sizeof(float) * ne16 + (size_t)(threadIdx.x >> 5) * (2 * buf_bytes + 256);
    unsigned char* s_list = s_warp + 2 * buf_bytes;
    const int mode = stage_edges<DT>(A, 0, naxes, s_edges, T);

    const int lane = threadIdx.x & 31;
    const uint32_t sbr = A.sbr;
    uint32_t* const out = LIST ? nullptr : A.out + (size_t)(blockIdx.x % (unsigned)A.nout) * (naxes - 1) * A.bins * A.bins;

    // copies of chunk W into buffer b (lanes whose cells all fail copy nothing)
    auto prefetch = [&](const Walk& W, int b) {
        if (W.more() && W.kb) {
            unsigned char* dst = s_warp + b * buf_bytes + lane * 16;
            const char* src = static_cast<const char*>(A.cells) + W.off * (16 / VEC);
#pragma unroll
            for (int s = 0; s < kMaxVars; ++s)
                if (s < NAX || (s < nslot && (NAX < 0 || A.svar[s] >= 0))) cp_async16(dst + s * 512, src + A.soff[s]);
        }
        cp_async_commit();
    };

    ListSlots slots;
    slots.start(kListCells);
    int q = 0;                                                  // carried cells, in lanes 0..q-1
    unsigned cpk[(kMost + 1) / 2] = {};                         // a carried cell's values, binary16 pairs

    Walk cur;
    cur.start(A, (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), (int)((gridDim.x * blockDim.x) >> 5));
    cur.kb = 0u;                                                // an empty chunk before the first
    bool have = true;
    int b = 0;
    for (;;) {                                                  // no chunk left: only the last carried cells are
        if (!have && q == 0) break;
        Walk nxt = cur;
        const unsigned char* buf = s_warp + b * buf_bytes;
        int total = 0;
        if (have) {
            nxt.next(A, lane);
            prefetch(nxt, b ^ 1);
            cp_async_wait_prev();                               // this chunk's copies have landed
            __syncwarp();
            unsigned kb = cur.kb;
            // brushed slots
            if constexpr (DT == kF16) {
                unsigned acc[4] = {kFull, kFull, kFull, kFull};
#pragma unroll
                for (int s = 0; s < kMaxVars; ++s) {
                    if ((sbr >> s) & 1u) {
                        const uint4 v = *reinterpret_cast<const uint4*>(buf + s * 512 + lane * 16);
                        const __half2 lo2 = u32_as_half2(A.slo_h2[s]), hi2 = u32_as_half2(A.shi_h2[s]);
                        const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            acc[i] &= __hge2_mask(u32_as_half2(w[i]), lo2) & __hle2_mask(u32_as_half2(w[i]), hi2);
                    }
                }
                unsigned pass = 0u;
#pragma unroll
                for (int i = 0; i < 4; ++i) pass |= ((acc[i] & 1u) | ((acc[i] >> 15) & 2u)) << (2 * i);
                kb &= pass;
            } else {
#pragma unroll
                for (int s = 0; s < kMaxVars; ++s) {
                    if ((sbr >> s) & 1u) {
                        const uint4 v = *reinterpret_cast<const uint4*>(buf + s * 512 + lane * 16);
                        const float lo = A.slo[s], hi = A.shi[s];
#pragma unroll
                        for (int j = 0; j < VEC; ++j) {
                            const float x = chunk_elem<DT>(v, j);
                            if (!(x >= lo && x <= hi)) kb &= ~(1u << j);
                        }
                    }
                }
            }
            // compact list of the surviving cells (lane * VEC + j) in order: the exclusive
            // prefix of the per-lane counts from an inclusive shuffle scan
            const unsigned cnt = (unsigned)__popc(kb);
            unsigned inc = cnt;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned t = __shfl_up_sync(kFull, inc, d);
                if (lane >= d) inc += t;
            }
            int pos = (int)(inc - cnt);
            total = (int)__shfl_sync(kFull, inc, 31);
#pragma unroll
            for (int j = 0; j < VEC; ++j)
                if ((kb >> j) & 1u) s_list[pos++] = (unsigned char)(lane * VEC + j);
            __syncwarp();
        }
        // bin the surviving cells 32 per round. FP16 without position axes carries a remainder
        // of fewer than 32 cells to the next chunk (their values in the lanes' registers),
        // so that sparse chunks still fill whole rounds
        int consumed = 0;
#pragma unroll 1
        for (;;) {
            const int avail = q + total - consumed;
            if (avail == 0) break;
            if (kCarry && have && avail < 32) {
                if (lane >= q && lane < avail) {
                    const int c = s_list[consumed + lane - q];
#pragma unroll
                    for (int a = 0; a < kMost; ++a) {
                        if (NAX < 0 && a >= naxes) break;
                        const unsigned hb = reinterpret_cast<const unsigned short*>(buf + a * 512)[c];
                        cpk[a >> 1] = (cpk[a >> 1] & (0xffff0000u >> (16 * (a & 1)))) | (hb << (16 * (a & 1)));
                    }
                }
                q = avail;
                break;
            }
            const int take = min(32, avail);
            const bool kept = lane < take;
            const unsigned km = take == 32 ? kFull : (1u << take) - 1u;
            float val[kMaxVars];
#pragma unroll
            for (int a = 0; a < kMaxVars; ++a) val[a] = 0.0f;
            if (kCarry && kept && lane < q) {                   // a carried cell
#pragma unroll
                for (int a = 0; a < kMost; ++a)
                    val[a] = __half2float(__ushort_as_half((unsigned short)(cpk[a >> 1] >> (16 * (a & 1)))));
            } else if (kept) {
                const int c = s_list[consumed + lane - q];
                float cx = 0.0f, cy = 0.0f, cz = 0.0f, cr2 = 0.0f;
                if (!NAX && A.use_pos) {
                    cur.centre(A, c, cx, cy, cz);
                    cr2 = dot3_rn(cx, cy, cz, cx, cy, cz);
                }
#pragma unroll
                for (int a = 0; a < kMost; ++a) {
                    if (NAX <= 0 && a >= naxes) break;
                    if (!NAX && A.avar[a] >= kPosAxisBase)
                        val[a] = pos_axis(cx, cy, cz, cr2, A.avar[a] - kPosAxisBase);
                    else if (DT == kF16)
                        val[a] = __half2float(__ushort_as_half(reinterpret_cast<const unsigned short*>(buf + a * 512)[c]));
                    else
                        val[a] = reinterpret_cast<const float*>(buf + a * 512)[c];
                }
            }
            unsigned bn[kMaxVars] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
            if (DT == kF16 && NAX && mode == kBinExact) bins_of<(NAX > 0 ? NAX : 0), kBinExact>(A, s_edges, T, val, bn);
            else if (mode != kBinWalk) bins_of<(NAX > 0 ? NAX : 0), kBinNear>(A, s_edges, T, val, bn);
            else bins_of<(NAX > 0 ? NAX : 0), kBinWalk>(A, s_edges, T, val, bn);
            if (LIST) slots.put<(NAX > 0 ? NAX : 0)>(A, bn, kept, take, lane);
            else if (A.by_pair) add_pairs(A, out, bn, kept, km, lane);
            else add_tuples(A, out, bn, kept, km, lane);
            consumed += take - q;
            q = 0;
        }
        if (!have) break;
        __syncwarp();                                           // buffer b and the list are reused next
        cur = nxt;
        have = cur.more();
        b ^= 1;
    }
    if (LIST) {
        slots.close(A, lane);
        slots.finish(A, 32u, lane);
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}

// Lists the bins of every in-shell cell (no brush, no position axes; even grid edge,
// 16-byte aligned planes). A warp takes ROWS neighbouring rows and walks them side by side,
// 32 / ROWS lanes x 8 cells of each: the rows' geometry is computed at once, and 9 in 10
// lanes have cells (a whole warp per row: 2 in 3). Nothing is compacted: a lane
// bins its 8 cells straight from 16-byte loads, six axes (FP32: three) in flight, and
// stores a unit's bins of an axis with one store; cells outside the shell at the
// ends of a row stay unset in the unit's mask. Bound by HBM with its three instructions
// per value (205 -> 75 per 32 cells of 6 axes). ROWS is 8 on grids with at least five
// batches of 8 rows for each warp, else 4, which finish together sooner: whole calls at
// 512^3 FP16 with 1, 2, 4, 8 and 16 rows take 874, 698, 597, 535 and 627 us, at 256^3 FP32
// 161, 138, 136, 150 and 152.
template <int DT, int MODE, int ROWS, typename BIN>
__device__ __forceinline__ void list_rows(const HistLaunch& A, const float* s_edges, const BinTable& T) {
    constexpr int kUnit = 8, kBytes = DT == kF16 ? 16 : 32;    // cells and bytes of a unit
    constexpr int kLanes = 32 / ROWS;                          // of a row
    constexpr int kAxes = DT == kF16 ? 6 : 3;                  // axes in flight
    const int lane = threadIdx.x & 31;
    const float top = guess_top(A.bins);
    ListSlots slots;
    slots.start(32u);
    const unsigned nwarps = (gridDim.x * blockDim.x) >> 5;
    unsigned rq = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    for (;;) {
        const int first_row = A.item0 + (int)__shfl_sync(kFull, rq, 0) * ROWS;
        if (first_row >= A.items) break;
        if (lane == 0) rq = nwarps + atomicAdd(A.rowctr, 1u);
        const int r = first_row + lane / kLanes;
        RowSpan R;
        int x0 = 0;
        bool row = r < A.items && row_span(A, r, R);
        if (row) {
            // units start on 16-byte boundaries of the plane: before x = 0 of the row when the edge is no
            // multiple of 8 (the cells in front are another row's)
            const int lead = (int)(R.base & (kUnit - 1));
            x0 = ((R.xa + lead) & ~(kUnit - 1)) - lead + (lane & (kLanes - 1)) * kUnit;
        }
        for (; __ballot_sync(kFull, row && x0 <= R.xb) != 0u; x0 += kLanes * kUnit) {
            unsigned kb = 0u;
            if (row) kb = span_bits<kUnit>(R.xa - x0, R.xb - x0) & ~span_bits<kUnit>(R.ca - x0, R.cb - x0);
            // units with a cell to count, packed in lane order; those past the chunk's end go to the next
            const unsigned um = __ballot_sync(kFull, kb != 0u);
            if (um == 0u) continue;
            const unsigned first = slots.chunk;
            unsigned u = slots.fill + __popc(um & ((1u << lane) - 1u));
            slots.fill += __popc(um);
            if (slots.fill > 32u) {
                slots.advance(A, lane);
                slots.fill -= 32u;
            }
            const unsigned chunk = u < 32u ? first : slots.chunk;
            u &= 31u;
            if (!(kb && chunk < A.list_chunks)) continue;
            A.list_mask[(size_t)chunk * 32 + u] = (unsigned char)kb;
            const char* src = static_cast<const char*>(A.cells) + (R.base + x0) * (kBytes / kUnit);
            if (x0 + kLanes * kUnit <= R.xb)                   // the next step's lines on their way
                for (int a = 0; a < A.naxes; ++a)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(src + A.soff[a] + kLanes * kBytes));
            BIN* dst = reinterpret_cast<BIN*>(A.list) + (size_t)chunk * (size_t)(A.naxes * kListCells) + u * kUnit;
            for (int a0 = 0; a0 < A.naxes; a0 += kAxes) {
                uint4 v[kAxes][kBytes / 16];
#pragma unroll
                for (int i = 0; i < kAxes; ++i)
                    if (a0 + i < A.naxes) {
#pragma unroll
                        for (int h = 0; h < kBytes / 16; ++h)
                            v[i][h] = __ldg(reinterpret_cast<const uint4*>(src + A.soff[a0 + i]) + h);
                    }
#pragma unroll
                for (int i = 0; i < kAxes; ++i)
                    if (a0 + i < A.naxes) {
                        const int a = a0 + i;
                        const float* e = s_edges + a * (A.bins + 1);
                        const float scale = A.guess_scale[a], off = T.off[a];
                        unsigned bn[kUnit];                    // MODE kBinExact, bytes: in the low byte
#pragma unroll
                        for (int j = 0; j < kUnit; ++j) {
                            float x;
                            if constexpr (DT == kF16) {
                                const unsigned w = (j >> 1) == 0 ? v[i][0].x : (j >> 1) == 1 ? v[i][0].y : (j >> 1) == 2 ? v[i][0].z : v[i][0].w;
                                const float2 f = __half22float2(u32_as_half2(w));
                                x = (j & 1) ? f.y : f.x;
                            } else {
                                x = chunk_elem<kF32>(v[i][j >> 2], j & 3);
                            }
                            bn[j] = MODE == kBinExact ? bin_guess_raw(top, x, scale, off) : (unsigned)bin_of<MODE>(e, A.bins, top, x, scale, off);
                        }
                        if constexpr (sizeof(BIN) == 1) {
                            uint2 p;
                            p.x = __byte_perm(__byte_perm(bn[0], bn[1], 0x0040), __byte_perm(bn[2], bn[3], 0x0040), 0x5410);
                            p.y = __byte_perm(__byte_perm(bn[4], bn[5], 0x0040), __byte_perm(bn[6], bn[7], 0x0040), 0x5410);
                            *reinterpret_cast<uint2*>(dst + a * kListCells) = p;
                        } else {
                            *reinterpret_cast<uint4*>(dst + a * kListCells) =
                                make_uint4(__byte_perm(bn[0], bn[1], 0x5410), __byte_perm(bn[2], bn[3], 0x5410),
                                           __byte_perm(bn[4], bn[5], 0x5410), __byte_perm(bn[6], bn[7], 0x5410));
                        }
                    }
            }
        }
    }
    slots.finish(A, slots.fill, lane);
}

template <int DT, int ROWS, typename BIN>
__global__ void __launch_bounds__(kHistVecThreads, 2) k_hist_bins(const __grid_constant__ HistLaunch A) {
    extern __shared__ float s_edges[];
    __shared__ BinTable T;
    const int mode = stage_edges<DT>(A, 0, A.naxes, s_edges, T);
    if (DT == kF16 && mode == kBinExact) list_rows<DT, kBinExact, ROWS, BIN>(A, s_edges, T);
    else if (mode != kBinWalk) list_rows<DT, kBinNear, ROWS, BIN>(A, s_edges, T);
    else list_rows<DT, kBinWalk, ROWS, BIN>(A, s_edges, T);
}

// Counts of the listed cells. L2 atomics (5 per cell: neighbouring cells of a
// 256-bin histogram share few bin pairs) bound the calls on large grids; here one block
// per SM keeps the whole histogram of ONE adjacent-axis pair in its shared memory,
// reads two axes of the list's chunks (4 lanes to a chunk: lanes on neighbouring cells would
// meet at the same counters) and adds its non-zero counts to the output at the end. Pairs with hot bins take longer (adds of a warp to one counter serialise), so the
// warps take chunks from a counter per pair, and a block whose pair is done helps the one
// with the most chunks left (512^3, whole shell: 1138 -> 415 us). The bank conflicts and the
// instructions around the adds bound it: 4 lanes to a chunk and the keys' layout
// (count_pitch) 385 -> 327 us, predicated adds 327 -> 286 us.
//
// Counters are 32 bits where they fit (kPairBytes), else 16 bits, two to a word. A
// 16-bit count cannot overflow: the thread whose add makes it 2^15 moves 2^15 of it to
// the output, and should that take long, so does every thread that finds it at kFull16 or
// more, before it adds anything again (a thread adds the 8 cells of a unit at a time), so
// at most 8 kPairThreads single counts stand above kFull16 at any time. A move clears the
// counter's top bit: whoever finds it set owns the 2^15, and nobody tries twice. Adds of
// a warp to one 16-bit counter serialise (the hardware merges adds of 1 to 32-bit ones),
// so a warp with kSameUnits or more units of a single bin pair each adds those units
// whole (until a step of its batch has fewer: the check would cost smooth fields 1-2 %). A constant field at 512^3 FP16, 256 bins: 2138 us with every thread above
// 2^15 in a compare-and-swap loop, 1347 with the moves as they are, 506 with whole units
// (32-bit counters: 559); a smooth one 559, now 545.
constexpr int kPairThreads = 1024;
constexpr size_t kPairBytes = (size_t)200 << 10;    // shared memory for the counters of a block
constexpr unsigned kCountBatch = 8;                 // chunks a warp takes at a time, four lanes each
constexpr int kSameUnits = 8;                       // units of one bin pair in a warp from which they are added whole
constexpr unsigned kCountWorth = 64;                // chunks left per block for which changing the pair pays
                                                    // (its clearing and adding up take about 10 us)
constexpr size_t kListBytes = (size_t)512 << 20;    // bins of one slab
constexpr long long kListGrid = 1ll << 21, kListGridBrush = 1ll << 25;   // see hist_by_list
constexpr size_t kListWarps = 160 * 2 * kHistVecWarps;   // most warps of a launch that lists
constexpr int kListHead = 64;                       // bytes: row counter, chunks taken, chunks counted of each pair
constexpr unsigned kFull16 = 0xc000;                // see k_hist_count
static_assert(kFull16 + 8 * kPairThreads <= 0x10000, "16-bit counters");
static_assert(4 * (2 + kMaxVars - 1) <= kListHead, "list head");

struct CountArgs {
    const unsigned char* list;
    const unsigned char* mask;
    unsigned* head;                // [1]: chunks taken, [2 + p]: zeroed, chunks of pair p taken here
    unsigned chunks;               // chunks that fit
    int naxes, bins;
    uint32_t* out;
};

// Counter (x, y) of a pair has the key x * pitch + y. The pitch is 11 mod 32, so that the
// counters around one another, which cells around one another hit, lie in different banks;
// 16-bit counters k and k + words share a word for the same reason, not k and k + 1.
__host__ __device__ constexpr unsigned count_pitch(int bins) { return (unsigned)(bins + ((11 - bins) & 31)); }
__host__ __device__ constexpr unsigned count_words(int bins, bool wide) {
    const unsigned keys = (unsigned)bins * count_pitch(bins);
    return wide ? keys : (keys + 1u) / 2u;
}
// Most bins of 32-bit counters, and of 16-bit ones (of lists).
constexpr int kWideBins = 217, kListBins = 309;
static_assert(4 * count_words(kWideBins, true) <= kPairBytes && 4 * count_words(kWideBins + 1, true) > kPairBytes &&
              4 * count_words(kListBins, false) <= kPairBytes && 4 * count_words(kListBins + 1, false) > kPairBytes, "counters");

// Adds to a shared word (its shared-space address) if kept, predicated instead of branched around;
// its value before, or 0.
__device__ __forceinline__ unsigned add_if(bool kept, unsigned addr, unsigned v) {
    unsigned old = 0u;
    asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %3, 0;\n@p atom.shared.add.u32 %0, [%1], %2;\n}\n"
                 : "+r"(old) : "r"(addr), "r"(v), "r"((unsigned)kept) : "memory");
    return old;
}

// A 16-bit counter (top: its highest bit) that an add has taken from `was` to `at`: 2^15 of
// it to the output, if it is this thread's to move and still there.
__device__ __noinline__ void move_high(unsigned* word, unsigned top, unsigned was, unsigned at, uint32_t* out) {
    if (at >= 0x8000u && (was < 0x8000u || at >= kFull16))
        if (atomicAnd(word, ~top) & top) atomicAdd(out, 0x8000u);
}

template <typename BIN, bool WIDE>
__global__ void __launch_bounds__(kPairThreads, 1) k_hist_count(CountArgs A) {
    extern __shared__ unsigned s_hist[];
    __shared__ int s_pair;
    constexpr int kWords = 2 * (int)sizeof(BIN);              // 32-bit words of a unit
    const int bins = A.bins, npairs = A.naxes - 1, lane = threadIdx.x & 31;
    const unsigned pitch = count_pitch(bins), words = count_words(bins, WIDE);
    const unsigned chunks = min(A.head[1], A.chunks), s_base = (unsigned)__cvta_generic_to_shared(s_hist);
    int pair = (int)(blockIdx.x % (unsigned)npairs);
    for (;;) {
        uint32_t* const out = A.out + (size_t)pair * bins * bins;
        unsigned* taken = A.head + 2 + pair;
        for (unsigned i = threadIdx.x; i < words; i += kPairThreads) s_hist[i] = 0u;
        unsigned next = lane == 0 ? atomicAdd(taken, kCountBatch) : 0u;
        __syncthreads();
        for (;;) {
            const unsigned c0 = __shfl_sync(kFull, next, 0);
            if (c0 >= chunks) break;
            if (lane == 0) next = atomicAdd(taken, kCountBatch);
            const unsigned c = c0 + (lane >> 2);
            const bool any = c < chunks;
            unsigned m = 0u, a[kWords] = {}, b[kWords] = {};
            auto load = [&](int step, unsigned& m, unsigned (&a)[kWords], unsigned (&b)[kWords]) {
                const int unit = step * 4 + (lane & 3);
                m = __ldg(A.mask + (size_t)c * 32 + unit);
                const BIN* pa = reinterpret_cast<const BIN*>(A.list) + ((size_t)c * A.naxes + pair) * kListCells + unit * 8;
                if constexpr (sizeof(BIN) == 1) {
                    const uint2 x = __ldg(reinterpret_cast<const uint2*>(pa)), y = __ldg(reinterpret_cast<const uint2*>(pa + kListCells));
                    a[0] = x.x; a[1] = x.y; b[0] = y.x; b[1] = y.y;
                } else {
                    const uint4 x = __ldg(reinterpret_cast<const uint4*>(pa)), y = __ldg(reinterpret_cast<const uint4*>(pa + kListCells));
                    a[0] = x.x; a[1] = x.y; a[2] = x.z; a[3] = x.w; b[0] = y.x; b[1] = y.y; b[2] = y.z; b[3] = y.w;
                }
            };
            if (any) load(0, m, a, b);
            [[maybe_unused]] bool same = true;                   // the batch's steps so far had units of one bin pair
            for (int step = 0; step < 8; ++step) {
                unsigned mn = 0u, an[kWords] = {}, bn[kWords] = {};
                if (any && step < 7) load(step + 1, mn, an, bn);
                constexpr int kPer = 4 / (int)sizeof(BIN), kBits = 8 * (int)sizeof(BIN);
                if (!WIDE && same) {
                    // a unit of one bin pair: one add (see above)
                    constexpr unsigned kEach = sizeof(BIN) == 1 ? 0x01010101u : 0x00010001u;
                    unsigned differ = 0u;
#pragma unroll
                    for (int i = 1; i < kWords; ++i) differ |= (a[0] ^ a[i]) | (b[0] ^ b[i]);
                    same = __popc(__ballot_sync(kFull, differ == 0u && m != 0u)) >= kSameUnits;
                    if (same) {
                        const unsigned x = a[0] & ((1u << kBits) - 1u), y = b[0] & ((1u << kBits) - 1u);
                        if (differ == 0u && m && a[0] == x * kEach && b[0] == y * kEach) {
                            const unsigned k = x * pitch + y, sh = k >= words ? 16u : 0u, count = __popc(m);
                            unsigned* word = s_hist + (sh ? k - words : k);
                            const unsigned at = ((atomicAdd(word, count << sh) >> sh) & 0xffffu) + count;
                            if (at >= 0x8000u) move_high(word, 0x8000u << sh, at - count, at, out + x * bins + y);
                            m = 0u;
                        }
                    }
                }
                unsigned key[8], cur[8], over = 0u;
                if (WIDE || __any_sync(kFull, m != 0u)) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const unsigned x = (a[j / kPer] >> (kBits * (j % kPer))) & ((1u << kBits) - 1u);
                    const unsigned y = (b[j / kPer] >> (kBits * (j % kPer))) & ((1u << kBits) - 1u);
                    key[j] = x * pitch + y;
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const bool high = !WIDE && key[j] >= words;
                    const unsigned one = high ? 0x10000u : 1u;
                    cur[j] = add_if((m >> j) & 1u, s_base + 4u * (high ? key[j] - words : key[j]), one) + one;
                }
                if (!WIDE) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) over |= cur[j];
                    if (over & 0x80008000u) {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (((m >> j) & 1u) && (cur[j] & 0x80008000u)) {
                                const bool high = key[j] >= words;
                                const unsigned at = high ? cur[j] >> 16 : cur[j] & 0xffffu;
                                move_high(s_hist + (high ? key[j] - words : key[j]), high ? 0x80000000u : 0x8000u, at - 1u, at,
                                          out + (key[j] / pitch) * bins + key[j] % pitch);
                            }
                    }
                }
                }
                m = mn;
#pragma unroll
                for (int i = 0; i < kWords; ++i) { a[i] = an[i]; b[i] = bn[i]; }
            }
        }
        __syncthreads();
        for (unsigned i = threadIdx.x; i < (unsigned)(bins * bins); i += kPairThreads) {
            const unsigned x = i / (unsigned)bins, key = i + x * (pitch - bins);
            const unsigned v = WIDE ? s_hist[key] : key >= words ? s_hist[key - words] >> 16 : s_hist[key] & 0xffffu;
            if (v) atomicAdd(out + i, v);
        }
        if (threadIdx.x == 0) {
            unsigned most = 0u;
            int to = -1;
            for (int p = 0; p < npairs; ++p) {
                const unsigned t = *reinterpret_cast<volatile unsigned*>(A.head + 2 + p);
                if (t < chunks && chunks - t > most) {
                    most = chunks - t;
                    to = p;
                }
            }
            s_pair = most >= kCountWorth * gridDim.x ? to : -1;
        }
        __syncthreads();
        pair = s_pair;
        if (pair < 0) break;
    }
}

// out[i] = sum over the copies of copy[c][i] (count a multiple of 4, 16-byte aligned).
__global__ void __launch_bounds__(256) k_hist_reduce(const uint4* __restrict__ copies, int ncopies, size_t count4,
                                                     uint4* __restrict__ out) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count4; i += (size_t)gridDim.x * blockDim.x) {
        uint4 s = __ldcs(copies + i);
        for (int c = 1; c < ncopies; ++c) {
            const uint4 v = __ldcs(copies + (size_t)c * count4 + i);
            s.x += v.x;
            s.y += v.y;
            s.z += v.z;
            s.w += v.w;
        }
        out[i] = s;
    }
}

// Kernel view of h. False when the edge table is neither small enough for the
// launch parameters nor on the device.
template <int DT>
bool fill_launch(const HistArgs& h, HistLaunch& a) {
    a.cells = h.cells;
    a.n = h.n;
    a.bins = h.bins;
    if (h.use_brush)
        for (int v = 0; v < h.nvars && v < kMaxVars; ++v)
            if ((h.brush.mask >> v) & 1u) {
                a.bvar[a.nbr] = v;
                a.blo[a.nbr] = h.brush.lo[v];
                a.bhi[a.nbr] = h.brush.hi[v];
                ++a.nbr;
            }
    if (h.use_brush && h.brush.pmask) {
        for (int i = 0; i < kNumPos; ++i) { a.plo[i] = h.brush.plo[i]; a.phi[i] = h.brush.phi[i]; }
        a.pmask = h.brush.pmask;
        a.use_pos = 1;
    }
    a.naxes = h.naxes;
    for (int i = 0; i < h.naxes && i < kMaxVars; ++i) {
        a.avar[i] = h.axis[i];
        if (h.axis[i] >= kPosAxisBase) a.use_pos = 1;
        a.guess_scale[i] = h.guess_scale[i] / (float)h.bins;
        a.guess_off[i] = -h.guess_e0[i] * a.guess_scale[i];
    }
    // load slots of the vector kernel: the axes, then the brushed variables that are no axis (those
    // that fit: see load_slots)
    a.nslot = h.naxes;
    for (int i = 0; i < h.naxes && i < kMaxVars; ++i) {
        a.svar[i] = h.axis[i] >= kPosAxisBase ? -1 : h.axis[i];
        a.slo[i] = -INFINITY;
        a.shi[i] = INFINITY;
    }
    for (int k = 0; k < a.nbr; ++k) {
        int s = -1;
        for (int i = 0; i < h.naxes; ++i)
            if (a.svar[i] == a.bvar[k]) { s = i; break; }
        if (s < 0) {
            if (a.nslot >= kMaxVars) break;
            s = a.nslot++;
            a.svar[s] = a.bvar[k];
        }
        a.sbr |= 1u << s;
        a.slo[s] = a.blo[k];
        a.shi[s] = a.bhi[k];
    }
    const long long plane_bytes = (long long)h.n * h.n * h.n * (DT == kF16 ? 2 : 4);
    for (int s = 0; s < a.nslot && s < kMaxVars; ++s) a.soff[s] = a.svar[s] >= 0 ? a.svar[s] * plane_bytes : 0;
    a.rowctr = h.rowctr;
    a.rot = h.rowctr ? 0 : (int)(0.6180339887498949 * h.n);
    if (DT == kF16)
        for (int s = 0; s < a.nslot && s < kMaxVars; ++s) {
            const uint32_t lo = half_ceil_bits(a.slo[s]), hi = half_floor_bits(a.shi[s]);
            a.slo_h2[s] = lo | (lo << 16);
            a.shi_h2[s] = hi | (hi << 16);
        }
    const int64_t imax = 0x7fffffff;
    a.s_in = (int)std::min<int64_t>(std::max<int64_t>(h.s_in, 0), imax);
    a.s_out = (int)std::min<int64_t>(h.s_out, imax);
    a.out = h.ncopies > 1 ? h.copies : h.out;
    a.nout = h.ncopies > 1 ? h.ncopies : 1;
    // Runs of each pair merge more than runs of whole tuples, but take five times the votes. Without copies
    // the adds that meet in L2 decide: 250^3 FP16 without scratch, whole shell, 4 / 32 / 256 bins 2589 /
    // 1762 / 474 us by tuples, 718 / 446 / 412 by pairs (one cell per lane: 777 / 492 / 391), brushed 913 /
    // 476 / 167 and 239 / 182 / 160. With copies the votes do, unless every in-shell cell counts: 256^3 FP32,
    // 256 bins, brushed 117 by tuples, 126 by pairs; unbrushed 218 and 189.
    a.by_pair = a.nout == 1 || (a.nbr == 0 && a.pmask == 0);
    a.sactive = h.sactive;
    a.nsb = h.nsb;
    const int ne = h.naxes * (h.bins + 1);
    if (h.edges_host && ne <= kInlineEdges) {
        for (int i = 0; i < ne; ++i) a.edges_inl[i] = h.edges_host[i];
        a.edges = nullptr;
    } else if (h.edges) {
        a.edges = h.edges;
    } else {
        return false;
    }
    return true;
}

// The limit of a kernel's dynamic shared memory is the process's, not the call's: it is always set to
// the most that any call takes, because one set to a call's own size could be lowered by another
// thread's call between here and the launch.
constexpr size_t kMostShared = sizeof(float) * ((kMaxVars * (1024 + 1) + 3) & ~3) + (size_t)kHistVecWarps * (2 * kMaxVars * 512 + 256);

template <typename K>
cudaError_t launch_k(K kernel, const HistLaunch& a, int threads, size_t smem, long long items, int sms, cudaStream_t stream) {
    int per_sm = 0;
    cudaError_t e = cudaSuccess;
    if (smem > 48 * 1024) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMostShared);
    // persistent grid: as many blocks as fit at once
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
    if (e != cudaSuccess) return e;
    const long long want = (items + threads / 32 - 1) / (threads / 32);
    long long most = (long long)sms * std::max(1, per_sm);
    if (a.list) most = std::min<long long>(most, kListWarps / kHistVecWarps);   // as many as the list allows for
    const int blocks = (int)std::max<long long>(1, std::min<long long>(want, most));
    kernel<<<blocks, threads, smem, stream>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

typedef void (*HistKernel)(const HistLaunch);
template <int DT, int VEC>
HistKernel list_kernel(int nax, bool groups) {
    if (!groups) return nax ? k_hist<DT, RowWalk<VEC>, -1, true> : k_hist<DT, RowWalk<VEC>, 0, true>;
    switch (nax) {
        case 2: return k_hist<DT, GroupWalk<VEC>, 2, true>;
        case 3: return k_hist<DT, GroupWalk<VEC>, 3, true>;
        case 4: return k_hist<DT, GroupWalk<VEC>, 4, true>;
        case 5: return k_hist<DT, GroupWalk<VEC>, 5, true>;
        case 6: return k_hist<DT, GroupWalk<VEC>, 6, true>;
        case 7: return k_hist<DT, GroupWalk<VEC>, 7, true>;
        case 8: return k_hist<DT, GroupWalk<VEC>, 8, true>;
        default: return k_hist<DT, GroupWalk<VEC>, 0, true>;
    }
}

// Shared memory of the count kernel's counters (wide: 32 bits).
size_t count_bytes(int bins, bool wide) { return sizeof(unsigned) * (size_t)count_words(bins, wide); }

cudaError_t launch_count(const CountArgs& c, int sms, cudaStream_t stream) {
    const bool wide = c.bins <= kWideBins;
    const size_t smem = count_bytes(c.bins, wide);
    const auto kernel = c.bins > 256 ? k_hist_count<unsigned short, false> : wide ? k_hist_count<unsigned char, true> : k_hist_count<unsigned char, false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPairBytes);
    if (e != cudaSuccess) return e;
    kernel<<<std::max(sms, c.naxes - 1), kPairThreads, smem, stream>>>(c);
    count_launches(1);
    return cudaGetLastError();
}

// Load slots that the vector kernels would take: the axes, and the brushed variables that are no axis.
int load_slots(const HistArgs& h) {
    int slots = h.naxes;
    for (int v = 0; h.use_brush && v < h.nvars && v < kMaxVars; ++v) {
        bool axis = !((h.brush.mask >> v) & 1u);
        for (int i = 0; i < h.naxes; ++i) axis = axis || h.axis[i] == v;
        if (!axis) ++slots;
    }
    return slots;
}

// Vector kernels' conditions: 16-byte aligned planes (an even edge makes n^3 a multiple of 8)
// and load slots that fit; the group walk also needs whole chunks and sub-bricks per row.
bool vector_walk(const HistArgs& h) {
    return h.n % 2 == 0 && (reinterpret_cast<uintptr_t>(h.cells) & 15u) == 0 && load_slots(h) <= kMaxVars;
}

// Whether a call counts every in-shell cell by stored values alone.
bool lists_whole_rows(const HistArgs& h) {
    if (h.use_brush && (h.brush.mask || h.brush.pmask)) return false;
    for (int i = 0; i < h.naxes; ++i)
        if (h.axis[i] >= kPosAxisBase) return false;
    return true;
}

template <int DT>
cudaError_t launch_t(const HistArgs& h, cudaStream_t stream) {
    HistLaunch a{};                      // about 8.6 KB with the inline edges (host stack)
    if (!fill_launch<DT>(h, a)) return cudaErrorInvalidValue;
    const int ne = h.naxes * (h.bins + 1);
    if (h.s_out < 0) return cudaSuccess;                 // no cell in the shell: the zeroed output is the answer
    constexpr int VEC = DT == kF16 ? 8 : 4;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int rows = a.n * a.n;
    if (!vector_walk(h)) {
        a.rot = 0;
        a.rowctr = nullptr;
        return launch_k(k_hist_scalar<DT>, a, kHistThreads, sizeof(float) * (size_t)ne, rows, sms, stream);
    }
    const size_t smem = sizeof(float) * (size_t)((ne + 3) & ~3) + (size_t)kHistVecWarps * (2 * a.nslot * 512 + 256);
    // brushed listed calls by groups: 512^3 FP16 3 / 4 variables 230 / 315 us, by rows 263 / 339; direct calls are
    // faster by rows (256^3 FP16 77 us, by groups 86)
    const bool groups = h.list && a.sactive && h.n % VEC == 0;
    const int per_plane = groups ? h.nsb * ((h.nsb + 7) / 8) : h.n;      // items of a (sub-brick) plane in z
    const int planes = groups ? h.nsb : h.n;
    const int nax = a.use_pos ? 0 : a.naxes;
    if (!h.list) {
        a.items = per_plane * planes;
        const HistKernel k = a.use_pos ? k_hist<DT, RowWalk<VEC>, 0, false> : k_hist<DT, RowWalk<VEC>, -1, false>;
        return launch_k(k, a, kHistVecThreads, smem, a.items, sms, stream);
    }
    // in slabs of planes whose cells fit the list, each counted before the next
    const HistList L = hist_list(h);
    unsigned* head = static_cast<unsigned*>(h.list);
    a.rowctr = head;
    a.rot = 0;
    a.list_next = head + 1;
    a.list_mask = static_cast<unsigned char*>(h.list) + kListHead;
    a.list_chunks = L.chunks;
    a.list_batch = L.batch;
    a.list = static_cast<unsigned char*>(h.list) + L.bins_at;
    const bool whole = lists_whole_rows(h) && !groups;
    const bool wide_rows = rows >= 8 * 5 * sms * 2 * kHistVecWarps;      // see list_rows
    const int step = groups ? std::max(1, L.planes / 4) : L.planes;
    for (int p = 0; p < planes; p += step) {
        a.item0 = p * per_plane;
        a.items = std::min(planes, p + step) * per_plane;
        const int count = a.items - a.item0;
        a.batch = std::max(1, std::min(32, count / (sms * 2 * kHistVecWarps * 8)));   // about eight batches per warp
        e = cudaMemsetAsync(head, 0, kListHead, stream);
        if (e != cudaSuccess) return e;
        if (whole) {
            const HistKernel k = wide_rows ? (h.bins <= 256 ? k_hist_bins<DT, 8, unsigned char> : k_hist_bins<DT, 8, unsigned short>)
                                           : (h.bins <= 256 ? k_hist_bins<DT, 4, unsigned char> : k_hist_bins<DT, 4, unsigned short>);
            e = launch_k(k, a, kHistVecThreads, sizeof(float) * (size_t)ne, (count + 3) / 4, sms, stream);
        } else {
            e = launch_k(list_kernel<DT, VEC>(nax, groups), a, kHistVecThreads, smem, count, sms, stream);
        }
        if (e == cudaSuccess)
            e = launch_count(CountArgs{a.list, a.list_mask, head, a.list_chunks, h.naxes, h.bins, h.out}, sms, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

// List of a call: the in-shell cells of as many planes as kListBytes hold (every cell of a
// plane taken as in the shell when there is more than one slab).
HistList hist_list(const HistArgs& h) {
    const size_t n = (size_t)h.n, cell = (size_t)h.naxes * (h.bins <= 256 ? 1 : 2);
    // in-shell cells: their unit cubes lie between two spheres sqrt(3)/2 beyond the shell's
    const double ro = 0.5 * std::sqrt((double)std::max<int64_t>(h.s_out, 0)) + 0.87;
    const double ri = std::max(0.0, 0.5 * std::sqrt((double)std::max<int64_t>(h.s_in, 0)) - 0.87);
    const double shell = std::min((double)n * n * n, 4.18880 * (ro * ro * ro - ri * ri * ri) + 1.0);
    // units: whole rows leave up to four partly filled ones (two chords' ends) per row; the
    // compacting kernels may leave 31 of a chunk's 256 cells unused
    const auto units = [&](size_t cells, size_t planes) {
        return lists_whole_rows(h) ? std::max(cells / 8 + 4 * n * planes, cells / 7) : cells / 7 + 1;
    };
    HistList L{};
    L.planes = h.n;
    size_t u = units((size_t)shell, n);
    if (u * 8 * cell > kListBytes) {
        L.planes = (int)std::min<size_t>(n, std::max<size_t>(4, kListBytes / (n * n * cell * 8 / 7 + 32 * n * cell) / 4 * 4));
        u = units((size_t)L.planes * n * n, (size_t)L.planes);
    }
    // a warp may leave its current chunk, the rest of its batch and the next batch unused
    L.batch = (unsigned)std::max<size_t>(1, std::min<size_t>(kListBatch, u / (32 * 8 * kListWarps)));
    L.chunks = (unsigned)(u / 32 + 1 + 2 * L.batch * kListWarps);
    L.bins_at = ((size_t)kListHead + 32 * (size_t)L.chunks + 255) / 256 * 256;
    L.bytes = L.bins_at + (size_t)L.chunks * kListCells * cell;
    return L;
}

// Large grids on the vector path whose pair histogram fits a block (up to kListBins bins). On smaller
// ones the second kernel and the blocks' clearing and adding up cost more than the
// atomics. Listed / direct, us: whole shell 128^3 FP32 59 / 62, 256^3 FP32 141 / 189; brushed, after a render has
// filled the caches, 256^3 FP16 83 / 77, 256^3 FP32 97 / 99 (a whole step with it 1031 / 1017), 512^3 315 / 400.
bool hist_by_list(const HistArgs& h) {
    return (long long)h.n * h.n * h.n >= (h.use_brush ? kListGridBrush : kListGrid) && vector_walk(h) && h.bins <= kListBins;
}

int hist_copies(int n, int naxes, int bins) {
    const size_t bytes = sizeof(uint32_t) * (size_t)(naxes - 1) * bins * bins;
    if ((long long)n * n * n < (1LL << 21) || bytes % 16) return 1;      // small grids: not worth a pass
    const size_t fit = kHistCopyBytes / bytes;
    return (int)std::min<size_t>(kHistMaxCopies, fit);
}

cudaError_t launch_histogram_reduce(const uint32_t* copies, int ncopies, size_t count, uint32_t* out,
                                    cudaStream_t stream) {
    const size_t count4 = count / 4;
    const unsigned blocks = (unsigned)std::min<size_t>((count4 + 255) / 256, 4096);
    k_hist_reduce<<<blocks, 256, 0, stream>>>(reinterpret_cast<const uint4*>(copies), ncopies, count4,
                                               reinterpret_cast<uint4*>(out));
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_histogram(const HistArgs& a, int dtype, cudaStream_t stream) {
    if (dtype == kF16) return launch_t<kF16>(a, stream);
    return launch_t<kF32>(a, stream);
}

}  // namespace raypc
