// Volume preparation kernels: ingest/relayout and level-of-detail mean fused
// with brick min/max; the empty-space distance of classified sub-bricks.
//
// Section 2.1 of the paper prepares the data once (levels of detail, derived
// variables); Section 2.2 relies on that preparation not depending on the
// restrictions, so a brush edit only re-runs the (cheap) classification.
#include <algorithm>

#include "common.cuh"

namespace raypc {

namespace {

// Round to the storage dtype (the stored value, as a float).
template <int DT> __device__ __forceinline__ float to_stored(float v);
template <> __device__ __forceinline__ float to_stored<kF32>(float v) { return v; }
template <> __device__ __forceinline__ float to_stored<kF16>(float v) { return __half2float(__float2half_rn(v)); }

struct RowsArgs {
    const void* src;      // ingest: planar source (src_dtype); LOD: planar cells of the finer level;
                          // bricks only: planar cells of this level
    int src_dtype;        // ingest only
    int n_src;            // LOD: edge of the finer level
    void* cells;          // this level, planar
    void* pairs;          // this level, x-pairs
    int n;                // edge of this level
    int nvars;
    float* bmin;          // [nb^3][nvars]
    float* bmax;
    float* sbmin;         // [nsb^3][nvars], sub-bricks of edge kSub
    float* sbmax;
    void* ccells;         // ingest with the next level: its planar cells (edge n / 2) ...
    void* cpairs;         // ... and x-pairs
    LevelStats stats;
};

__device__ __forceinline__ void fold(float& mn, float& mx, float a_mn, float a_mx) {
    mn = fminf(mn, a_mn);
    mx = fmaxf(mx, a_mx);
}

// VEC consecutive values of a planar array of element type T (kF32 / kF16)
// starting at element i (aligned to VEC elements when VEC > 1), as floats.
template <int T, int VEC> __device__ __forceinline__ void load_run(const void* base, size_t i, float* out);
template <> __device__ __forceinline__ void load_run<kF32, 1>(const void* base, size_t i, float* out) {
    out[0] = __ldg(reinterpret_cast<const float*>(base) + i);
}
template <> __device__ __forceinline__ void load_run<kF16, 1>(const void* base, size_t i, float* out) {
    out[0] = __half2float(__ushort_as_half(__ldg(reinterpret_cast<const unsigned short*>(base) + i)));
}
template <> __device__ __forceinline__ void load_run<kF32, 2>(const void* base, size_t i, float* out) {
    const float2 a = __ldg(reinterpret_cast<const float2*>(reinterpret_cast<const float*>(base) + i));
    out[0] = a.x; out[1] = a.y;
}
template <> __device__ __forceinline__ void load_run<kF16, 2>(const void* base, size_t i, float* out) {
    const unsigned w = __ldg(reinterpret_cast<const unsigned*>(reinterpret_cast<const __half*>(base) + i));
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w));
    out[0] = f.x; out[1] = f.y;
}
template <> __device__ __forceinline__ void load_run<kF32, 4>(const void* base, size_t i, float* out) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(base) + i));
    out[0] = a.x; out[1] = a.y; out[2] = a.z; out[3] = a.w;
}
template <> __device__ __forceinline__ void load_run<kF32, 8>(const void* base, size_t i, float* out) {
    load_run<kF32, 4>(base, i, out);
    load_run<kF32, 4>(base, i + 4, out + 4);
}
template <> __device__ __forceinline__ void load_run<kF16, 8>(const void* base, size_t i, float* out) {
    const uint4 w = __ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const __half*>(base) + i));
    const unsigned ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&ws[q]));
        out[2 * q] = f.x;
        out[2 * q + 1] = f.y;
    }
}

// The same in two steps, so that no conversion waits between the loads of several runs.
template <int T, int VEC> struct RawRun;
template <> struct RawRun<kF32, 1> {
    float v;
    __device__ __forceinline__ void load(const void* base, size_t i) { v = __ldg(reinterpret_cast<const float*>(base) + i); }
    __device__ __forceinline__ void get(float* out) const { out[0] = v; }
};
template <> struct RawRun<kF32, 4> {
    float4 v;
    __device__ __forceinline__ void load(const void* base, size_t i) {
        v = __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(base) + i));
    }
    __device__ __forceinline__ void get(float* out) const { out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w; }
};
template <> struct RawRun<kF16, 1> {
    unsigned short v;
    __device__ __forceinline__ void load(const void* base, size_t i) { v = __ldg(reinterpret_cast<const unsigned short*>(base) + i); }
    __device__ __forceinline__ void get(float* out) const { out[0] = __half2float(__ushort_as_half(v)); }
};
template <> struct RawRun<kF16, 4> {
    uint2 v;
    __device__ __forceinline__ void load(const void* base, size_t i) {
        v = __ldg(reinterpret_cast<const uint2*>(reinterpret_cast<const __half*>(base) + i));
    }
    __device__ __forceinline__ void get(float* out) const {
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&v.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&v.y));
        out[0] = a.x; out[1] = a.y; out[2] = b.x; out[3] = b.y;
    }
};

// Store VEC stored values (already rounded to DT) of one row run: the cells
// and their x-pairs (c[x], c[x+1]); val[VEC] is the value right of the run.
template <int DT, int VEC>
__device__ __forceinline__ void store_run(void* cells, void* pairs, size_t i, const float* val) {
    if (DT == kF32) {
        float* c = reinterpret_cast<float*>(cells) + i;
        float2* p = reinterpret_cast<float2*>(pairs) + i;
        if (VEC == 4) {
            *reinterpret_cast<float4*>(c) = make_float4(val[0], val[1], val[2], val[3]);
            reinterpret_cast<float4*>(p)[0] = make_float4(val[0], val[1], val[1], val[2]);
            reinterpret_cast<float4*>(p)[1] = make_float4(val[2], val[3], val[3], val[4]);
        } else {
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
                c[q] = val[q];
                p[q] = make_float2(val[q], val[q + 1]);
            }
        }
    } else {
        __half h[VEC + 1];
#pragma unroll
        for (int q = 0; q <= VEC; ++q) h[q] = __float2half_rn(val[q]);   // exact: values are stored halves
        __half* c = reinterpret_cast<__half*>(cells) + i;
        __half2* p = reinterpret_cast<__half2*>(pairs) + i;
        if (VEC == 4) {
            __half2 c01 = __halves2half2(h[0], h[1]), c23 = __halves2half2(h[2], h[3]);
            uint2 cw;
            cw.x = *reinterpret_cast<unsigned*>(&c01);
            cw.y = *reinterpret_cast<unsigned*>(&c23);
            *reinterpret_cast<uint2*>(c) = cw;
            __half2 p0 = __halves2half2(h[0], h[1]), p1 = __halves2half2(h[1], h[2]);
            __half2 p2 = __halves2half2(h[2], h[3]), p3 = __halves2half2(h[3], h[4]);
            uint4 pw;
            pw.x = *reinterpret_cast<unsigned*>(&p0);
            pw.y = *reinterpret_cast<unsigned*>(&p1);
            pw.z = *reinterpret_cast<unsigned*>(&p2);
            pw.w = *reinterpret_cast<unsigned*>(&p3);
            *reinterpret_cast<uint4*>(p) = pw;
        } else {
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
                c[q] = h[q];
                p[q] = __halves2half2(h[q], h[q + 1]);
            }
        }
    }
}

// Values of columns X .. X+VEC of row (y, z) of variable v of a coarser level, rounded to the
// storage dtype; column X+VEC is clamped to n-1: the FP32 mean of the 2x2x2 fine cells, fine
// indices clamped, ((c000 + c100) + (c010 + c110)) + ((c001 + c101) + (c011 + c111)), x 1/8.
// With VEC > 1 the caller guarantees n % VEC == 0 and an even fine edge.
template <int DT, int VEC>
__device__ __forceinline__ void produce_run(const RowsArgs& A, int X, int y, int z, int v, float* val) {
    const int n = A.n;
    const bool right = X + VEC < n;
    {
        const int nf = A.n_src;
        const int y0 = 2 * y, y1 = min(y0 + 1, nf - 1), z0 = 2 * z, z1 = min(z0 + 1, nf - 1);
        const size_t plane = (size_t)v * nf * nf * nf;
        const size_t r00 = plane + ((size_t)z0 * nf + y0) * nf, r10 = plane + ((size_t)z0 * nf + y1) * nf;
        const size_t r01 = plane + ((size_t)z1 * nf + y0) * nf, r11 = plane + ((size_t)z1 * nf + y1) * nf;
        // fine columns 2X .. 2X+2VEC+1 (the last two for the right neighbour), clamped
        constexpr int W = 2 * VEC + 2;
        float f00[W], f10[W], f01[W], f11[W];
        const int fx = 2 * X;
        if (VEC > 1) {
            load_run<DT, 2 * VEC>(A.src, r00 + fx, f00);
            load_run<DT, 2 * VEC>(A.src, r10 + fx, f10);
            load_run<DT, 2 * VEC>(A.src, r01 + fx, f01);
            load_run<DT, 2 * VEC>(A.src, r11 + fx, f11);
            const int e0 = right ? fx + 2 * VEC : fx + 2 * VEC - 2;    // even: a 2-run stays in the row
            load_run<DT, 2>(A.src, r00 + e0, f00 + 2 * VEC);
            load_run<DT, 2>(A.src, r10 + e0, f10 + 2 * VEC);
            load_run<DT, 2>(A.src, r01 + e0, f01 + 2 * VEC);
            load_run<DT, 2>(A.src, r11 + e0, f11 + 2 * VEC);
        } else {
            // fine columns of X, then of the right neighbour X+1 (of X itself at the edge)
            const int g = right ? fx + 2 : fx;
            const int cc[4] = {fx, min(fx + 1, nf - 1), g, min(g + 1, nf - 1)};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                load_run<DT, 1>(A.src, r00 + cc[q], f00 + q);
                load_run<DT, 1>(A.src, r10 + cc[q], f10 + q);
                load_run<DT, 1>(A.src, r01 + cc[q], f01 + q);
                load_run<DT, 1>(A.src, r11 + cc[q], f11 + q);
            }
        }
#pragma unroll
        for (int q = 0; q <= VEC; ++q) {
            const int a = 2 * q, b = 2 * q + 1;
            const float s0 = __fadd_rn(__fadd_rn(f00[a], f00[b]), __fadd_rn(f10[a], f10[b]));
            const float s1 = __fadd_rn(__fadd_rn(f01[a], f01[b]), __fadd_rn(f11[a], f11[b]));
            val[q] = to_stored<DT>(__fmul_rn(__fadd_rn(s0, s1), 0.125f));
        }
    }
}

// Level-of-detail pass. One block per (brick row (by, bz), variable), threads (t, dz): thread t owns
// the VEC columns X = VEC t .. VEC t + VEC-1 (striding over the level when it
// is wider than the block) of z-slice z = 8bz + dz, dz in 0..8, and also reads
// column X+VEC, the right element of its last pair. Each thread streams the
// (up to) 9 x-rows y in [8by, 8by+8] of its slice, writes the rows it owns
// (dy, dz < 8: cells and x-pairs) and folds every row, apron rows included,
// with the right column, into NaN-ignoring min/max for the two y halves of
// the brick (half 0 is rows 0..4, half 1 rows 4..8; row 4 is in both). The
// slices are folded into the two z halves in shared memory, then lanes are
// reduced with shuffles: 4/VEC lanes make a sub-brick of edge 4 (x in
// 4s..min(4s+4, n-1)), two sub-bricks a brick (x in 8b..min(8b+8, n-1)).
constexpr int kRowCols = 64;                            // column threads per block (blockDim.x)
constexpr int kRowSlices = kBrick + 1;                  // blockDim.y

// The next level's two cells (2 t, 2 t + 1) of one row, from the per-slice sums in
// shared memory, stored with their x-pairs at flat index i (even). The pair of cell
// 2 t + 1 needs cell 2 t + 2: from the neighbouring thread, the cell itself at the
// row's end, or -- at the end of a column chunk -- from the next chunk's first
// thread, which writes that half (`whole` false: only the first half here).
template <int DT>
__device__ __forceinline__ void store_next_level(void* cells, void* pairs, size_t i, float v0, float v1, float r,
                                                 bool whole) {
    if (DT == kF32) {
        float* c = reinterpret_cast<float*>(cells) + i;
        float* p = reinterpret_cast<float*>(pairs) + 2 * i;
        *reinterpret_cast<float2*>(c) = make_float2(v0, v1);
        if (whole) {
            *reinterpret_cast<float4*>(p) = make_float4(v0, v1, v1, r);
        } else {
            *reinterpret_cast<float2*>(p) = make_float2(v0, v1);
            p[2] = v1;
        }
    } else {
        const __half h0 = __float2half_rn(v0), h1 = __float2half_rn(v1), hr = __float2half_rn(r);   // exact
        __half2 c01 = __halves2half2(h0, h1), c1r = __halves2half2(h1, hr);
        *reinterpret_cast<__half2*>(reinterpret_cast<__half*>(cells) + i) = c01;
        __half* p = reinterpret_cast<__half*>(pairs) + 2 * i;
        if (whole) {
            uint2 w;
            w.x = *reinterpret_cast<unsigned*>(&c01);
            w.y = *reinterpret_cast<unsigned*>(&c1r);
            *reinterpret_cast<uint2*>(p) = w;
        } else {
            *reinterpret_cast<__half2*>(p) = c01;
            p[2] = h1;
        }
    }
}

template <int DT>
__device__ __forceinline__ void store_pair_second(void* pairs, size_t i, float v) {
    if (DT == kF32) reinterpret_cast<float*>(pairs)[2 * i + 1] = v;
    else reinterpret_cast<__half*>(pairs)[2 * i + 1] = __float2half_rn(v);
}

// Record the magnitudes of variable v: odd is NaN in a thread that met a NaN or
// infinite value, mag the largest |value| the thread knows of (NaN: none), in the
// warps with `all` set. One atomic per warp that may raise the level's: an atomic per
// thread that met a NaN took 512^3 FP16 with NaN outside the shell from 1.79 to 9.42 ms.
__device__ __forceinline__ void level_stats(unsigned* stats, int v, float odd, float mag, bool all) {
    auto raise = [&](int k, unsigned bits) {
        if ((threadIdx.x & 31) == 0 && *(volatile unsigned*)(stats + k) < bits) atomicMax(stats + k, bits);
    };
    if (__any_sync(0xffffffffu, odd != odd)) raise(kMaxVars, 1u);
    if (all) raise(v, __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(mag, 0.0f))));
}

template <int DT, int VEC>
__global__ void __launch_bounds__(kRowCols * kRowSlices, 2) k_lod(RowsArgs A) {
    constexpr int G = kSub / VEC;                       // lanes per sub-brick column
    __shared__ float s_half[kRowSlices][4][kRowCols];  // per slice: min, max of y half 0, then of half 1
    __shared__ float s_odd[kRowSlices][kRowCols];
    const int n = A.n;
    const int nb = (n + kBrick - 1) / kBrick;
    const int nsb = (n + kSub - 1) / kSub;
    const int ncol = (n + VEC - 1) / VEC;
    const int by = blockIdx.x % nb, bz = blockIdx.x / nb, v = blockIdx.y;
    const int dz = threadIdx.y, tx = threadIdx.x;
    const int z = bz * kBrick + dz;
    const float qnan = __int_as_float(0x7fffffff);
    float all_odd = 0.0f, mag = 0.0f;                    // NaN once a value is NaN or infinite; largest |value|
    for (int c0 = 0; c0 < ncol; c0 += blockDim.x) {
        const int t = c0 + tx;
        const bool valid = t < ncol && z < n;
        const int X = t * VEC;
        float ymn[2] = {qnan, qnan}, ymx[2] = {qnan, qnan}, odd = 0.0f;
#pragma unroll
        for (int dy = 0; dy <= kBrick; ++dy) {
            const int y = by * kBrick + dy;
            if (!valid || y >= n) continue;
            float val[VEC + 1];
            produce_run<DT, VEC>(A, X, y, z, v, val);
            float rmn = val[0], rmx = val[0];
#pragma unroll
            for (int q = 1; q <= VEC; ++q) fold(rmn, rmx, val[q], val[q]);
#pragma unroll
            for (int q = 0; q < VEC; ++q) odd = fmaf(val[q], 0.0f, odd);
            if (dy <= kSub) fold(ymn[0], ymx[0], rmn, rmx);
            if (dy >= kSub) fold(ymn[1], ymx[1], rmn, rmx);
            if (dy < kBrick && dz < kBrick)
                store_run<DT, VEC>(A.cells, A.pairs, (((size_t)v * n + z) * n + y) * n + X, val);
        }
        s_half[dz][0][tx] = ymn[0];
        s_half[dz][1][tx] = ymx[0];
        s_half[dz][2][tx] = ymn[1];
        s_half[dz][3][tx] = ymx[1];
        s_odd[dz][tx] = odd;
        all_odd += odd;
        __syncthreads();
        if (dz == 0) {
            // (y half, z half) h = j + 2i: slices 0..4 make z half 0, slices 4..8 z half 1
            float mn[4] = {qnan, qnan, qnan, qnan}, mx[4] = {qnan, qnan, qnan, qnan};
#pragma unroll
            for (int sl = 0; sl < kRowSlices; ++sl) {
                const float a0 = s_half[sl][0][tx], b0 = s_half[sl][1][tx];
                const float a1 = s_half[sl][2][tx], b1 = s_half[sl][3][tx];
                if (sl <= kSub) { fold(mn[0], mx[0], a0, b0); fold(mn[1], mx[1], a1, b1); }
                if (sl >= kSub) { fold(mn[2], mx[2], a0, b0); fold(mn[3], mx[3], a1, b1); }
            }
            // sub-bricks: reduce over the G lanes of a sub-brick column
#pragma unroll
            for (int m = 1; m < G; m <<= 1)
#pragma unroll
                for (int h = 0; h < 4; ++h)
                    fold(mn[h], mx[h], __shfl_xor_sync(0xffffffffu, mn[h], m), __shfl_xor_sync(0xffffffffu, mx[h], m));
            // a NaN or infinite value in any of the column's rows marks its four sub-bricks
            float any = 0.0f;
#pragma unroll
            for (int sl = 0; sl < kRowSlices; ++sl) any += s_odd[sl][tx];
#pragma unroll
            for (int m = 1; m < G; m <<= 1) any += __shfl_xor_sync(0xffffffffu, any, m);
            const bool tcol = t < ncol;
            const int sx = t / G;
            if (tcol && t % G == 0) {
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const int sy = 2 * by + (h & 1), sz = 2 * bz + (h >> 1);
                    if (sy < nsb && sz < nsb && sx < nsb) {
                        const size_t sb = ((size_t)sz * nsb + sy) * nsb + sx, nsub = (size_t)nsb * nsb * nsb;
                        A.sbmin[sb * A.nvars + v] = mn[h];
                        A.sbmax[sb * A.nvars + v] = mx[h];
                        A.stats.odd[v * nsub + sb] = any != any;
                    }
                }
            }
            // bricks: all four halves of two neighbouring sub-brick columns
            float bmn = mn[0], bmx = mx[0];
#pragma unroll
            for (int h = 1; h < 4; ++h) fold(bmn, bmx, mn[h], mx[h]);
            fold(bmn, bmx, __shfl_xor_sync(0xffffffffu, bmn, G), __shfl_xor_sync(0xffffffffu, bmx, G));
            const int bx = t / (2 * G);
            if (tcol && t % (2 * G) == 0 && bx < nb) {
                const size_t b = ((size_t)bz * nb + by) * nb + bx;
                A.bmin[b * A.nvars + v] = bmn;
                A.bmax[b * A.nvars + v] = bmx;
            }
            mag = fmaxf(mag, fmaxf(fabsf(bmn), fabsf(bmx)));
        }
        __syncthreads();                                 // s_half is rewritten by the next column chunk
    }
    level_stats(A.stats.mag, v, all_odd, mag, dz == 0);
}

// Ingest and brick passes, by MODE: 0 ingest (the converted source, element type SRC), 2 ingest
// and the next level's cells (n a multiple of 16), 3 the min/max of the level's own
// stored cells, 4 those and the next level's cells (1 is the level-of-detail pass).
//
// A block takes 32 VEC columns of one brick row of one
// variable, a warp one of its four (y half, z half) quadrants, 5 x 5 rows with the
// apron, a thread a run of VEC columns (4 where every run is aligned, else 1). The
// five rows of a slice are loaded together; a run's right neighbour comes from the
// next lane; a sub-brick in x is 4 / VEC neighbouring lanes; the next level's sums
// stay in registers from the even to the odd fine slice, and the warps meet once, for
// the brick.
//
// Bound by HBM: 5.7 TB/s of algorithmic bytes at 512^3, FP32 into FP16 with the next
// level (1.51 ms against 1.79 for blocks of 9 slices with two barriers per 64
// column runs, which left memory idle at the barriers; 2.32 against 2.40 ms for
// FP32 storage; 250^3 FP32, one column per thread, 307 against 419 us). Fewer registers than
// the five rows need spill (8 blocks per SM: 327 against 302 us at 256^3 FP32; FP16 into FP16
// still gains from 8). The loads are raw: with the conversion of an FP16 source behind
// each, the next one waited for it (with the next level, 256^3 FP32 from FP16 325 -> 277 us,
// 512^3 FP16 from FP16 1729 -> 1307; 251^3 FP32 from FP16 435 -> 306).
constexpr int kQuadThreads = 128;
constexpr int quad_blocks(int mode, int dt, int src) { return mode >= 3 ? 10 : dt == kF16 && src == kF16 ? 8 : 5; }

template <int DT, int MODE, int SRC, int VEC>
__global__ void __launch_bounds__(kQuadThreads, quad_blocks(MODE, DT, SRC)) k_quads(RowsArgs A) {
    constexpr int kRows = kSub + 1, G = kSub / VEC;          // rows of a quadrant; lanes of a sub-brick
    constexpr bool kNext = (MODE == 2 || MODE == 4) && VEC == 4, kStore = MODE == 0 || MODE == 2;
    __shared__ float s_mn[4][32], s_mx[4][32];
    const int n = A.n, ncol = (n + VEC - 1) / VEC, nb = (n + kBrick - 1) / kBrick, nsb = (n + kSub - 1) / kSub;
    const int nxc = (ncol + 31) / 32;
    const int lane = threadIdx.x & 31, quad = threadIdx.x >> 5, yh = quad & 1, zh = quad >> 1;
    const int xc = blockIdx.x % nxc, by = (blockIdx.x / nxc) % nb, bz = blockIdx.x / (nxc * nb), v = blockIdx.y;
    const int t = xc * 32 + lane, X = t * VEC;
    const int y0 = by * kBrick + yh * kSub, z0 = bz * kBrick + zh * kSub;
    const bool valid = t < ncol, last = t == ncol - 1;
    const float qnan = __int_as_float(0x7fffffff);
    float mn = qnan, mx = qnan;
    float odd = 0.0f;                                        // NaN once a value is NaN or infinite
    float even[kNext ? 2 : 1][2];                            // sums of the even slice: [coarse row][cell]
#pragma unroll
    for (int dz = 0; dz < kRows; ++dz) {
        const int z = z0 + dz;
        float val[kRows][VEC + 1];
        RawRun<SRC, VEC> raw[kRows];
        RawRun<SRC, 1> edge[kRows];
        // the slice's rows (rows beyond the grid repeat the last one: no new value)
#pragma unroll
        for (int dy = 0; dy < kRows; ++dy) {
            const int y = min(y0 + dy, n - 1);
            raw[dy] = {};
            edge[dy] = {};
            if (!valid || z >= n) continue;
            const size_t row = (((size_t)v * n + z) * n + y) * n;
            raw[dy].load(A.src, row + X);
            if (lane == 31 && !last) edge[dy].load(A.src, row + X + VEC);
        }
#pragma unroll
        for (int dy = 0; dy < kRows; ++dy) {
            raw[dy].get(val[dy]);
            edge[dy].get(val[dy] + VEC);
#pragma unroll
            for (int q = 0; q <= VEC; ++q) val[dy][q] = to_stored<DT>(val[dy][q]);
            const float right = __shfl_down_sync(0xffffffffu, val[dy][0], 1);
            if (last) val[dy][VEC] = val[dy][VEC - 1];
            else if (lane < 31) val[dy][VEC] = right;
            if (!valid || z >= n) continue;
#pragma unroll
            for (int q = 0; q <= VEC; ++q) fold(mn, mx, val[dy][q], val[dy][q]);
#pragma unroll
            for (int q = 0; q < VEC; ++q) odd = fmaf(val[dy][q], 0.0f, odd);
            if (kStore && dy < kSub && dz < kSub && y0 + dy < n)
                store_run<DT, VEC>(A.cells, A.pairs, (((size_t)v * n + z) * n + y0 + dy) * n + X, val[dy]);
        }
        if constexpr (kNext) {
            if (dz == kSub) continue;
            // the next level's cells 2t, 2t+1 of its rows (y0 + {0, 2}) / 2, in its order:
            // (c000 + c100) + (c010 + c110) per fine slice, then the two slices, / 8
            const int m = n >> 1;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                float sum[2];
#pragma unroll
                for (int c = 0; c < 2; ++c)
                    sum[c] = __fadd_rn(__fadd_rn(val[2 * k][2 * c], val[2 * k][2 * c + 1]),
                                       __fadd_rn(val[2 * k + 1][2 * c], val[2 * k + 1][2 * c + 1]));
                if ((dz & 1) == 0) {
                    even[k][0] = sum[0];
                    even[k][1] = sum[1];
                    continue;
                }
                const float v0 = to_stored<DT>(__fmul_rn(__fadd_rn(even[k][0], sum[0]), 0.125f));
                const float v1 = to_stored<DT>(__fmul_rn(__fadd_rn(even[k][1], sum[1]), 0.125f));
                const float r = __shfl_down_sync(0xffffffffu, v0, 1);
                if (!valid) continue;
                const size_t i = (((size_t)v * m + (z >> 1)) * m + ((y0 >> 1) + k)) * m + 2 * t;
                // the pair of cell 2t+1 needs cell 2t+2: the next lane's, the cell itself at the row's
                // end, or from the next column chunk's first lane, which writes that half
                store_next_level<DT>(A.ccells, A.cpairs, i, v0, v1, last ? v1 : r, last || lane < 31);
                if (lane == 0 && t > 0) store_pair_second<DT>(A.cpairs, i - 1, v0);
            }
        }
    }
    // sub-bricks, then bricks
#pragma unroll
    for (int m = 1; m < G; m <<= 1) fold(mn, mx, __shfl_xor_sync(0xffffffffu, mn, m), __shfl_xor_sync(0xffffffffu, mx, m));
    const unsigned om = __ballot_sync(0xffffffffu, odd != odd) >> (lane & ~(G - 1));
    if (valid && t % G == 0 && y0 < n && z0 < n) {
        const size_t sb = ((size_t)(z0 >> 2) * nsb + (y0 >> 2)) * nsb + t / G;
        A.sbmin[sb * A.nvars + v] = mn;
        A.sbmax[sb * A.nvars + v] = mx;
        A.stats.odd[(size_t)v * nsb * nsb * nsb + sb] = (om & ((1u << G) - 1u)) != 0u;
    }
    s_mn[quad][lane] = y0 < n ? mn : qnan;                   // an absent quadrant adds nothing
    s_mx[quad][lane] = y0 < n ? mx : qnan;
    __syncthreads();
    level_stats(A.stats.mag, v, odd, 0.0f, false);
    if (quad != 0) return;
#pragma unroll
    for (int q = 1; q < 4; ++q) fold(mn, mx, s_mn[q][lane], s_mx[q][lane]);
    fold(mn, mx, __shfl_xor_sync(0xffffffffu, mn, G), __shfl_xor_sync(0xffffffffu, mx, G));
    if (valid && t % (2 * G) == 0) {
        const size_t b = ((size_t)bz * nb + by) * nb + t / (2 * G);
        A.bmin[b * A.nvars + v] = mn;
        A.bmax[b * A.nvars + v] = mx;
    }
    level_stats(A.stats.mag, v, 0.0f, fmaxf(fabsf(mn), fabsf(mx)), true);
}

template <int DT, int MODE, int SRC, int VEC>
void launch_quads_t(const RowsArgs& a, cudaStream_t stream) {
    const int nb = (a.n + kBrick - 1) / kBrick, nxc = ((a.n + VEC - 1) / VEC + 31) / 32;
    k_quads<DT, MODE, SRC, VEC><<<dim3((unsigned)(nb * nb * nxc), (unsigned)a.nvars), kQuadThreads, 0, stream>>>(a);
}

template <int DT, int MODE, int SRC>
void launch_quads_t(const RowsArgs& a, bool vec, cudaStream_t stream) {
    if constexpr (MODE == 2 || MODE == 4) launch_quads_t<DT, MODE, SRC, 4>(a, stream);
    else if (vec) launch_quads_t<DT, MODE, SRC, 4>(a, stream);
    else launch_quads_t<DT, MODE, SRC, 1>(a, stream);
}

template <int DT, int VEC>
void launch_lod_t(const RowsArgs& a, cudaStream_t stream) {
    const int nb = (a.n + kBrick - 1) / kBrick, ncol = (a.n + VEC - 1) / VEC;
    // one thread per column run up to kRowCols (narrow levels use narrow blocks), per z-slice
    const dim3 block(min(kRowCols, max(32, (ncol + 31) / 32 * 32)), kRowSlices);
    k_lod<DT, VEC><<<dim3((unsigned)(nb * nb), (unsigned)a.nvars), block, 0, stream>>>(a);
}

template <int MODE>
cudaError_t launch_rows(const RowsArgs& a, int dtype, cudaStream_t stream) {
    if (a.n < 2 || a.n > kMaxRowsEdge) return cudaErrorInvalidValue;
    if constexpr (MODE == 1) {
        // 4-column runs when every run is aligned (n % 4 == 0 and an even fine edge make it 8k)
        // and the level is wide enough to fill a warp with runs
        const bool vec = a.n % 4 == 0 && a.n_src == 2 * a.n && a.n >= 128;
        if (dtype == kF16) { if (vec) launch_lod_t<kF16, 4>(a, stream); else launch_lod_t<kF16, 1>(a, stream); }
        else               { if (vec) launch_lod_t<kF32, 4>(a, stream); else launch_lod_t<kF32, 1>(a, stream); }
    } else {
        // 4-column runs when every run is aligned: n % 4 == 0 and a 16-byte aligned source
        const bool vec = a.n % 4 == 0 && (uintptr_t)a.src % 16 == 0;
        // the fused next level needs them and whole bricks of both levels
        if ((MODE == 2 || MODE == 4) && (!vec || a.n % 16 != 0 || !a.ccells || !a.cpairs)) return cudaErrorInvalidValue;
        if constexpr (MODE >= 3) {
            if (dtype == kF16) launch_quads_t<kF16, MODE, kF16>(a, vec, stream);
            else launch_quads_t<kF32, MODE, kF32>(a, vec, stream);
        } else if (a.src_dtype == kF16) {
            if (dtype == kF16) launch_quads_t<kF16, MODE, kF16>(a, vec, stream);
            else launch_quads_t<kF32, MODE, kF16>(a, vec, stream);
        } else {
            if (dtype == kF16) launch_quads_t<kF16, MODE, kF32>(a, vec, stream);
            else launch_quads_t<kF32, MODE, kF32>(a, vec, stream);
        }
    }
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_ingest(const void* src, int src_dtype, void* cells, void* pairs, int dtype, int n,
                          int nvars, float* bmin, float* bmax, float* sbmin, float* sbmax,
                          LevelStats stats, cudaStream_t stream) {
    RowsArgs a{};
    a.src = src;
    a.src_dtype = src_dtype;
    a.cells = cells;
    a.pairs = pairs;
    a.n = n;
    a.nvars = nvars;
    a.bmin = bmin;
    a.bmax = bmax;
    a.sbmin = sbmin;
    a.sbmax = sbmax;
    a.stats = stats;
    return launch_rows<0>(a, dtype, stream);
}

bool ingest_next_level_fits(const void* src, int n) {
    return n % 16 == 0 && n >= 128 && n <= kMaxRowsEdge && (uintptr_t)src % 16 == 0;
}

cudaError_t launch_ingest_next_level(const void* src, int src_dtype, void* cells, void* pairs, int dtype, int n,
                                     int nvars, float* bmin, float* bmax, float* sbmin, float* sbmax,
                                     void* next_cells, void* next_pairs, LevelStats stats, cudaStream_t stream) {
    RowsArgs a{};
    a.src = src;
    a.src_dtype = src_dtype;
    a.cells = cells;
    a.pairs = pairs;
    a.n = n;
    a.nvars = nvars;
    a.bmin = bmin;
    a.bmax = bmax;
    a.sbmin = sbmin;
    a.sbmax = sbmax;
    a.stats = stats;
    a.ccells = next_cells;
    a.cpairs = next_pairs;
    return launch_rows<2>(a, dtype, stream);
}

cudaError_t launch_level_bricks(const void* cells, int dtype, int n, int nvars, float* bmin, float* bmax,
                                float* sbmin, float* sbmax, void* next_cells, void* next_pairs, LevelStats stats,
                                cudaStream_t stream) {
    RowsArgs a{};
    a.src = cells;
    a.src_dtype = dtype;
    a.n = n;
    a.nvars = nvars;
    a.bmin = bmin;
    a.bmax = bmax;
    a.sbmin = sbmin;
    a.sbmax = sbmax;
    a.ccells = next_cells;
    a.cpairs = next_pairs;
    a.stats = stats;
    return next_cells ? launch_rows<4>(a, dtype, stream) : launch_rows<3>(a, dtype, stream);
}

cudaError_t launch_lod(const void* fine, int n_fine, void* cells, void* pairs, int dtype, int nvars,
                       float* bmin, float* bmax, float* sbmin, float* sbmax, LevelStats stats, cudaStream_t stream) {
    RowsArgs a{};
    a.src = fine;
    a.n_src = n_fine;
    a.cells = cells;
    a.pairs = pairs;
    a.n = (n_fine + 1) / 2;
    a.nvars = nvars;
    a.bmin = bmin;
    a.bmax = bmax;
    a.sbmin = sbmin;
    a.sbmax = sbmax;
    a.stats = stats;
    return launch_rows<1>(a, dtype, stream);
}

namespace {

// One thread per sub-brick: activity AND TF visibility (tf_range_visible).
__global__ void __launch_bounds__(256) k_tf_visibility(TfVisArgs A) {
    const size_t b = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t nsub = (size_t)A.nsb * A.nsb * A.nsb;
    bool bit = b < nsub && ((A.sactive[b >> 5] >> (b & 31)) & 1u);
    if (bit) {
        const size_t o = b * A.nvars + A.color_var;
        bit = tf_range_visible(A.sbmin[o], A.sbmax[o], A.tf_prefix, A.tf_lo, A.tf_scale);
    }
    const unsigned word = __ballot_sync(0xffffffffu, bit);
    if ((threadIdx.x & 31) == 0 && b < nsub) A.out_sactive[b >> 5] = word;
}

}  // namespace

// Empty-space distance of the 4^3 sub-bricks: the Chebyshev distance, in
// sub-bricks, to the nearest active one, capped at kDistCap (0: active). A block
// takes a tile of kDistTile x kDistTile sub-brick rows (y, z) and up to
// 32 kDistWords sub-bricks in x, with a halo of kDistCap rows and one word, as
// bitmasks: one thread per row, a row's words in its registers. It grows the
// active set by one 3x3x3 dilation per step (x in registers, y and z through
// shared memory); the step at which a bit first appears is its distance.
constexpr int kDistTile = 8;
constexpr int kDistWords = 4;
constexpr int kDistRows = kDistTile + 2 * kDistCap;          // rows per axis with the halo
constexpr int kDistThreads = kDistRows * kDistRows;

struct DistanceTiles {
    int lim, ntx, nt;             // sub-bricks per axis that the tiles cover, tiles in x and in y (= z)
};

__host__ __device__ inline DistanceTiles distance_tiles(int n, bool raw) {
    DistanceTiles d;
    d.lim = raw ? (n + kSub - 1) / kSub : ((n - 2) >> 2) + 1;
    d.ntx = (d.lim + 32 * kDistWords - 1) / (32 * kDistWords);
    d.nt = (d.lim + kDistTile - 1) / kDistTile;
    return d;
}

// Tile `tile` of a level; all kDistThreads threads of the block call it.
__device__ __forceinline__ void subbrick_distance_tile(const uint32_t* __restrict__ act, int n, int tile,
                                                       uint8_t* __restrict__ out, bool raw) {
    constexpr int W = kDistWords + 2;                        // one halo word on either side
    __shared__ uint32_t s_row[W][kDistThreads];
    const int nsb = (n + kSub - 1) / kSub;
    const uint32_t nbits = (uint32_t)nsb * nsb * nsb;
    const DistanceTiles T = distance_tiles(n, raw);
    const int w0 = (tile % T.ntx) * kDistWords, ty = (tile / T.ntx) % T.nt, tz = tile / (T.ntx * T.nt);
    const int t = threadIdx.x, ry = t % kDistRows, rz = t / kDistRows;
    const int y = ty * kDistTile + ry - kDistCap, z = tz * kDistTile + rz - kDistCap;
    const bool row = y >= 0 && y < nsb && z >= 0 && z < nsb;
    uint32_t a[W], p[3][kDistWords];
#pragma unroll
    for (int w = 0; w < W; ++w) {
        // bits 32 (w0 + w - 1) .. + 31 of the row, 0 outside it
        const int x = 32 * (w0 + w - 1);
        uint32_t v = 0u;
        if (row && x >= 0 && x < nsb) {
            const uint32_t id = ((uint32_t)z * nsb + y) * nsb + x;
            v = __ldg(act + (id >> 5)) >> (id & 31);
            if ((id & 31) && (id | 31u) + 1u < nbits) v |= __ldg(act + (id >> 5) + 1) << (32 - (id & 31));
            if (nsb - x < 32) v &= (1u << (nsb - x)) - 1u;
        }
        a[w] = v;
    }
#pragma unroll
    for (int w = 0; w < kDistWords; ++w) p[0][w] = p[1][w] = p[2][w] = 0u;
    uint32_t seen[kDistWords];
#pragma unroll
    for (int w = 0; w < kDistWords; ++w) seen[w] = a[w + 1];
    const int up = ry + 1 < kDistRows ? 1 : 0, dn = ry > 0 ? 1 : 0;
    const int fw = rz + 1 < kDistRows ? kDistRows : 0, bk = rz > 0 ? kDistRows : 0;
#pragma unroll 1
    for (int d = 1; d < kDistCap; ++d) {
        // x: within the row (the outer halo words only need the bits next to the inner ones)
        uint32_t prev = 0u;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const uint32_t cur = a[w], next = w + 1 < W ? a[w + 1] : 0u;
            a[w] = cur | (cur << 1) | (cur >> 1) | (prev >> 31) | (next << 31);
            prev = cur;
        }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < W; ++w) s_row[w][t] = a[w];
        __syncthreads();
#pragma unroll
        for (int w = 0; w < W; ++w) a[w] |= s_row[w][t + up] | s_row[w][t - dn];
        __syncthreads();
#pragma unroll
        for (int w = 0; w < W; ++w) s_row[w][t] = a[w];
        __syncthreads();
#pragma unroll
        for (int w = 0; w < W; ++w) a[w] |= s_row[w][t + fw] | s_row[w][t - bk];
        // first seen at this step: the distance, in three bit planes
#pragma unroll
        for (int w = 0; w < kDistWords; ++w) {
            const uint32_t fresh = a[w + 1] & ~seen[w];
            seen[w] |= fresh;
#pragma unroll
            for (int k = 0; k < 3; ++k) p[k][w] |= ((d >> k) & 1) ? fresh : 0u;
        }
    }
    // bytes of the tile's inner rows: planes 0..2 and "never seen" (kDistCap) through shared memory
    __syncthreads();
    static_assert(4 * kDistWords * kDistTile * kDistTile <= W * kDistThreads, "planes fit the row buffer");
    uint32_t* s_plane = &s_row[0][0];                        // [inner row][word][plane]
    const int iy = ry - kDistCap, iz = rz - kDistCap;
    if (iy >= 0 && iy < kDistTile && iz >= 0 && iz < kDistTile) {
        uint32_t* q = s_plane + (iz * kDistTile + iy) * kDistWords * 4;
#pragma unroll
        for (int w = 0; w < kDistWords; ++w) {
            q[4 * w] = p[0][w];
            q[4 * w + 1] = p[1][w];
            q[4 * w + 2] = p[2][w];
            q[4 * w + 3] = ~seen[w];
        }
    }
    __syncthreads();
    // output entries e of the tile on each axis: its own sub-bricks, and in the padded grid the
    // borders before the first and after the last one
    const int pd = raw ? nsb : subbrick_pad(n), pad = raw ? 0 : 1, last = T.lim - 1, end = raw ? nsb - 1 : (n - 1) >> 2;
    auto range = [&](int first, int len, int& e0, int& e1) {
        e0 = first == 0 ? -pad : first;
        e1 = first + len > last ? end : first + len - 1;
    };
    int x0, x1, y0, y1, z0, z1;
    range(32 * w0, 32 * kDistWords, x0, x1);
    range(ty * kDistTile, kDistTile, y0, y1);
    range(tz * kDistTile, kDistTile, z0, z1);
    const int nx = x1 - x0 + 1, ny = y1 - y0 + 1, total = nx * ny * (z1 - z0 + 1);
    for (int i = t; i < total; i += kDistThreads) {
        const int ex = x0 + i % nx, ey = y0 + (i / nx) % ny, ez = z0 + i / (nx * ny);
        const int sx = min(max(ex, 0), last) - 32 * w0;
        const int sy = min(max(ey, 0), last) - ty * kDistTile, sz = min(max(ez, 0), last) - tz * kDistTile;
        const uint32_t* q = s_plane + ((sz * kDistTile + sy) * kDistWords + (sx >> 5)) * 4;
        const int b = sx & 31;
        const unsigned dist = ((q[0] >> b) & 1u) | (((q[1] >> b) & 1u) << 1) | (((q[2] >> b) & 1u) << 2) |
                              (((q[3] >> b) & 1u) << 3);
        out[((size_t)(ez + pad) * pd + ey + pad) * pd + ex + pad] = (uint8_t)dist;
    }
    __syncthreads();                                         // s_row is reused by the block's next tile
}

static_assert(kDistCap == 8, "three bit planes and the never-seen bit");

__global__ void __launch_bounds__(kDistThreads) k_subbrick_distance(const uint32_t* __restrict__ act, int n,
                                                                    uint8_t* __restrict__ out, bool raw) {
    subbrick_distance_tile(act, n, blockIdx.x, out, raw);
}

// Every view of a batch: the blocks walk the views' concatenated tiles.
__global__ void __launch_bounds__(kDistThreads) k_subbrick_distance_views(const BatchHeader* __restrict__ hdr,
                                                                          const BrushItem* __restrict__ views) {
    const int total = hdr->dist_total, nviews = hdr->nviews;
    for (int g = blockIdx.x; g < total; g += gridDim.x) {
        int lo = 0, hi = nviews - 1;                 // the last view whose tiles start at or before g
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (views[mid].dist_begin <= g) lo = mid; else hi = mid - 1;
        }
        const BrushItem& V = views[lo];
        subbrick_distance_tile(V.active, V.n, g - V.dist_begin, V.sdist, false);
    }
}

static int distance_tile_count(int n, bool raw) {
    const DistanceTiles T = distance_tiles(n, raw);
    return T.ntx * T.nt * T.nt;
}

int subbrick_distance_tiles(int n) { return distance_tile_count(n, false); }

cudaError_t launch_subbrick_distance(const uint32_t* sactive, int n, uint8_t* out, bool raw, cudaStream_t stream) {
    k_subbrick_distance<<<distance_tile_count(n, raw), kDistThreads, 0, stream>>>(sactive, n, out, raw);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_subbrick_distance_views(const BatchHeader* hdr, const BrushItem* views, unsigned blocks,
                                           cudaStream_t stream) {
    k_subbrick_distance_views<<<blocks, kDistThreads, 0, stream>>>(hdr, views);
    return cudaGetLastError();
}

cudaError_t launch_tf_visibility(const TfVisArgs& a, cudaStream_t stream) {
    const size_t nsub = (size_t)a.nsb * a.nsb * a.nsb;
    k_tf_visibility<<<(unsigned)((nsub + 255) / 256), 256, 0, stream>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace raypc
