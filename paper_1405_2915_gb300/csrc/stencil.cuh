// Building blocks of the 2D MapOverlap kernels shared by the stencil
// skeleton (k_stencil.cu) and the composed Map -> MapOverlap -> MapReduce
// chain (k_compose.cu): the boundary map of an axis and the 3x3 weighted sum
// in its fixed tap order, so that both evaluate a stencil output with the
// same operations.
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace skel {

// cuTensorMapEncodeTiled, or nullptr where the driver has none (k_stencil.cu).
using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiled encode_tiled();

struct W9 { float w[9]; };
struct W33 { float w[33]; };

// Source index of logical index k on an axis of length n, or -1 (read as 0).
__device__ __forceinline__ int64_t bmap(int64_t k, int64_t n, int b)
{
    if (k >= 0 && k < n) return k;
    if (b == SKEL_CLAMP) return k < 0 ? 0 : n - 1;
    if (b == SKEL_PERIODIC) { int64_t m = k % n; return m < 0 ? m + n : m; }
    return -1;
}

__device__ __forceinline__ float at2(const float *__restrict__ in, int64_t r, int64_t c, int64_t rows,
                                     int64_t cols, int b)
{
    const int64_t sr = bmap(r, rows, b), sc = bmap(c, cols, b);
    return (sr < 0 || sc < 0) ? 0.f : __ldg(in + sr * cols + sc);
}

// The input rows of a warp that walks down a strip of 128 columns (4 per
// lane): rows q0, q0 + 1, ... of columns g0 .. g0 + 127 arrive in a ring of
// kStripRing rows in shared memory, 3.5 KiB in flight per warp without
// holding registers.  Columns outside the grid are left unwritten; wrap: rows
// and columns are taken modulo the grid.  VEC: 16-byte aligned rows.
constexpr int kStripCols = 128, kStripRing = 8;

template <bool VEC>
struct StripRing {
    static constexpr int NL = VEC ? 1 : 4;   // copies per lane and row
    uint32_t ring;
    const float *src[NL];
    bool ok[NL];
    int64_t rows, cols, wrap_at;             // wrap_at: the row index that starts over
    int nin, lane;                           // nin: rows to copy

    __device__ __forceinline__ StripRing(const float *in, int64_t rows_, int64_t cols_, bool wrap, int64_t q0, int64_t g0,
                                         int nin_, float *smem)
        : rows(rows_), cols(cols_), nin(nin_)
    {
        lane = threadIdx.x & 31;
        ring = (uint32_t)__cvta_generic_to_shared(smem);
        int64_t row = q0;
        if (wrap) { row %= rows; if (row < 0) row += rows; }
        wrap_at = wrap ? rows - row : INT64_MAX;
#pragma unroll
        for (int k = 0; k < NL; ++k) {
            int64_t c = VEC ? g0 + 4 * lane : g0 + 32 * k + lane;
            if (wrap) { c %= cols; if (c < 0) c += cols; }
            ok[k] = c >= 0 && c < cols;
            src[k] = in + row * cols + (ok[k] ? c : 0);
        }
    }
    // starts the copy of row q0 + i (called for i = 0, 1, ... in order)
    __device__ __forceinline__ void copy(int i)
    {
        if (i < nin) {
            const uint32_t d = ring + (uint32_t)(i & (kStripRing - 1)) * (kStripCols * 4u);
            if (i == wrap_at) {
                wrap_at += rows;
#pragma unroll
                for (int k = 0; k < NL; ++k) src[k] -= rows * cols;
            }
#pragma unroll
            for (int k = 0; k < NL; ++k) {
                if (ok[k]) {
                    if (VEC) dev::cp_async16(d + 16u * lane, src[k]);
                    else dev::cp_async4(d + 4u * (32 * k + lane), src[k]);
                }
                src[k] += cols;
            }
        }
        dev::cp_commit();
    }
    __device__ __forceinline__ void start()
    {
#pragma unroll
        for (int i = 0; i < kStripRing - 1; ++i) copy(i);
    }
};

// The 3x3 weighted sum in a fixed tap order (row-major over di, dj).
template <bool TAPS5>
__device__ __forceinline__ float stencil9(const W9 &w, float a0, float a1, float a2, float b0, float b1,
                                          float b2, float c0, float c1, float c2)
{
    float acc = 0.f;
    if (!TAPS5) acc = fmaf(w.w[0], a0, acc);
    acc = fmaf(w.w[1], a1, acc);
    if (!TAPS5) acc = fmaf(w.w[2], a2, acc);
    acc = fmaf(w.w[3], b0, acc);
    acc = fmaf(w.w[4], b1, acc);
    acc = fmaf(w.w[5], b2, acc);
    if (!TAPS5) acc = fmaf(w.w[6], c0, acc);
    acc = fmaf(w.w[7], c1, acc);
    if (!TAPS5) acc = fmaf(w.w[8], c2, acc);
    return acc;
}

}  // namespace skel
