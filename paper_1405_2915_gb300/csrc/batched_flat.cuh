// Shared pieces of the flat segmented batched variants (k_batched_seg.cu,
// k_batched_rr.cu): the instances lie end to end in `values`, so the call is
// one scan of the whole array that restarts at every instance start, plus a
// segmented sum of squares read at every instance's last element.
#pragma once

#include "scan_tile.cuh"

namespace skel {
namespace {

using dev::Pair;
constexpr int kBlock = 256;
constexpr int kSubTile = 4096;   // elements of a 16 KiB sub-tile

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// (sum, sum of squares, has-head) triples; combined in order by
// (a, b) -> b.head ? b : (a.s + b.s, a.q + b.q, a.head).
struct Seg {
    float s, q;
    int h;
};
__device__ __forceinline__ Seg seg_add(const Seg &a, const Seg &b)
{
    return b.h ? b : Seg{a.s + b.s, a.q + b.q, a.h};
}
// Inclusive segmented scan over the lanes of a warp.
__device__ __forceinline__ Seg warp_seg_scan(Seg v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float s = __shfl_up_sync(0xffffffffu, v.s, o);
        const float q = __shfl_up_sync(0xffffffffu, v.q, o);
        const int h = __shfl_up_sync(0xffffffffu, v.h, o);
        if (lane >= o && !v.h) {
            v.s += s;
            v.q += q;
            v.h = h;
        }
    }
    return v;
}
// N warp scans at once: inc the inclusive sums of the lanes' values v, ex the
// exclusive ones.  ex is summed on the way: inc minus v loses what v swamps,
// and is NaN where v is infinite; a shuffle from the lane before takes longer
// (variant 7, 4096 instances of 64 to 2^20: 708 us, 726 by shuffles, 705 by
// the difference).
template <int N>
__device__ __forceinline__ void warp_scans(const float (&v)[N], float (&inc)[N], float (&ex)[N])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        inc[k] = v[k];
        ex[k] = 0.f;
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const float u = __shfl_up_sync(0xffffffffu, inc[k], o);
            if (lane >= o) {
                ex[k] += u;
                inc[k] += u;
            }
        }
}

}  // namespace
}  // namespace skel
