// Device-side helpers shared by the kernel translation units: cache-hinted
// 128-bit loads/stores, warp/block reductions and scans, the map functors,
// and the acquire/release accesses of the look-back protocol.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <math.h>

#include "internal.h"

namespace skel {
namespace dev {

constexpr int kWarp = 32;

// ------------------------------------------------------ memory accesses ---
// Streaming read: bypass L1 allocation (each byte is read once).
__device__ __forceinline__ float4 ld_stream(const float4 *p)
{
    float4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint4 ld_stream(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
// Streaming write: evict-first in L2 (the output is not re-read by this kernel).
__device__ __forceinline__ void st_stream(float4 *p, float4 v)
{
    asm volatile("st.global.cs.v4.f32 [%0], {%1,%2,%3,%4};"
                 :: "l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void st_stream(uint4 *p, uint4 v)
{
    asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};"
                 :: "l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// Release store / acquire load at GPU scope (look-back flags).
__device__ __forceinline__ void st_release(uint32_t *p, uint32_t v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" :: "l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_volatile(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.volatile.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint64_t globaltimer()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Asynchronous copies into shared memory (16 bytes bypass L1; 4 bytes for
// rows of any alignment), in groups that are waited for in order.
__device__ __forceinline__ void cp_async16(uint32_t dst, const float *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const float *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" :: "r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory"); }

// A running float32 sum hi + lo: lo holds the rounding errors of hi, each
// exact (Knuth's TwoSum), about 48 bits together with float32 operations only
// (float64 units are few on this GPU).  The error term of an infinite sum is
// inf - inf, so lo is read through low(), which is 0 there.
struct Sum2 {
    float hi = 0.f, lo = 0.f;
    Sum2() = default;
    __device__ __forceinline__ explicit Sum2(double v) : hi((float)v), lo((float)(v - (double)(float)v)) {}
    __device__ __forceinline__ void add(float v)
    {
        const float s = hi + v, bv = s - hi;
        lo += (hi - (s - bv)) + (v - bv);
        hi = s;
    }
    __device__ __forceinline__ float low() const { return isinf(hi) ? 0.f : lo; }
    __device__ __forceinline__ double value() const { return (double)hi + (double)low(); }
};

// The first statement of every kernel.  launch_kernel lets a kernel's blocks
// be set up while the stream's previous kernel drains (programmatic dependent
// launch); this waits until that kernel has completed and its writes are
// visible, so a kernel's memory accesses still follow those of everything
// before it on the stream.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ------------------------------------------------------------ operators ---
struct AddF { __device__ __forceinline__ static float id() { return 0.f; }
              __device__ __forceinline__ static float op(float a, float b) { return a + b; } };
struct MaxF { __device__ __forceinline__ static float id() { return -INFINITY; }
              __device__ __forceinline__ static float op(float a, float b) { return fmaxf(a, b); } };
// int32 (+) wraps modulo 2^32: computed on the unsigned bit pattern.
struct AddU { __device__ __forceinline__ static uint32_t id() { return 0u; }
              __device__ __forceinline__ static uint32_t op(uint32_t a, uint32_t b) { return a + b; } };
// int32 max on the unsigned bit pattern, compared as signed.
struct MaxI { __device__ __forceinline__ static uint32_t id() { return 0x80000000u; }
              __device__ __forceinline__ static uint32_t op(uint32_t a, uint32_t b) {
                  return (int32_t)a > (int32_t)b ? a : b; } };

template <class Op, class T>
__device__ __forceinline__ T warp_reduce(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = Op::op(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Block-wide reduction; result valid in every thread.  smem: >= 32 entries.
template <class Op, class T, int BLOCK>
__device__ __forceinline__ T block_reduce(T v, T *smem)
{
    constexpr int NW = BLOCK / kWarp;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    v = warp_reduce<Op>(v);
    if (lane == 0) smem[w] = v;
    __syncthreads();
    if (w == 0) {
        T t = lane < NW ? smem[lane] : Op::id();
        t = warp_reduce<Op>(t);
        if (lane == 0) smem[0] = t;
    }
    __syncthreads();
    T r = smem[0];
    __syncthreads();
    return r;
}

// Inclusive warp scan (Hillis-Steele over 32 lanes).
template <class T>
__device__ __forceinline__ T warp_incl_scan_add(T v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v = v + t;
    }
    return v;
}
// Its exclusive form, from the lane before (the inclusive value minus the
// lane's own is NaN where that is infinite).
template <class T>
__device__ __forceinline__ T warp_exclusive(T incl)
{
    const T t = __shfl_up_sync(0xffffffffu, incl, 1);
    return (threadIdx.x & 31) == 0 ? T(0) : t;
}

// ----------------------------------------------------------- map functors --
// out = f(x, y; a), one instantiation per skel_fn (the compiled-in user
// functions of the map skeleton).
template <int FN> struct MapF;
template <> struct MapF<SKEL_FN_ADD>   { static constexpr int nin = 2; __device__ __forceinline__ static float f(float x, float y, float) { return x + y; } };
template <> struct MapF<SKEL_FN_SUB>   { static constexpr int nin = 2; __device__ __forceinline__ static float f(float x, float y, float) { return x - y; } };
template <> struct MapF<SKEL_FN_MUL>   { static constexpr int nin = 2; __device__ __forceinline__ static float f(float x, float y, float) { return x * y; } };
template <> struct MapF<SKEL_FN_MAX>   { static constexpr int nin = 2; __device__ __forceinline__ static float f(float x, float y, float) { return fmaxf(x, y); } };
template <> struct MapF<SKEL_FN_AXPY>  { static constexpr int nin = 2; __device__ __forceinline__ static float f(float x, float y, float a) { return fmaf(a, x, y); } };
template <> struct MapF<SKEL_FN_TANH>  { static constexpr int nin = 1; __device__ __forceinline__ static float f(float x, float, float) { return tanhf(x); } };
template <> struct MapF<SKEL_FN_SQ>    { static constexpr int nin = 1; __device__ __forceinline__ static float f(float x, float, float) { return x * x; } };
template <> struct MapF<SKEL_FN_SCALE> { static constexpr int nin = 1; __device__ __forceinline__ static float f(float x, float, float a) { return a * x; } };
template <> struct MapF<SKEL_FN_COPY>  { static constexpr int nin = 1; __device__ __forceinline__ static float f(float x, float, float) { return x; } };

__device__ __forceinline__ float4 map4_apply(float4 x, float4 y, float a,
                                             float (*fn)(float, float, float))
{
    return make_float4(fn(x.x, y.x, a), fn(x.y, y.y, a), fn(x.z, y.z, a), fn(x.w, y.w, a));
}

}  // namespace dev

// Host helpers ------------------------------------------------------------
inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Every kernel of the library is launched through this wrapper, which
// counts launches (skel_launch_count).  The launch may overlap the tail of
// the previous kernel of the stream (dev::grid_wait holds the kernel's own
// accesses back until that one is complete): back to back, a kernel of one
// block takes 0.8 us instead of 2.1, one of 1216 blocks of 10 us 11.6 instead
// of 14.3.  No kernel signals its dependents early: that gained nothing more
// and took residency from the running kernel (20000 blocks: 21.6 us).
template <class... KArgs, class... Args>
inline void launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                          Args &&...args)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);   // errors: the callers peek at the last error
    note_launch();
}
inline bool aligned16(const void *p) { return ((uintptr_t)p & 15u) == 0; }

}  // namespace skel
