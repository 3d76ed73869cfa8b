// The differentiable composed pipeline in one pass each way (Sec. II: the
// implementation is chosen for the composition, not call by call):
//
//   t = tanh(x), u = S t, s = row-wise inclusive scan of t
//   L = sum u^2 + (1/N) sum s^2                                   (forward)
//   gx = (S^T (2 g u) + rscan(2 (g/N) s)) (1 - t^2)               (backward)
//
// S: the 3x3 MapOverlap stencil (CLAMP or ZERO), rscan: the reverse scan of
// each row, g = dL.  Run as separate skeleton calls the pipeline moves 80
// bytes per point through HBM; here the forward reads x and writes t (8
// bytes), the backward reads t and writes gx (8 bytes), and u, s and both
// intermediate gradients never leave the SM.
//
// A block owns a segment of rows and all columns: thread k holds columns
// Ck .. Ck+C-1 and walks down the rows.  The stencils keep partial tap sums
// as the row stream of k_stream.cu does; the neighbours of a thread's columns
// come by shuffle, across warps through shared memory.  A row's scan is
// local sums, a warp scan, and the sum of the other warps' totals.
// The forward needs one block barrier per row, the backward two (the scan's
// totals and the second stencil's edges travel with the first stencil's).
// Rows come through a ring in shared memory, three of them in flight, and a
// row's slot also carries the finished row back out.  Aligned rows of a
// multiple of 16 columns travel as TMA boxes, others by cp.async into C / 4
// planes (plane p holds the p-th group of four columns of every thread, so
// 16-byte reads are free of bank conflicts) and out by contiguous stores.
//
// What bounds it (8192 x 8192): the forward takes 127 us, the backward 174
// (180 and 235 with cp.async), against 79 us each for their HBM traffic
// (which ncu shows at 1.0 of the algorithmic bytes): instruction issue, active
// 71 and 64 % of the time, with 16 warps per SM whose barriers keep them in the
// same phase (52 and 64 instructions per 32 points: two MUFUs and about 15
// others of tanhf, 9 FMAs per stencil, 5 to 6 per scan).  The forward
// therefore splits its barrier into an arrival and a wait, with the stencil's
// inner columns and the next row's tanh between them (136 us with one whole
// barrier; the backward, at 128 registers, spills when split so: 209).  As
// fifteen separate calls the loss and its gradient took 927 us, here 301.  512
// threads of 16 columns: with 1024 of 8 the scans' shuffles and the edges
// weigh twice as much.
//
// The two sums of squares run per thread with their rounding errors kept, then
// in float64 over threads and blocks; the last block to finish adds the
// blocks' partial sums in index order (deterministic) and writes L.
//
// Row prefixes are float32: a value passes at most 17 roundings (6 in its
// thread, 5 in its warp, 4 between warps, 2 to put them together), so the
// error of s is at most 17 2^-24 of the prefix of |t|.  The reverse scan keeps
// the rounding errors between warps, where its sums are the largest, as its
// error reaches gx directly.  Relative error of gx (norm) on rows of one sign,
// U[0, 0.02], plain -> kept, and separate calls whose scans carry float64
// between tiles of 4096: 2048 x 8191 5.9e-8 -> 5.4e-8, 5.6e-8; 64 x 8192 7.3e-8
// -> 6.3e-8, 7.7e-8.
#include <type_traits>

#include "stencil.cuh"

namespace skel {
namespace {

constexpr int kFwdC = 16, kBwdC = 16;         // columns per thread (forward with 8: 203 us for 180, with cp.async)
constexpr int kLMaxCols = 8192;
constexpr int kLWarps = 32;                   // most warps of a block
constexpr int kFwdRing = 4, kBwdRing = 6;     // rows in shared memory; 3 of them in flight

// How rows travel: 4-byte copies, 16-byte copies (aligned rows), or TMA boxes
// of one warp's columns (aligned rows of a multiple of 16 columns).
enum { kCopy4, kCopy16, kTma };
constexpr int kSwizzleAlign = 1024;           // TMA: alignment of the ring

// Floats of one ring row of `threads` threads with C columns each: C / 4
// planes of 4 floats per thread, each plane 32 / (C / 4) floats longer so that
// 4-byte copies of 32 consecutive columns meet no bank twice.
template <int C>
__host__ __device__ constexpr int plane_floats(int threads) { return threads * 4 + 128 / C; }
template <int C>
__host__ __device__ constexpr int row_floats(int threads) { return C / 4 * plane_floats<C>(threads); }

// One arriving row e (columns c-1 .. c+C of a thread) added to the outputs
// it touches: o completes the row above, P2 the row itself so far (taps m),
// P1 the row below; taps in row-major order.
struct W3 { float w[3]; };
// ROW_INNER: the columns that need no neighbour's value; ROW_EDGES: the others.
enum { ROW_ALL, ROW_INNER, ROW_EDGES };
template <int PART, int C>
__device__ __forceinline__ void add_row(const W9 &w, const W3 &m, const float (&e)[C + 2], float (&P1)[C],
                                        float (&P2)[C], float (&o)[C])
{
#pragma unroll
    for (int j = 0; j < C; ++j) {
        if (PART != ROW_ALL && (j == 0 || j == C - 1) != (PART == ROW_EDGES)) continue;
        o[j] = fmaf(w.w[8], e[j + 2], fmaf(w.w[7], e[j + 1], fmaf(w.w[6], e[j], P2[j])));
        P2[j] = fmaf(m.w[2], e[j + 2], fmaf(m.w[1], e[j + 1], fmaf(m.w[0], e[j], P1[j])));
        P1[j] = fmaf(w.w[2], e[j + 2], fmaf(w.w[1], e[j + 1], fmaf(w.w[0], e[j], 0.f)));
    }
}

// A CLAMP grid's row above row 0 (e: row 0): the sums of row 0 start from it.
template <int PART, int C>
__device__ __forceinline__ void add_row_above(const W9 &w, const float (&e)[C + 2], float (&P1)[C])
{
#pragma unroll
    for (int j = 0; j < C; ++j) {
        if (PART != ROW_ALL && (j == 0 || j == C - 1) != (PART == ROW_EDGES)) continue;
        P1[j] = fmaf(w.w[2], e[j + 2], fmaf(w.w[1], e[j + 1], fmaf(w.w[0], e[j], 0.f)));
    }
}

// Inclusive scan of a thread's values in place (groups of four, then the
// groups' offsets); returns their sum.  REV scans from the last value.
template <bool REV, int C>
__device__ __forceinline__ float scan_thread(float (&v)[C])
{
    constexpr int d = REV ? -1 : 1;
    float off = 0.f;
#pragma unroll
    for (int g = 0; g < C / 4; ++g) {
        const int b = REV ? C - 1 - 4 * g : 4 * g;
        v[b + d] += v[b];
        v[b + 2 * d] += v[b + d];
        v[b + 3 * d] += v[b + 2 * d];
        const float tot = v[b + 3 * d];
        if (g > 0) {
#pragma unroll
            for (int k = 0; k < 4; ++k) v[b + d * k] += off;
        }
        off += tot;
    }
    return off;
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The part of a thread's work both directions share: its columns, the ring,
// the edges of the row.
//
// With TMA the row's layout is the grid's own: 64 bytes per thread, the four
// 16-byte groups swizzled by the lane (SWIZZLE_64B) so that each group's reads
// meet every bank once.  A warp loads, reads, rewrites and stores its own 2 KB
// only, each load completing on the warp's own mbarrier of the slot, so the
// copies need no block barrier and take none of the load/store unit's issue:
// the plane copies of 16 bytes per lane (32 KB per row in 64 instructions,
// queued ahead of the shuffles and edge reads behind the barrier) cost the
// forward 57 of its 183 us and the backward 67 of 241 (timed without them).
template <int MODE, int C, int R>
struct RowStream {
    static constexpr int NP = C / 4;   // planes
    int nthr, lane, warp, nwarps, nv, pf;
    int64_t rows, cols;
    bool lead, trail, cedge;      // first / last column of the row here; the warp touches either or a column past the grid
    float *ring;
    uint32_t ring_s;
    const float *next;            // row of the next copy, at this thread's first element
    int nrows, ncopied;
    // TMA
    const CUtensorMap *tin, *tout;
    Control *ctl;
    uint32_t bar_s;               // the warp's R mbarriers
    int q0i;                      // first row of the block
    bool ok;                      // no wait has run out

    __device__ __forceinline__ RowStream(const float *in, int64_t rows_, int64_t cols_, int64_t q0, int nin, float *ring_,
                                         const CUtensorMap *tin_, const CUtensorMap *tout_, Control *ctl_)
    {
        nthr = blockDim.x;
        lane = threadIdx.x & 31;
        warp = threadIdx.x >> 5;
        nwarps = nthr >> 5;
        rows = rows_;
        cols = cols_;
        pf = plane_floats<C>(nthr);
        const int c0 = C * threadIdx.x;
        const int n = (int)cols - c0;
        nv = n < 0 ? 0 : (n > C ? C : n);
        lead = threadIdx.x == 0;
        trail = n > 0 && n <= C;
        cedge = warp == 0 || (warp + 1) * 32 * C >= cols;
        ring = MODE == kTma ? ring_ + (0u - (uint32_t)__cvta_generic_to_shared(ring_)) % kSwizzleAlign / 4 : ring_;
        ring_s = (uint32_t)__cvta_generic_to_shared(ring);
        next = in + q0 * cols;
        nrows = nin;
        ncopied = 0;
        tin = tin_;
        tout = tout_;
        ctl = ctl_;
        q0i = (int)q0;
        ok = true;
        if constexpr (MODE == kTma) {
            bar_s = ring_s + (uint32_t)(R * nthr * C) * 4u + (uint32_t)(warp * R) * 8u;
            if (lane == 0) {
#pragma unroll
                for (int k = 0; k < R; ++k)
                    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(bar_s + 8u * k) : "memory");
                asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            __syncwarp();
        }
    }
    // zeroes the columns past the grid (only the warps that hold some)
    __device__ __forceinline__ void mask(float (&v)[C]) const
    {
        if (cedge) {
#pragma unroll
            for (int j = 0; j < C; ++j) v[j] = j < nv ? v[j] : 0.f;
        }
    }
    __device__ __forceinline__ float *slot(int i) const { return ring + (i % R) * NP * pf; }
    // TMA: the warp's part of slot i, and this thread's p-th 16-byte group in it
    __device__ __forceinline__ uint32_t tma_slot(int i) const
    {
        return ring_s + (uint32_t)((i % R) * nthr + warp * 32) * (C * 4);
    }
    __device__ __forceinline__ float *tma_group(int i, int p) const
    {
        return ring + ((i % R) * nthr + (int)threadIdx.x) * C + 4 * (p ^ (lane >> 1 & 3));
    }
    // Starts the copy of the next row, if there is one.  TMA: the store out of
    // its slot, at most PENDING stores back, must have left shared memory.
    template <int PENDING>
    __device__ __forceinline__ void copy_next()
    {
        if constexpr (MODE == kTma) {
            if (ncopied < nrows && ok) {
                if (lane == 0) {
                    const uint32_t bar = bar_s + 8u * (uint32_t)(ncopied % R);
                    asm volatile("cp.async.bulk.wait_group.read %0;" :: "n"(PENDING) : "memory");
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(32 * C * 4) : "memory");
                    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                                 " [%0], [%1, {%2, %3, %4}], [%5];"
                                 :: "r"(tma_slot(ncopied)), "l"(tin), "r"(0), "r"(warp * 32), "r"(q0i + ncopied), "r"(bar)
                                 : "memory");
                }
                ++ncopied;
            }
            return;
        }
        if (ncopied < nrows) {
            const uint32_t d = ring_s + (uint32_t)((ncopied % R) * NP * pf) * 4u;
            if (MODE == kCopy16) {
#pragma unroll
                for (int m = 0; m < NP; ++m) {  // group q of four columns: plane q % NP, thread q / NP
                    const int q = m * nthr + threadIdx.x;
                    if (4 * q < cols) dev::cp_async16(d + (uint32_t)((q % NP) * pf + (q / NP) * 4) * 4u, next + 4 * q);
                }
            } else {
#pragma unroll
                for (int m = 0; m < C; ++m) {
                    const int e = m * nthr + threadIdx.x;
                    if (e < cols) dev::cp_async4(d + (uint32_t)((e / 4 % NP) * pf + (e / C) * 4 + e % 4) * 4u, next + e);
                }
            }
            next += cols;
            ++ncopied;
        }
        dev::cp_commit();
    }
    // this thread's copies but the last N have landed (not with TMA)
    template <int N>
    __device__ __forceinline__ void landed() const
    {
        if constexpr (MODE != kTma) dev::cp_wait<N>();
    }
    // TMA: row i of the warp has landed.  After a bounded number of tries the
    // error is recorded and the block goes on without copies or waits.
    __device__ __forceinline__ bool await_once(int i) const
    {
        uint32_t done = 0;
        for (uint32_t it = 0; it < (1u << 22) && !done; ++it)
            asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                         : "=r"(done) : "r"(bar_s + 8u * (uint32_t)(i % R)), "r"((uint32_t)(i / R & 1)) : "memory");
        return __all_sync(0xffffffffu, done != 0);
    }
    __device__ __forceinline__ void await(int i)
    {
        if constexpr (MODE == kTma) {
            if (ok && !await_once(i)) {
                ok = false;
                if (lane == 0) atomicOr(&ctl->error, kErrTimeout);
            }
        }
    }
    __device__ __forceinline__ void read(int i, float (&v)[C]) const
    {
        const float *s = slot(i) + 4 * threadIdx.x;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const float4 q = *reinterpret_cast<const float4 *>(MODE == kTma ? tma_group(i, p) : s + p * pf);
            v[4 * p] = q.x; v[4 * p + 1] = q.y; v[4 * p + 2] = q.z; v[4 * p + 3] = q.w;
        }
    }
    // Writes v into the slot of row i (the warp's own part of it) and from
    // there to row r of the grid out.  The warp's lanes have read the slot.
    __device__ __forceinline__ void write(int i, const float (&v)[C], float *out, int64_t r) const
    {
        if constexpr (MODE == kTma) {
            __syncwarp();
#pragma unroll
            for (int p = 0; p < NP; ++p)
                *reinterpret_cast<float4 *>(tma_group(i, p)) = make_float4(v[4 * p], v[4 * p + 1], v[4 * p + 2], v[4 * p + 3]);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0)
                asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];"
                             :: "l"(tout), "r"(0), "r"(warp * 32), "r"((int)r), "r"(tma_slot(i)) : "memory");
            return;
        }
        float *s = slot(i), *dst = out + r * cols;
        __syncwarp();
#pragma unroll
        for (int p = 0; p < NP; ++p)
            *reinterpret_cast<float4 *>(s + p * pf + 4 * threadIdx.x) =
                make_float4(v[4 * p], v[4 * p + 1], v[4 * p + 2], v[4 * p + 3]);
        __syncwarp();
        if (MODE == kCopy16) {
#pragma unroll
            for (int m = 0; m < NP; ++m) {
                const int q = warp * 32 * NP + 32 * m + lane;
                if (4 * q < cols)
                    *reinterpret_cast<float4 *>(dst + 4 * q) =
                        *reinterpret_cast<const float4 *>(s + (q % NP) * pf + (q / NP) * 4);
            }
        } else {
#pragma unroll
            for (int m = 0; m < C; ++m) {
                const int e = warp * 32 * C + 32 * m + lane;
                if (e < cols) dst[e] = s[(e / 4 % NP) * pf + (e / C) * 4 + e % 4];
            }
        }
    }
    // TMA: closes the iteration's group of stores (which may be empty).
    __device__ __forceinline__ void end_stores() const
    {
        if constexpr (MODE == kTma) {
            if (lane == 0) asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
    }
    // Every copy of the thread has ended (three loads at most are in flight).
    __device__ __forceinline__ void drain() const
    {
        if constexpr (MODE == kTma) {
            if (!ok)
                for (int k = ncopied > 3 ? ncopied - 3 : 0; k < ncopied; ++k) await_once(k);
            if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        } else {
            dev::cp_wait<0>();
        }
    }
};

// What a row's warps tell each other between two barriers.
struct Exchange {
    float first[kLWarps], last[kLWarps];   // the warps' outermost columns
    float total[kLWarps];                  // scan: the warps' sums
};

// The forward's barrier, in two halves so that work which needs nothing of the
// other warps stands between them: every warp arrives, later waits until all
// have.  One mbarrier, one phase per row; the wait is bounded as the copies' is.
struct BlockSync {
    uint32_t bar;
    uint32_t phase;
    bool ok;

    __device__ __forceinline__ BlockSync(uint64_t *b, int nwarps)   // a __syncthreads follows
    {
        bar = (uint32_t)__cvta_generic_to_shared(b);
        phase = 0;
        ok = true;
        if (threadIdx.x == 0) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(bar), "r"(nwarps) : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
    }
    __device__ __forceinline__ void arrive(int lane) const
    {
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(bar) : "memory");
    }
    __device__ __forceinline__ void wait(Control *ctl)
    {
        uint32_t done = ok ? 0u : 1u;
        for (uint32_t it = 0; it < (1u << 22) && !done; ++it)
            asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                         : "=r"(done) : "r"(bar), "r"(phase) : "memory");
        phase ^= 1u;
        if (!done) {
            ok = false;
            atomicOr(&ctl->error, kErrTimeout);
        }
        __syncwarp();
    }
};

// The columns c-1 and c+C of the row v, from the neighbouring lanes; 0 where
// they are another warp's or outside the row.
template <int C>
__device__ __forceinline__ void neighbours(const float (&v)[C], int lane, float (&e)[C + 2])
{
    const float l = __shfl_up_sync(0xffffffffu, v[C - 1], 1), r = __shfl_down_sync(0xffffffffu, v[0], 1);
    e[0] = lane == 0 ? 0.f : l;
    e[C + 1] = lane == 31 ? 0.f : r;
#pragma unroll
    for (int j = 0; j < C; ++j) e[j + 1] = v[j];
}
// The same from the neighbouring warps, whose part of ex is complete.
template <int C>
__device__ __forceinline__ void warp_neighbours(const Exchange &ex, int lane, int warp, int nwarps, float (&e)[C + 2])
{
    if (lane == 0 && warp > 0) e[0] = ex.last[warp - 1];
    if (lane == 31 && warp + 1 < nwarps) e[C + 1] = ex.first[warp + 1];
}

// The exclusive form of a warp scan's inclusive value (not wi minus the
// lane's own sum: that would round once more, and carry a NaN backwards).
template <bool REV>
__device__ __forceinline__ float warp_exclusive(float wi, int lane)
{
    const float q = REV ? __shfl_down_sync(0xffffffffu, wi, 1) : __shfl_up_sync(0xffffffffu, wi, 1);
    return lane == (REV ? 31 : 0) ? 0.f : q;
}

// Sum of the totals of the warps before (REV: after) `warp`: each half-warp
// adds them up in a tree.
constexpr int kOffsetLanes = 16;
static_assert(kLMaxCols / kFwdC <= 32 * kOffsetLanes && kLMaxCols / kBwdC <= 32 * kOffsetLanes, "a lane per warp");
template <bool REV>
__device__ __forceinline__ float lane_total(const Exchange &ex, int lane, int warp, int nwarps)
{
    const int k = lane & (kOffsetLanes - 1);
    return (REV ? k > warp && k < nwarps : k < warp) ? ex.total[k] : 0.f;
}
template <bool REV>
__device__ __forceinline__ float warp_offset(const Exchange &ex, int lane, int warp, int nwarps)
{
    float v = lane_total<REV>(ex, lane, warp, nwarps);
#pragma unroll
    for (int o = kOffsetLanes / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// The same with its rounding errors kept.
template <bool REV>
__device__ __forceinline__ dev::Sum2 warp_offset2(const Exchange &ex, int lane, int warp, int nwarps)
{
    dev::Sum2 r;
    r.hi = lane_total<REV>(ex, lane, warp, nwarps);
    r.add(__shfl_xor_sync(0xffffffffu, r.hi, kOffsetLanes / 2));
#pragma unroll
    for (int o = kOffsetLanes / 4; o > 0; o >>= 1) {
        const float h = __shfl_xor_sync(0xffffffffu, r.hi, o), l = __shfl_xor_sync(0xffffffffu, r.lo, o);
        r.add(h);
        r.lo += l;
    }
    return r;
}

// ------------------------------------------------------------- forward --
template <int MODE>
__global__ void __launch_bounds__(kLMaxCols / kFwdC, 1)
loss_fwd(const __grid_constant__ CUtensorMap tin, const __grid_constant__ CUtensorMap tout, const float *__restrict__ x, float *__restrict__ t_out, int64_t rows, int64_t cols, int b, W9 w, int H,
         double2 *__restrict__ partials, float *__restrict__ L, Control *ctl)
{
    dev::grid_wait();
    constexpr int C = kFwdC;
    extern __shared__ __align__(16) float dyn[];
    __shared__ Exchange ex[2];                // by the row's parity
    __shared__ uint64_t sync_bar;
    __shared__ double2 red[kLWarps];
    __shared__ int am_last;
    const int64_t r0 = (int64_t)blockIdx.x * H, r1 = r0 + H < rows ? r0 + H : rows;
    const int64_t q0 = r0 > 0 ? r0 - 1 : 0;
    const bool top = r0 == 0, bottom = r1 == rows, clamp = b == SKEL_CLAMP;
    const int nin = (int)((bottom ? rows : r1 + 1) - q0);
    RowStream<MODE, C, kFwdRing> rs(x, rows, cols, q0, nin, dyn, &tin, &tout, ctl);
    const int lane = rs.lane, warp = rs.warp;
    BlockSync sync(&sync_bar, rs.nwarps);
    dev::Sum2 su, ss;
    float P1[C], P2[C];
#pragma unroll
    for (int j = 0; j < C; ++j) P1[j] = P2[j] = 0.f;
#pragma unroll
    for (int k = 0; k < kFwdRing - 1; ++k) rs.template copy_next<1>();
    rs.template landed<kFwdRing - 2>();
    __syncthreads();

    auto sum_sq = [&](float (&o)[C], dev::Sum2 &k) {   // the grid's columns only
        rs.mask(o);
        float q[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < C; ++j) q[j & 3] = fmaf(o[j], o[j], q[j & 3]);
        k.add((q[0] + q[1]) + (q[2] + q[3]));
    };
    // t of row i (its copy has landed)
    auto load_t = [&](int i, float (&v)[C]) {
        rs.await(i);
        rs.read(i, v);
#pragma unroll
        for (int j = 0; j < C; ++j) v[j] = tanhf(v[j]);
        rs.mask(v);
    };
    const W3 mid{{w.w[3], w.w[4], w.w[5]}};
    float e[C + 2], v[C];
    load_t(0, v);
    for (int i = 0; i < nin; ++i) {
        Exchange &exi = ex[i & 1];
        const int64_t row = q0 + i;
        const bool own = row >= r0 && row < r1;
        if (t_out && own) rs.write(i, v, t_out, row);
        rs.end_stores();
        float sc[C];
#pragma unroll
        for (int j = 0; j < C; ++j) sc[j] = v[j];
        const float wi = dev::warp_incl_scan_add(scan_thread<false>(sc));
        if (lane == 0) exi.first[warp] = v[0];
        if (lane == 31) {
            exi.last[warp] = v[C - 1];
            exi.total[warp] = wi;
        }
        rs.template landed<kFwdRing - 3>();   // row i + 1 has landed (its copies by every thread, after the barrier)
        sync.arrive(lane);
        neighbours(v, lane, e);
        if (rs.cedge) {
            if (rs.lead) e[0] = clamp ? v[0] : 0.f;
#pragma unroll
            for (int j = 1; j <= C; ++j)   // the column after the grid's last one
                if (rs.trail && j == rs.nv) e[j + 1] = clamp ? v[j - 1] : 0.f;
        }
        const bool above = top && i == 0 && clamp;   // ZERO: the sums start from 0
        float o[C];
        if (above) add_row_above<ROW_INNER>(w, e, P1);
        add_row<ROW_INNER>(w, mid, e, P1, P2, o);
        // the next row's tanh, independent of this row's sums: the two overlap
        if (MODE == kTma && i + 1 < nin) load_t(i + 1, v);
        sync.wait(ctl);
        if (MODE != kTma && i + 1 < nin) load_t(i + 1, v);
        warp_neighbours<C>(exi, lane, warp, rs.nwarps, e);
        if (above) add_row_above<ROW_EDGES>(w, e, P1);
        add_row<ROW_EDGES>(w, mid, e, P1, P2, o);
        if (row > r0) sum_sq(o, su);         // u of row - 1
        if (own) {
            const float base = warp_offset<false>(exi, lane, warp, rs.nwarps) + warp_exclusive<false>(wi, lane);
#pragma unroll
            for (int j = 0; j < C; ++j) sc[j] += base;
            sum_sq(sc, ss);
        }
        rs.template copy_next<1>();   // into the slot of row i - 1; here, behind the row's other work: 136 us, right after the barrier 140
    }
    if (bottom) {                            // the row below the last one
        float o[C];
        if (!clamp) {
#pragma unroll
            for (int j = 0; j < C + 2; ++j) e[j] = 0.f;
        }
        add_row<ROW_ALL>(w, mid, e, P1, P2, o);
        sum_sq(o, su);
    }
    rs.drain();
    double a = warp_sum(su.value()), c = warp_sum(ss.value());
    if (lane == 0) red[warp] = make_double2(a, c);
    __syncthreads();
    if (warp == 0) {
        a = warp_sum(lane < rs.nwarps ? red[lane].x : 0.0);
        c = warp_sum(lane < rs.nwarps ? red[lane].y : 0.0);
        if (lane == 0) {
            partials[blockIdx.x] = make_double2(a, c);
            __threadfence();
            am_last = atomicAdd(&ctl->done, 1u) == gridDim.x - 1;
        }
    }
    __syncthreads();
    if (!am_last || warp != 0) return;
    __threadfence();
    a = c = 0.0;
    for (int k = lane; k < (int)gridDim.x; k += 32) {
        const double2 p = __ldcg(partials + k);
        a += p.x;
        c += p.y;
    }
    a = warp_sum(a);
    c = warp_sum(c);
    if (lane == 0) {
        *L = (float)(a + c / ((double)rows * (double)cols));
        ctl->done = 0u;
    }
}

// ------------------------------------------------------------ backward --
// Iteration i takes row q0 + i of t in, completes u of the row above it (the
// upstream gradient gu = 2 g u of the second stencil), and completes gx of
// the row above that.
template <int MODE>
__global__ void __launch_bounds__(kLMaxCols / kBwdC, 1)
loss_bwd(const __grid_constant__ CUtensorMap tin, const __grid_constant__ CUtensorMap tout, const float *__restrict__ t, const float *__restrict__ g, float *__restrict__ gx, int64_t rows, int64_t cols,
         int b, W9 w, int H, Control *ctl)
{
    dev::grid_wait();
    constexpr int C = kBwdC;
    extern __shared__ __align__(16) float dyn[];
    __shared__ Exchange ex[2];                // of phase 1 (t and the scan) and of phase 2 (gu and the reverse scan)
    const int64_t r0 = (int64_t)blockIdx.x * H, r1 = r0 + H < rows ? r0 + H : rows;
    const int64_t q0 = r0 > 2 ? r0 - 2 : 0;
    const bool clamp = b == SKEL_CLAMP;
    const int nin = (int)((r1 + 2 < rows ? r1 + 2 : rows) - q0), niter = (int)(r1 + 2 - q0);
    // the iterations of rows 1, `rows` (past them if it is not reached) and r0 + 2
    const int i1 = q0 > 1 ? -1 : (int)(1 - q0), ilast = rows - q0 < niter ? (int)(rows - q0) : niter, iout = (int)(r0 + 2 - q0);
    RowStream<MODE, C, kBwdRing> rs(t, rows, cols, q0, nin, dyn, &tin, &tout, ctl);
    const int lane = rs.lane, warp = rs.warp;
    const float g2 = 2.f * __ldg(g), gc2 = 2.f * ((float)(1.0 / ((double)rows * (double)cols)) * __ldg(g));
    W9 wt;                                    // the mirrored taps of the adjoint
#pragma unroll
    for (int k = 0; k < 9; ++k) wt.w[k] = w.w[8 - k];
    float P1[C], P2[C], Q1[C], Q2[C];
#pragma unroll
    for (int j = 0; j < C; ++j) P1[j] = P2[j] = Q1[j] = Q2[j] = 0.f;
    float L1 = 0.f, L2 = 0.f, R1 = 0.f, R2 = 0.f;   // the columns beside the grid (below)
#pragma unroll
    for (int k = 0; k < 3; ++k) rs.template copy_next<0>();
    rs.template landed<2>();
    __syncthreads();

    for (int i = 0; i < niter; ++i) {
        const bool out_row = i >= iout;       // row q0 + i - 2 is one of the block's (below r1 by the loop's bound)
        // ---- phase 1: the arriving row, the scan of row - 2 ----
        float v[C];
        if (i < nin) rs.await(i);
        rs.read(i < nin ? i : nin - 1, v);    // below the grid: the last row again (ZERO: 0)
        rs.mask(v);
        if (i >= nin && !clamp) {
#pragma unroll
            for (int j = 0; j < C; ++j) v[j] = 0.f;
        }
        float sc[C], wi = 0.f;
        if (out_row) {
            rs.read(i - 2, sc);
            rs.mask(sc);
            wi = dev::warp_incl_scan_add(scan_thread<false>(sc));
        }
        if (lane == 0) ex[0].first[warp] = v[0];
        if (lane == 31) {
            ex[0].last[warp] = v[C - 1];
            ex[0].total[warp] = wi;
        }
        __syncthreads();
        if (MODE != kTma) rs.template copy_next<0>();   // into the slot of row i - 3
        // ---- phase 2: u of row - 1, the reverse scan of row - 2 ----
        float e[C + 2];
        neighbours(v, lane, e);
        warp_neighbours<C>(ex[0], lane, warp, rs.nwarps, e);
        if (rs.cedge) {
            if (rs.lead) e[0] = clamp ? v[0] : 0.f;
#pragma unroll
            for (int j = 1; j <= C; ++j)
                if (rs.trail && j == rs.nv) e[j + 1] = clamp ? v[j - 1] : 0.f;
        }
        float u[C];
        if (i == i1 - 1 && clamp) add_row_above<ROW_ALL>(w, e, P1);
        add_row<ROW_ALL>(w, W3{{w.w[3], w.w[4], w.w[5]}}, e, P1, P2, u);
        if (i >= i1 && i <= ilast) {                       // the row above is a row of the grid
#pragma unroll
            for (int j = 0; j < C; ++j) u[j] *= g2;
            rs.mask(u);
        } else {
#pragma unroll
            for (int j = 0; j < C; ++j) u[j] = 0.f;
        }
        float rwi = 0.f;
        if (out_row) {
            const float base = warp_offset<false>(ex[0], lane, warp, rs.nwarps) + warp_exclusive<false>(wi, lane);
#pragma unroll
            for (int j = 0; j < C; ++j) sc[j] = gc2 * (sc[j] + base);
            rs.mask(sc);
            rwi = scan_thread<true>(sc);           // the warp's reverse inclusive scan of the threads' sums
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const float q = __shfl_down_sync(0xffffffffu, rwi, d);
                if (lane + d < 32) rwi += q;
            }
        }
        if (lane == 0) {
            ex[1].first[warp] = u[0];
            ex[1].total[warp] = rwi;
        }
        if (lane == 31) ex[1].last[warp] = u[C - 1];
        rs.template landed<2>();                   // row i + 1 has landed (visible after the barrier)
        __syncthreads();
        if (MODE == kTma) rs.template copy_next<0>();   // here: the slot's store has had this row's two phases to end
        // ---- phase 3: the adjoint stencil of row - 2, gx of row - 2 ----
        float back = 0.f;                     // the reverse scan's offset; formed before the stencil: both passes 301 us, after it 306
        if (out_row) {
            const dev::Sum2 off = warp_offset2<true>(ex[1], lane, warp, rs.nwarps);
            back = off.hi + (off.low() + warp_exclusive<true>(rwi, lane));
        }
        neighbours(u, lane, e);               // 0 outside the grid
        warp_neighbours<C>(ex[1], lane, warp, rs.nwarps, e);
        // CLAMP: taps that the forward clamped onto the grid's edge.  The
        // first row also receives what the row above it would, the last row
        // what the row below would: those taps join the middle row's when
        // that row arrives.  What the columns beside the grid would receive
        // (one tap per row of the first, and of the last, column) is summed
        // apart and added to the edge column.
        W3 m{{wt.w[3], wt.w[4], wt.w[5]}};
        if (clamp && i == i1) {
#pragma unroll
            for (int k = 0; k < 3; ++k) m.w[k] += wt.w[6 + k];
        }
        if (clamp && i == ilast) {
#pragma unroll
            for (int k = 0; k < 3; ++k) m.w[k] += wt.w[k];
        }
        float gt[C];
        add_row<ROW_ALL>(wt, m, e, Q1, Q2, gt);
        if (clamp && rs.cedge) {
            float ul = 0.f;                   // the thread's last column of the grid
#pragma unroll
            for (int j = 0; j < C; ++j) ul = j < rs.nv ? u[j] : ul;
            const float ol = fmaf(wt.w[8], u[0], L2), orr = fmaf(wt.w[6], ul, R2);
            L2 = fmaf(m.w[2], u[0], L1);
            R2 = fmaf(m.w[0], ul, R1);
            L1 = wt.w[2] * u[0];
            R1 = wt.w[0] * ul;
            gt[0] += rs.lead ? ol : 0.f;
#pragma unroll
            for (int j = 0; j < C; ++j) gt[j] += rs.trail && j == rs.nv - 1 ? orr : 0.f;
        }
        if (out_row) {
            float y[C];
            rs.read(i - 2, y);
#pragma unroll
            for (int j = 0; j < C; ++j) y[j] = (gt[j] + (sc[j] + back)) * fmaf(-y[j], y[j], 1.f);
            rs.write(i - 2, y, gx, q0 + i - 2);
        }
        rs.end_stores();
    }
    rs.drain();
}

// Threads of a block with C columns each: whole warps.
int threads_for(int64_t cols, int C) { return (int)ceil_div(cols, 32 * C) * 32; }

// Rows per block: one wave of blocks, but at least min_rows (the halo rows
// and the ring's start-up are per block).
int rows_per_block(int64_t rows, int occ, int min_rows)
{
    int64_t H = ceil_div(rows, (int64_t)device_info().sms * occ);
    return (int)(H < min_rows ? min_rows : H);
}

// A grid as rows of 16-column groups, in boxes of one warp's 32 groups.
bool encode_rows(CUtensorMap *map, const float *p, int64_t rows, int64_t cols)
{
    EncodeTiled enc = encode_tiled();
    if (!enc) return false;
    const cuuint64_t dims[3] = {16, (cuuint64_t)(cols / 16), (cuuint64_t)rows};
    const cuuint64_t strides[2] = {64, (cuuint64_t)cols * 4};
    const cuuint32_t box[3] = {16, 32, 1}, estr[3] = {1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float *>(p), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Dynamic shared memory: the ring, and with TMA its alignment and the warps' mbarriers.
template <int MODE, int C, int R>
int ring_bytes(int nthr)
{
    return MODE == kTma ? kSwizzleAlign + R * nthr * C * 4 + nthr / 32 * R * 8 : R * row_floats<C>(nthr) * 4;
}

template <int MODE>
int run_fwd(const LossLaunch &l, const CUtensorMap &tin, const CUtensorMap &tout, cudaStream_t s)
{
    const int nthr = threads_for(l.cols, kFwdC), smem = ring_bytes<MODE, kFwdC, kFwdRing>(nthr);
    auto kern = loss_fwd<MODE>;
    const int occ = kernel_occupancy(kern, nthr, smem);
    if (occ < 1) return fail(SKEL_ERR_UNSUPPORTED, "composed loss: kernel does not fit an SM");
    const int H = rows_per_block(l.rows, occ, 4);
    const int64_t grid = ceil_div(l.rows, (int64_t)H);
    Scratch scr{};
    int rc = get_scratch(s, (size_t)grid * sizeof(double2), 0, &scr);
    if (rc) return rc;
    W9 w;
    for (int k = 0; k < 9; ++k) w.w[k] = l.w[k];
    launch_kernel(kern, (unsigned)grid, nthr, (size_t)smem, s, tin, tout, l.x, l.t, l.rows, l.cols, l.boundary, w, H,
                  reinterpret_cast<double2 *>(scr.data), l.L, scr.ctl);
    cudaError_t e = cudaPeekAtLastError();
    return e == cudaSuccess ? SKEL_OK : fail_cuda(cudaGetLastError(), "composed loss launch");
}

template <int MODE>
int run_bwd(const LossLaunch &l, const CUtensorMap &tin, const CUtensorMap &tout, cudaStream_t s)
{
    const int nthr = threads_for(l.cols, kBwdC), smem = ring_bytes<MODE, kBwdC, kBwdRing>(nthr);
    auto kern = loss_bwd<MODE>;
    const int occ = kernel_occupancy(kern, nthr, smem);
    if (occ < 1) return fail(SKEL_ERR_UNSUPPORTED, "composed loss: kernel does not fit an SM");
    const int H = rows_per_block(l.rows, occ, 4);
    Scratch scr{};
    int rc = get_scratch(s, 0, 0, &scr);
    if (rc) return rc;
    W9 w;
    for (int k = 0; k < 9; ++k) w.w[k] = l.w[k];
    launch_kernel(kern, (unsigned)ceil_div(l.rows, (int64_t)H), nthr, (size_t)smem, s, tin, tout, (const float *)l.t, l.g,
                  l.gx, l.rows, l.cols, l.boundary, w, H, scr.ctl);
    cudaError_t e = cudaPeekAtLastError();
    return e == cudaSuccess ? SKEL_OK : fail_cuda(cudaGetLastError(), "composed loss adjoint launch");
}

}  // namespace

int loss_fused_check(int64_t rows, int64_t cols, int boundary)
{
    if (boundary == SKEL_PERIODIC) return fail(SKEL_ERR_UNSUPPORTED, "composed loss: PERIODIC is not fused");
    if (rows < 1 || cols < 1 || cols > kLMaxCols)
        return fail(SKEL_ERR_UNSUPPORTED, "composed loss: fused for 1 to 8192 columns");
    if (rows > 0x7fffffff) return fail(SKEL_ERR_UNSUPPORTED, "composed loss: too many rows");
    return SKEL_OK;
}

int launch_loss(const LossLaunch &l, cudaStream_t s)
{
    const bool back = l.gx != nullptr;
    const float *in = back ? l.t : l.x;
    float *out = back ? l.gx : l.t;
    const bool vec = l.cols % 4 == 0 && aligned16(in) && aligned16(out);
    CUtensorMap tin{}, tout{};
    if (vec && l.cols % 16 == 0 && encode_rows(&tin, in, l.rows, l.cols) && (!out || encode_rows(&tout, out, l.rows, l.cols)))
        return back ? run_bwd<kTma>(l, tin, tout, s) : run_fwd<kTma>(l, tin, tout, s);
    if (vec) return back ? run_bwd<kCopy16>(l, tin, tout, s) : run_fwd<kCopy16>(l, tin, tout, s);
    return back ? run_bwd<kCopy4>(l, tin, tout, s) : run_fwd<kCopy4>(l, tin, tout, s);
}

}  // namespace skel
