// A composed chain of three skeleton calls selected as a whole (Sec. II:
// composition of components, implementations selected for the composition
// rather than call by call):
//
//   t = Map f(x)                 f one of TANH, SQ, SCALE, COPY
//   u = MapOverlap S t           2D, radius 1 (5-point or 3x3 weights)
//   result = MapReduce(sq, +) u  sum of squares
//
// Variant 0 (per_call, in api.cpp) runs the three calls, each dispatched as
// usual, through two n-element temporaries: 8 + 8 + 4 = 20 bytes per point
// of HBM traffic.  Variants 1 and 2 (fused, here) read x once, 4 bytes per
// point, in one launch: 1 needs 16-byte aligned rows, 2 takes any.
//
// A warp walks a strip of 128 columns down a segment of rows (the row stream
// of k_stream.cu with one step): rows arrive through a shared-memory ring,
// f is applied on arrival, the stencil keeps the partial tap sums of its next
// two rows in registers, neighbours come by shuffle, and each finished row's
// squares go into the lane's sum (with its rounding errors kept).  Every
// offered f has f(0) = 0, so a ZERO boundary pads t as it pads x.  The
// outputs use the stencil skeleton's operations, so u is the same float per
// point as in variant 0.  Lanes, warps and blocks are added in float64; the
// last block to finish adds the blocks' sums in index order.
//
// What bounds it: instruction issue (tanhf is about 18 of some 33
// instructions per point, two of them on the 16-per-clock special function
// units); see the measurements at compose_warps.
#include <type_traits>

#include "stencil.cuh"

namespace skel {
namespace {

constexpr int kCWarps = 4;                        // warps per block
constexpr int kCHalo = 4, kCOut = kStripCols - 2 * kCHalo;   // halo columns on each side, columns summed

template <bool TAPS5, int FN, bool VEC>
__global__ void __launch_bounds__(32 * kCWarps)
compose_stream(const float *__restrict__ in, int64_t rows, int64_t cols, int b, W9 w, float a, int H, int64_t strips,
               int64_t nwork, double *__restrict__ partials, float *__restrict__ out, Control *ctl)
{
    dev::grid_wait();
    __shared__ __align__(16) float ring_all[kCWarps * kStripRing * kStripCols];
    __shared__ double wsum[kCWarps];
    __shared__ int am_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t gw = (int64_t)blockIdx.x * kCWarps + warp;
    double total = 0.0;
    if (gw < nwork) {                                   // warp-uniform
        float *ring = ring_all + warp * kStripRing * kStripCols;
        const int64_t seg = gw / strips, strip = gw - seg * strips;
        const int64_t g0 = strip * kCOut - kCHalo, c0 = g0 + 4 * lane;
        const int64_t r0 = seg * H, r1 = r0 + H < rows ? r0 + H : rows;
        const bool wrap = b == SKEL_PERIODIC, clamp = b == SKEL_CLAMP;
        const int64_t q0 = wrap || r0 >= 1 ? r0 - 1 : 0;                // first input row
        const bool top = !wrap && r0 == 0, bottom = !wrap && r1 == rows;
        const int nin = (int)((bottom ? rows : r1 + 1) - q0);
        const int ifirst = (int)(r0 - q0) + 1;                          // iteration that completes row r0
        const bool cedge = !wrap && (g0 < 0 || g0 + kStripCols > cols); // warp-uniform
        const bool lead = !wrap && c0 == 0, trail = !wrap && c0 + 4 >= cols;
        // columns of the lane that lie in the grid; PERIODIC strips past it sum nothing there either
        const int nv = c0 >= cols ? 0 : (c0 + 4 > cols ? (int)(cols - c0) : 4);
        const bool mine = 4 * lane >= kCHalo && 4 * lane < kCHalo + kCOut && nv > 0;
        StripRing<VEC> rows_in(in, rows, cols, wrap, q0, g0, nin, ring);
        rows_in.start();
        dev::Sum2 sum;
        float P1[4] = {0.f, 0.f, 0.f, 0.f}, P2[4] = {0.f, 0.f, 0.f, 0.f}, e[6];
        auto square = [&](float (&o)[4]) {
            if (!VEC && nv < 4) {                       // the grid ends inside the lane
#pragma unroll
                for (int j = 1; j < 4; ++j) o[j] = j < nv ? o[j] : 0.f;
            }
            sum.add((o[0] * o[0] + o[1] * o[1]) + (o[2] * o[2] + o[3] * o[3]));
        };
        auto walk = [&](auto cole_t) {
            constexpr bool COLE = decltype(cole_t)::value;
#pragma unroll 2
            for (int i = 0; i < nin; ++i) {
                dev::cp_wait<kStripRing - 2>();
                __syncwarp();
                const float4 q = *reinterpret_cast<const float4 *>(ring + (i & (kStripRing - 1)) * kStripCols + 4 * lane);
                rows_in.copy(i + kStripRing - 1);
                float x[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) x[j] = dev::MapF<FN>::f(x[j], 0.f, a);
                if (COLE && !VEC) {
#pragma unroll
                    for (int j = 1; j < 4; ++j) x[j] = trail && nv <= j ? (clamp ? x[j - 1] : 0.f) : x[j];
                }
                float l = __shfl_up_sync(0xffffffffu, x[3], 1), r = __shfl_down_sync(0xffffffffu, x[0], 1);
                if (COLE) {
                    l = lead ? (clamp ? x[0] : 0.f) : l;
                    r = trail ? (clamp ? x[3] : 0.f) : r;
                }
                e[0] = l;
                e[5] = r;
#pragma unroll
                for (int j = 0; j < 4; ++j) e[j + 1] = x[j];
                if (i == 0 && top && clamp) {           // the row above row 0
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float p = 0.f;
                        if (!TAPS5) p = fmaf(w.w[0], e[j], p);
                        p = fmaf(w.w[1], e[j + 1], p);
                        if (!TAPS5) p = fmaf(w.w[2], e[j + 2], p);
                        P1[j] = p;
                    }
                }
                float o[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float s = P2[j], n = 0.f;
                    if (!TAPS5) s = fmaf(w.w[6], e[j], s);
                    s = fmaf(w.w[7], e[j + 1], s);
                    if (!TAPS5) s = fmaf(w.w[8], e[j + 2], s);
                    o[j] = s;
                    P2[j] = fmaf(w.w[5], e[j + 2], fmaf(w.w[4], e[j + 1], fmaf(w.w[3], e[j], P1[j])));
                    if (!TAPS5) n = fmaf(w.w[0], e[j], n);
                    n = fmaf(w.w[1], e[j + 1], n);
                    if (!TAPS5) n = fmaf(w.w[2], e[j + 2], n);
                    P1[j] = n;
                }
                if (i >= ifirst) square(o);
            }
        };
        if (cedge) walk(std::true_type{});
        else walk(std::false_type{});
        if (bottom) {                                   // the row below the last one: it again, or zeros
            float o[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float s = P2[j];
                if (!TAPS5) s = fmaf(w.w[6], clamp ? e[j] : 0.f, s);
                s = fmaf(w.w[7], clamp ? e[j + 1] : 0.f, s);
                if (!TAPS5) s = fmaf(w.w[8], clamp ? e[j + 2] : 0.f, s);
                o[j] = s;
            }
            square(o);
        }
        dev::cp_wait<0>();
        total = mine ? sum.value() : 0.0;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) total += __shfl_xor_sync(0xffffffffu, total, d);
    if (lane == 0) wsum[warp] = total;
    __syncthreads();
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = (wsum[0] + wsum[1]) + (wsum[2] + wsum[3]);
        __threadfence();
        am_last = atomicAdd(&ctl->done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    total = 0.0;
    for (int k = threadIdx.x; k < (int)gridDim.x; k += 32 * kCWarps) total += __ldcg(partials + k);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) total += __shfl_xor_sync(0xffffffffu, total, d);
    if (lane == 0) wsum[warp] = total;
    __syncthreads();
    if (threadIdx.x == 0) {
        *out = (float)((wsum[0] + wsum[1]) + (wsum[2] + wsum[3]));
        ctl->done = 0u;
    }
}

// Warps per SM of the launch's one wave (tile 0, 1, 2).  Measured (tanh,
// 9-point, 8192 x 8192): 100.7 / 105.2 / 108.7 us, COPY 62.5 / 64.3 / 65.3,
// HBM 39; the column walk through registers that this replaces took 125 us
// and a second launch, the three calls 202.  ncu: 44 instructions per point,
// issued at 82 % of the peak rate.  4097 x 4099: 35.8 us, three calls 59.3.
// The table takes it from 2^14 points (64 x 64: 4.8 us, three calls 4.4).
int compose_warps(int tile) { return tile == 0 ? 32 : tile == 1 ? 24 : 16; }

template <bool TAPS5, int FN, bool VEC>
int run_fn(const ComposeLaunch &cl, int tile, float *out, cudaStream_t s)
{
    auto kern = compose_stream<TAPS5, FN, VEC>;
    const int occ = kernel_occupancy(kern, 32 * kCWarps, 0);
    if (occ < 1) return fail(SKEL_ERR_UNSUPPORTED, "fused chain: kernel does not fit an SM");
    const int64_t strips = ceil_div(cl.cols, (int64_t)kCOut);
    const int fill = occ * kCWarps < compose_warps(tile) ? occ * kCWarps : compose_warps(tile);
    int64_t segs = (int64_t)device_info().sms * fill / strips;
    if (segs < 1) segs = 1;
    int64_t H = ceil_div(cl.rows, segs);
    if (H < 4) H = 4;                                  // two more rows are read than summed
    if (H > (1 << 20)) H = 1 << 20;
    const int64_t nwork = strips * ceil_div(cl.rows, H), grid = ceil_div(nwork, (int64_t)kCWarps);
    if (grid > 0x7fffffffLL) return fail(SKEL_ERR_SHAPE, "fused chain: grid too large");
    Scratch scr{};
    int rc = get_scratch(s, (size_t)grid * sizeof(double), 0, &scr);
    if (rc) return rc;
    W9 w;
    for (int k = 0; k < 9; ++k) w.w[k] = cl.w[k];
    launch_kernel(kern, (unsigned)grid, 32 * kCWarps, 0, s, cl.in, cl.rows, cl.cols, cl.boundary, w, cl.a, (int)H, strips,
                  nwork, reinterpret_cast<double *>(scr.data), out, scr.ctl);
    cudaError_t e = cudaPeekAtLastError();
    return e == cudaSuccess ? SKEL_OK : fail_cuda(cudaGetLastError(), "fused chain launch");
}

template <bool TAPS5, bool VEC>
int run_taps(const ComposeLaunch &cl, int tile, float *out, cudaStream_t s)
{
    switch (cl.map_fn) {
    case SKEL_FN_TANH: return run_fn<TAPS5, SKEL_FN_TANH, VEC>(cl, tile, out, s);
    case SKEL_FN_SQ: return run_fn<TAPS5, SKEL_FN_SQ, VEC>(cl, tile, out, s);
    case SKEL_FN_SCALE: return run_fn<TAPS5, SKEL_FN_SCALE, VEC>(cl, tile, out, s);
    case SKEL_FN_COPY: return run_fn<TAPS5, SKEL_FN_COPY, VEC>(cl, tile, out, s);
    default: return fail(SKEL_ERR_UNSUPPORTED, "fused chain: map function not offered");
    }
}

}  // namespace

int launch_compose_fused(const ComposeLaunch &cl, const Choice &c, float *out, cudaStream_t s)
{
    if (c.tile < 0 || c.tile > 2) return fail(SKEL_ERR_INVALID_ARG, "fused chain: tile must be 0..2");
    const bool vec = cl.cols % 4 == 0 && aligned16(cl.in);
    if (c.variant == 1 && !vec)
        return fail(SKEL_ERR_UNSUPPORTED, "fused chain: 16-byte aligned rows needed (cols % 4 == 0)");
    if (vec) return cl.taps5 ? run_taps<true, true>(cl, c.tile, out, s) : run_taps<false, true>(cl, c.tile, out, s);
    return cl.taps5 ? run_taps<true, false>(cl, c.tile, out, s) : run_taps<false, false>(cl, c.tile, out, s);
}

int compose_variant_count() { return 3; }
const char *compose_variant_name(int v)
{
    static const char *names[] = {"per_call", "fused", "fused_any"};
    return v >= 0 && v < 3 ? names[v] : "?";
}
Choice compose_default() { return Choice{0, 0, 0, 0}; }

}  // namespace skel
