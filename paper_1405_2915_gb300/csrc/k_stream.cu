// 2D MapOverlap (radius 1) as a stream of rows: one kernel for K = 1..8
// steps of the same stencil in one pass over the grid (temporal blocking),
// any alignment and any number of columns.
//
// A warp owns a strip of 128 columns (4 per lane) and walks down a segment of
// rows.  Row q of the input enters stage 1; stage s turns row q of step s-1
// into row q-1 of step s, which enters stage s+1 in the same iteration, and
// the row that leaves stage K is stored.  A stage keeps no rows: it keeps,
// for its next two outputs, the sums of the taps whose rows have arrived
// (P1: the top row's taps, P2: the top and middle rows'), 8 registers per
// stage, and adds an arriving row's taps to three outputs at once.  Each
// output still accumulates its taps in row-major order (stencil9's order), so
// K fused steps equal K single calls bit for bit.  The two columns beside a
// lane's four come from its neighbours by shuffle (two per row and stage).
//
// A strip's outer columns lose one valid column per step and side, so it
// stores its middle 128 - 2*HL columns (HL: K rounded up to 4, which keeps
// 16-byte rows aligned); a segment of H rows starts K rows early and runs K
// rows late.  Input rows come through a ring of 8 rows per warp in shared
// memory filled by cp.async (16 bytes per lane where rows are 16-byte
// aligned, else four coalesced 4-byte copies), so about 3.5 KiB per warp are
// in flight without holding registers.
//
// Boundaries.  CLAMP / ZERO cells outside the grid hold what a single call
// reads there, at every step: columns by selecting the lane's own edge value
// or 0 instead of the shuffled neighbour; the row above the grid by starting
// the accumulators from row 0 (or 0); rows below it from a copy of the
// stage's last row kept in shared memory (only warps whose rows touch an edge
// run that code).  PERIODIC wraps the rows and columns that are loaded.
//
// What bounds it: one step on aligned rows streams at 5.6 TB/s (8192 x 8192:
// 96 us; the TMA tile of k_stencil.cu, without halo columns to reload, 82 us,
// stays the choice there); unaligned rows run at 4.1 TB/s (4097 x 4099: 33
// us, against 141 us for nine cached loads per point).  Several steps are
// bound by instruction issue: per row of 4 columns and stage 36 FMAs (5-point
// 20), two shuffles and about 11 others, issued at 75 % of the peak rate
// (register-port conflicts of three-operand FMAs hold the rest).  8192 x
// 8192, K = 5: 175 us (5-point 119) a pass, against 317 (280) for a shared-
// memory tile whose every step read and wrote its whole tile there.  Packed
// two-column FMAs (fma.rn.f32x2) halve the FMA issues but not the FMA pipe's
// time, and the register moves that pair the columns cost more than they
// save (223 / 166 us); 8 columns per lane measured the same on large grids
// (166 / 121) and slower on small ones.
#include <type_traits>

#include "stencil.cuh"

namespace skel {
namespace {

constexpr int kStreamWarps = 4;   // warps per block

template <int K>
struct StreamGeom {
    static constexpr int HL = (K + 3) / 4 * 4;           // halo columns on each side, whole lanes
    static constexpr int W = kStripCols - 2 * HL;       // output columns per strip
    // rows of shared memory per warp: the ring, a held row per stage, a row being stored
    static constexpr int rows = kStripRing + K + 1;
    static constexpr int smem_bytes = kStreamWarps * rows * kStripCols * 4;
};

// VEC: rows start on 16-byte boundaries (in, out aligned, cols % 4 == 0).
// FOLD (one step, ZERO): the adjoint of a CLAMP stencil: w are the mirrored
// taps, and what a cell beside the grid would receive goes to the edge cell it
// stands for (taps that the forward pass clamped onto that cell).
// H: output rows per segment; strips: strips per row of the grid; nwork:
// strips * segments.
template <bool TAPS5, int K, bool VEC, bool FOLD>
__global__ void __launch_bounds__(32 * kStreamWarps)
st2_stream(const float *__restrict__ in, float *__restrict__ out, int64_t rows, int64_t cols, int b, W9 w, int H,
           int64_t strips, int64_t nwork)
{
    dev::grid_wait();
    using G = StreamGeom<K>;
    constexpr int C = 4, SW = kStripCols, RING = kStripRing;
    extern __shared__ __align__(16) float sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t gw = (int64_t)blockIdx.x * kStreamWarps + warp;
    if (gw >= nwork) return;   // no block-wide barrier below
    float *ring = sm + warp * G::rows * SW, *hold = ring + RING * SW, *srow = hold + K * SW;
    // the last segment first: the slower edge segments must not end the launch
    const int64_t segs = nwork / strips, sk = gw / strips, strip = gw - sk * strips, seg = sk == 0 ? segs - 1 : sk - 1;
    const int64_t s0 = strip * G::W;                    // first output column
    const int64_t g0 = s0 - G::HL;                      // column of the strip's element 0
    const int64_t c0 = g0 + C * lane;                   // first of this lane's columns
    const int64_t r0 = seg * H, r1 = r0 + H < rows ? r0 + H : rows;
    const bool wrap = b == SKEL_PERIODIC, clamp = b == SKEL_CLAMP;
    // first input row; segments at the top start at row 0 (PERIODIC: wrapped)
    const int64_t q0 = wrap || r0 >= K ? r0 - K : 0;
    const int niter = (int)(r1 - q0) + K;
    const int ifirst = (int)(r0 - q0) + K;              // iteration that completes output row r0
    const bool top = !wrap && q0 == 0;                  // row 0's accumulators start from the boundary
    const bool bottom = !wrap && r1 + K > rows;
    // arrivals with this index or more lie below the grid
    const int nin = bottom ? (int)(rows - q0) : niter;
    const bool cedge = !wrap && (g0 < 0 || g0 + SW > cols);    // warp-uniform
    const bool lead = !wrap && c0 == 0, trail = !wrap && c0 + C >= cols;
    const int nv = trail ? (int)(cols - c0) : C;        // grid columns of the lane (<= 0: none)

    StripRing<VEC> rows_in(in, rows, cols, wrap, q0, g0, nin, ring);
    rows_in.start();

    float P1[K][C], P2[K][C];
#pragma unroll
    for (int s = 0; s < K; ++s)
#pragma unroll
        for (int j = 0; j < C; ++j) P1[s][j] = P2[s][j] = 0.f;

    const bool mine = C * lane >= G::HL && C * lane < G::HL + G::W && c0 < cols;   // VEC: the lane's columns are stored
    float *orow = out + r0 * cols + (VEC ? c0 : s0);                  // the next output row
    auto store = [&](const float (&x)[C]) {
        if (VEC) {
            if (mine) *reinterpret_cast<float4 *>(orow) = make_float4(x[0], x[1], x[2], x[3]);
        } else {
            *reinterpret_cast<float4 *>(srow + C * lane) = make_float4(x[0], x[1], x[2], x[3]);
            __syncwarp();
#pragma unroll
            for (int k = 0; k < (G::W + 31) / 32; ++k) {
                const int e = 32 * k + lane;
                if (e < G::W && s0 + e < cols) orow[e] = srow[G::HL + e];
            }
        }
        orow += cols;
    };
    // Iterations [i0, i1).  ROWE: a row of some stage may lie at or past the
    // edge of the grid's rows; COLE: a column of the strip may.
    auto walk = [&](int i0, int i1, auto rowe_t, auto cole_t) {
        constexpr bool ROWE = decltype(rowe_t)::value, COLE = decltype(cole_t)::value;
#pragma unroll 1
        for (int i = i0; i < i1; ++i) {
            dev::cp_wait<RING - 2>();
            __syncwarp();   // the row has landed for every lane; the last row's readers are done
            const float4 q = *reinterpret_cast<const float4 *>(ring + (i & (RING - 1)) * SW + C * lane);
            float x[C] = {q.x, q.y, q.z, q.w};
            rows_in.copy(i + RING - 1);
#pragma unroll
            for (int s = 0; s < K; ++s) {
                if (ROWE) {
                    const int a = i - s;   // the arriving row of step s, relative to q0
                    float4 *h = reinterpret_cast<float4 *>(hold + s * SW + C * lane);
                    if (a == nin - 1) *h = make_float4(x[0], x[1], x[2], x[3]);
                    if (a >= nin) {
                        const float4 p = *h;
                        x[0] = clamp ? p.x : 0.f; x[1] = clamp ? p.y : 0.f;
                        x[2] = clamp ? p.z : 0.f; x[3] = clamp ? p.w : 0.f;
                    }
                }
                if (COLE && !VEC) {   // columns past the grid inside the lane
#pragma unroll
                    for (int j = 1; j < C; ++j) x[j] = nv <= j ? (clamp ? x[j - 1] : 0.f) : x[j];
                }
                float e[C + 2];   // columns c0 - 1 .. c0 + C
                e[0] = __shfl_up_sync(0xffffffffu, x[C - 1], 1);
                e[C + 1] = __shfl_down_sync(0xffffffffu, x[0], 1);
#pragma unroll
                for (int j = 0; j < C; ++j) e[j + 1] = x[j];
                if (COLE) {
                    e[0] = lead ? (clamp ? x[0] : 0.f) : e[0];
                    e[C + 1] = trail ? (clamp ? x[C - 1] : 0.f) : e[C + 1];
                }
                if (ROWE) {
                    if (top && i == s) {   // the row above row 0
#pragma unroll
                        for (int j = 0; j < C; ++j) {
                            float p = 0.f;
                            if (!TAPS5) p = fmaf(w.w[0], clamp ? e[j] : 0.f, p);
                            p = fmaf(w.w[1], clamp ? e[j + 1] : 0.f, p);
                            if (!TAPS5) p = fmaf(w.w[2], clamp ? e[j + 2] : 0.f, p);
                            P1[s][j] = p;
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    float o = P2[s][j];
                    if (!TAPS5) o = fmaf(w.w[6], e[j], o);
                    o = fmaf(w.w[7], e[j + 1], o);
                    if (!TAPS5) o = fmaf(w.w[8], e[j + 2], o);
                    x[j] = o;   // (e still holds the row)
                    P2[s][j] = fmaf(w.w[5], e[j + 2], fmaf(w.w[4], e[j + 1], fmaf(w.w[3], e[j], P1[s][j])));
                    float n = 0.f;
                    if (!TAPS5) n = fmaf(w.w[0], e[j], n);
                    n = fmaf(w.w[1], e[j + 1], n);
                    if (!TAPS5) n = fmaf(w.w[2], e[j + 2], n);
                    P1[s][j] = n;
                }
                if (FOLD && (ROWE || COLE)) {
                    // the first row also receives what the row above the grid would, the last row what the row below would
                    const bool up = ROWE && top && i == 0, down = ROWE && bottom && i == nin - 1;
#pragma unroll
                    for (int j = 0; j < C; ++j) {
                        if (up) {
                            if (!TAPS5) P2[0][j] = fmaf(w.w[6], e[j], P2[0][j]);
                            P2[0][j] = fmaf(w.w[7], e[j + 1], P2[0][j]);
                            if (!TAPS5) P2[0][j] = fmaf(w.w[8], e[j + 2], P2[0][j]);
                        }
                        if (down) {
                            if (!TAPS5) P2[0][j] = fmaf(w.w[0], e[j], P2[0][j]);
                            P2[0][j] = fmaf(w.w[1], e[j + 1], P2[0][j]);
                            if (!TAPS5) P2[0][j] = fmaf(w.w[2], e[j + 2], P2[0][j]);
                        }
                        if (!COLE) continue;
                        // likewise the columns beside the grid: one tap per row of the first, of the last column
                        const float v = e[j + 1];
                        if (lead && j == 0) {
                            P2[0][j] = fmaf(w.w[5], v, P2[0][j]);
                            if (!TAPS5) {
                                x[j] = fmaf(w.w[8], v, x[j]);
                                P1[0][j] = fmaf(w.w[2], v, P1[0][j]);
                                if (up) P2[0][j] = fmaf(w.w[8], v, P2[0][j]);
                                if (down) P2[0][j] = fmaf(w.w[2], v, P2[0][j]);
                            }
                        }
                        if (trail && j == nv - 1) {
                            P2[0][j] = fmaf(w.w[3], v, P2[0][j]);
                            if (!TAPS5) {
                                x[j] = fmaf(w.w[6], v, x[j]);
                                P1[0][j] = fmaf(w.w[0], v, P1[0][j]);
                                if (up) P2[0][j] = fmaf(w.w[6], v, P2[0][j]);
                                if (down) P2[0][j] = fmaf(w.w[0], v, P2[0][j]);
                            }
                        }
                    }
                }
            }
            if (i >= ifirst) store(x);
        }
    };
    // the rows at the top, between the edges, and at the bottom
    const int e0 = top ? (K < niter ? K : niter) : 0, e1 = bottom ? (nin - 1 > e0 ? nin - 1 : e0) : niter;
    using T = std::true_type;
    using F = std::false_type;
#pragma unroll 1
    for (int part = 0; part < 3; ++part) {
        const int i0 = part == 0 ? 0 : part == 1 ? e0 : e1, i1 = part == 0 ? e0 : part == 1 ? e1 : niter;
        if (part != 1) walk(i0, i1, T{}, T{});
        else if (cedge) walk(i0, i1, F{}, T{});
        else walk(i0, i1, F{}, F{});
    }
    dev::cp_wait<0>();
}

// Rows per segment: one wave of kStreamFill warps per SM, so that the 2K
// extra rows of a segment stay a small share (8192 x 8192, K = 5, 9-point:
// 8 / 16 / 32 warps per SM 425 / 285 / 250 us in the first version, 16 and 32
// within 3 % in this one; K = 1 slower with 32), but at least K rows, below
// which the extra rows cost more than the shorter walk saves (512 x 512,
// K = 5: 2K, K rows 18.8, 14.6 us).
constexpr int kStreamFill = 16;

template <bool TAPS5, int K, bool VEC, bool FOLD = false>
int run_stream(const float *in, float *out, int64_t rows, int64_t cols, int b, const W9 &w, cudaStream_t s)
{
    using G = StreamGeom<K>;
    auto kern = st2_stream<TAPS5, K, VEC, FOLD>;
    const int occ = kernel_occupancy(kern, 32 * kStreamWarps, G::smem_bytes);
    if (occ < 1) return fail(SKEL_ERR_UNSUPPORTED, "mapoverlap stream: kernel does not fit an SM");
    const int64_t strips = ceil_div(cols, (int64_t)G::W);
    const int fill = occ * kStreamWarps < kStreamFill ? occ * kStreamWarps : kStreamFill;
    int64_t segs = (int64_t)device_info().sms * fill / strips;
    if (segs < 1) segs = 1;
    int64_t H = ceil_div(rows, segs);
    if (H < K) H = K;
    if (H < 2) H = 2;
    if (H > (1 << 20)) H = 1 << 20;
    const int64_t nwork = strips * ceil_div(rows, H);
    const int64_t grid = ceil_div(nwork, (int64_t)kStreamWarps);
    if (grid > 0x7fffffffLL) return fail(SKEL_ERR_SHAPE, "mapoverlap stream: grid too large");
    launch_kernel(kern, (unsigned)grid, 32 * kStreamWarps, (size_t)G::smem_bytes, s, in, out, rows, cols, b, w, (int)H,
                  strips, nwork);
    cudaError_t e = cudaPeekAtLastError();
    return e == cudaSuccess ? SKEL_OK : fail_cuda(cudaGetLastError(), "mapoverlap stream launch");
}

template <bool TAPS5, int K>
int run_stream_k(const float *in, float *out, int64_t rows, int64_t cols, int b, const W9 &w, cudaStream_t s)
{
    return cols % 4 == 0 && aligned16(in) && aligned16(out) ? run_stream<TAPS5, K, true>(in, out, rows, cols, b, w, s)
                                                            : run_stream<TAPS5, K, false>(in, out, rows, cols, b, w, s);
}

template <bool TAPS5>
int run_stream_taps(int k, const float *in, float *out, int64_t rows, int64_t cols, int b, const W9 &w, cudaStream_t s)
{
    switch (k) {
    case 1: return run_stream_k<TAPS5, 1>(in, out, rows, cols, b, w, s);
    case 2: return run_stream_k<TAPS5, 2>(in, out, rows, cols, b, w, s);
    case 3: return run_stream_k<TAPS5, 3>(in, out, rows, cols, b, w, s);
    case 4: return run_stream_k<TAPS5, 4>(in, out, rows, cols, b, w, s);
    case 5: return run_stream_k<TAPS5, 5>(in, out, rows, cols, b, w, s);
    case 6: return run_stream_k<TAPS5, 6>(in, out, rows, cols, b, w, s);
    case 7: return run_stream_k<TAPS5, 7>(in, out, rows, cols, b, w, s);
    case 8: return run_stream_k<TAPS5, 8>(in, out, rows, cols, b, w, s);
    default: return fail(SKEL_ERR_INVALID_ARG, "mapoverlap chain: steps per pass must be 1..8");
    }
}

template <bool TAPS5>
int run_stream_fold(const float *in, float *out, int64_t rows, int64_t cols, const W9 &w, cudaStream_t s)
{
    return cols % 4 == 0 && aligned16(in) && aligned16(out)
               ? run_stream<TAPS5, 1, true, true>(in, out, rows, cols, SKEL_ZERO, w, s)
               : run_stream<TAPS5, 1, false, true>(in, out, rows, cols, SKEL_ZERO, w, s);
}

}  // namespace

int launch_stream2d_fold(bool taps5, const float *in, float *out, int64_t rows, int64_t cols, const float *w9,
                         cudaStream_t s)
{
    W9 w;
    for (int q = 0; q < 9; ++q) w.w[q] = w9[q];
    return taps5 ? run_stream_fold<true>(in, out, rows, cols, w, s) : run_stream_fold<false>(in, out, rows, cols, w, s);
}

int launch_stream2d(bool taps5, int k, const float *in, float *out, int64_t rows, int64_t cols, int b, const float *w9,
                    cudaStream_t s)
{
    W9 w;
    for (int q = 0; q < 9; ++q) w.w[q] = w9[q];
    return taps5 ? run_stream_taps<true>(k, in, out, rows, cols, b, w, s)
                 : run_stream_taps<false>(k, in, out, rows, cols, b, w, s);
}

}  // namespace skel
