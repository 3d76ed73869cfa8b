// Scan variant 9 (the other variants and the dispatch are in k_scan.cu): a
// sequence that fits the SMs' shared memory, scanned in one wave of blocks;
// and row-wise scans, one block per row.
//
// Every block stages its whole chunk in shared memory (cp.async), sums it as
// it lands, publishes the sum, reads the sums of all blocks before it at
// once, and scans its chunk out of shared memory.  The look-back variants
// spend their time in short sequences on ramping up small tiles whose
// prefixes wait on one another (5,000,011 int32: 19.2 us with variant 8, of
// which 6 us are HBM time); here each block waits once, for one exchange of
// at most one word per SM.  One read and one write per element.
//
// A chunk is split into units of 128 elements (one 16-byte group per lane),
// consecutive units to a warp.  A warp copies and sums its own units; warp 0
// scans the warps' sums (float32: in float64), publishes the chunk's, adds
// the predecessors' and hands every warp its carry; a warp then scans its
// units in blocks of four interleaved warp scans from its carry, a float32
// pair.  Row-wise scans skip the exchange.
//
// Measured (us, int32 inclusive / float32 exclusive / float32 reverse, before
// -> now): 2^18 elements 5.9 -> 4.5 / 6.3 -> 5.3 / 4.1 -> 5.3 (the table
// keeps variant 1 for the last), 2^20 6.7 -> 5.9 / 9.8 -> 7.0 / 8.5 -> 7.0,
// 2^22 13.5 -> 9.5 / 15.3 -> 10.6 / 15.4 -> 10.6, 5000011 19.8 -> 11.8 /
// 20.7 -> 12.7 / 28.1 -> 12.2, 2^23 21.1 -> 18.7 / 22.9 -> 19.7 / 23.0 -> 20.1.
// float32 keeps the rounding errors of its sums and adds each element's small
// part first, one rounding at the prefix's magnitude: on U[-1, 1] the error
// against 64 bits is 4.7e-8 (variants 4, 5 and 8: 0.95 to 1.3e-7).
// At 5000011 the HBM time is 6 us; the rest is the launch, the first copies'
// latency, the exchange (about 2 us) and the stores, which cannot overlap
// within one chunk.
//
// Progress: a block's position is a ticket drawn in order, so it waits only
// for blocks that are already running and publish without waiting.  The wait
// is bounded as in the other variants (kErrTimeout and the call's abort tag).
#include <type_traits>

#include "scan_tile.cuh"

namespace skel {
namespace {

using dev::ScanTypes;

constexpr int kUnit = 128;                       // elements per warp scan
constexpr int kWaveMaxWarps = 32;
constexpr int kWaveMaxUnits = 432;               // 55296 elements, 216 KiB of shared memory per block

// A running sum of elements: float32 as dev::Sum2, integers as they are.
template <class T> struct Run;
template <> struct Run<uint32_t> {
    uint32_t hi;
    static constexpr uint32_t lo = 0u;
    __device__ __forceinline__ Run() : hi(0u) {}
    __device__ __forceinline__ explicit Run(uint32_t v) : hi(v) {}
    __device__ __forceinline__ void add(uint32_t v) { hi += v; }
    __device__ __forceinline__ uint32_t low() const { return 0u; }
    __device__ __forceinline__ uint32_t value() const { return hi; }
};
template <> struct Run<float> : dev::Sum2 {
    Run() = default;
    __device__ __forceinline__ explicit Run(double v) : dev::Sum2(v) {}
};
__device__ __forceinline__ void set_lo(Run<uint32_t> &, uint32_t) {}
__device__ __forceinline__ void set_lo(Run<float> &r, float lo) { r.lo = lo; }
__device__ __forceinline__ Run<uint32_t> warp_total(Run<uint32_t> r)
{
    r.hi = dev::warp_reduce<dev::AddU>(r.hi);
    return r;
}
__device__ __forceinline__ Run<float> warp_total(Run<float> r)
{
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const float h = __shfl_xor_sync(0xffffffffu, r.hi, d), l = __shfl_xor_sync(0xffffffffu, r.lo, d);
        r.add(h);
        r.lo += l;
    }
    return r;
}

// Shuffles of the carry type.
__device__ __forceinline__ uint32_t shfl_up_ct(uint32_t v, int d) { return __shfl_up_sync(0xffffffffu, v, d); }
__device__ __forceinline__ double shfl_up_ct(double v, int d) { return __shfl_up_sync(0xffffffffu, v, d); }

struct WaveGeom {
    int64_t n;          // elements of the sequence, or of a row
    int64_t chunk;      // elements per block (a multiple of 128)
    int64_t blocks;
    bool rows;          // one row of n elements per block
    bool vin, vout;     // 16-byte aligned chunk starts
};

template <class T, bool INCL, bool REV>
__global__ void __launch_bounds__(kWaveMaxWarps * 32)
scan_wave(const T *__restrict__ in, T *__restrict__ out, WaveGeom g, uint64_t *__restrict__ words, Control *ctl,
          uint32_t epoch, int64_t skip_block, uint64_t limit_ns)
{
    dev::grid_wait();
    using CT = typename ScanTypes<T>::CT;
    using V4 = typename ScanTypes<T>::V4;
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ T wtotal[2][kWaveMaxWarps];        // hi and lo
    __shared__ T wcarry[2][kWaveMaxWarps];
    __shared__ uint32_t s_ticket;
    T *buf = reinterpret_cast<T *>(dyn);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int64_t t = blockIdx.x;                       // position in scan order
    if (!g.rows && g.blocks > 1) {
        if (threadIdx.x == 0) {
            s_ticket = atomicAdd(&ctl->ticket, 1u);
            if ((int64_t)s_ticket == g.blocks - 1) ctl->ticket = 0u;   // every block has drawn
        }
        __syncthreads();
        t = s_ticket;
    }
    const int64_t p = g.rows || !REV ? t : g.blocks - 1 - t;   // position in memory
    const int64_t base = g.rows ? p * g.n : p * g.chunk;
    const int64_t left = g.rows ? g.n : g.n - base;
    const int len = (int)(left < g.chunk ? left : g.chunk);
    const int units = (len + kUnit - 1) / kUnit;
    const int u0 = w * units / nw, u1 = (w + 1) * units / nw;   // this warp's units
    const T *src = in + base;
    const bool vin = g.vin, vout = g.vout;

    // ---- copy the warp's units, in two groups ----
    const uint32_t sbuf = (uint32_t)__cvta_generic_to_shared(buf);
    auto copy = [&](int a, int b) {
        for (int u = a; u < b; ++u) {
            const int e0 = u * kUnit;
            if (e0 + kUnit <= len) {
                if (vin) {
                    dev::cp_async16(sbuf + (uint32_t)(e0 + 4 * lane) * 4u, reinterpret_cast<const float *>(src + e0 + 4 * lane));
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        dev::cp_async4(sbuf + (uint32_t)(e0 + 32 * k + lane) * 4u,
                                       reinterpret_cast<const float *>(src + e0 + 32 * k + lane));
                }
            } else {                              // the last, partial unit: zeros behind the end
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int e = e0 + 32 * k + lane;
                    buf[e] = e < len ? src[e] : T(0);
                }
            }
        }
        dev::cp_commit();
    };
    const int um = (u0 + u1 + 1) / 2;
    copy(u0, um);
    copy(um, u1);
    // ---- the warp's sum ----
    Run<T> acc;
    auto sum = [&](int a, int b) {
        for (int u = a; u < b; ++u) {
            const V4 q = *reinterpret_cast<const V4 *>(buf + u * kUnit + 4 * lane);
            acc.add((q.x + q.y) + (q.z + q.w));
        }
    };
    dev::cp_wait<1>();
    __syncwarp();
    sum(u0, um);
    dev::cp_wait<0>();
    __syncwarp();
    sum(um, u1);
    acc = warp_total(acc);
    if (lane == 0) {
        wtotal[0][w] = acc.hi;
        wtotal[1][w] = acc.lo;
    }
    __syncthreads();
    // ---- warp 0: the warps' offsets, the exchange between blocks ----
    if (w == 0) {
        const int k = REV ? nw - 1 - lane : lane;               // lanes in scan order
        Run<T> own;
        if (lane < nw) {
            own.hi = wtotal[0][k];
            set_lo(own, wtotal[1][k]);
        }
        CT incl = own.value();
#pragma unroll
        for (int d = 1; d < kWaveMaxWarps; d <<= 1) {
            const CT v = shfl_up_ct(incl, d);
            if (lane >= d) incl = incl + v;
        }
        CT excl = shfl_up_ct(incl, 1);
        if (lane == 0) excl = CT(0);
        if (!g.rows && g.blocks > 1) {
            if (lane == 31 && t != skip_block) dev::Codec<CT>::put(words + t, incl, epoch);   // the chunk's sum
            CT pre = CT(0);
            bool gave_up = false;
            uint64_t t0 = 0;
            for (int64_t j0 = 0; j0 < t; j0 += 32) {
                const int64_t j = j0 + lane;
                CT v = CT(0);
                bool ready = j >= t;
                while (true) {
                    if (!ready) ready = dev::Codec<CT>::get(words + j, epoch, v);
                    if (__all_sync(0xffffffffu, ready) || gave_up) break;
                    if (t0 == 0) t0 = dev::globaltimer();
                    const bool expired = dev::globaltimer() - t0 > limit_ns || dev::ld_volatile(&ctl->abort) == epoch;
                    if (__any_sync(0xffffffffu, expired)) {
                        if (lane == 0) {
                            atomicOr(&ctl->error, kErrTimeout);
                            atomicExch(&ctl->abort, epoch);
                        }
                        gave_up = true;
                    }
                }
                if (ready && j < t) pre = pre + v;
            }
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) pre = pre + __shfl_xor_sync(0xffffffffu, pre, d);
            excl = excl + pre;
        }
        if (lane < nw) {
            const Run<T> c(excl);
            wcarry[0][k] = c.hi;
            wcarry[1][k] = c.lo;
        }
    }
    __syncthreads();
    // ---- scan the warp's units from its carry ----
    Run<T> carry;
    carry.hi = wcarry[0][w];
    set_lo(carry, wcarry[1][w]);
    T *dst = out + base;
    // unit number i in scan order (of this warp)
    auto unit_at = [&](int i) { return REV ? u1 - 1 - i : u0 + i; };
    // N units from number i on: interleaved warp scans, then the stores
    auto scan_units = [&](int i, auto n_t) {
        constexpr int N = decltype(n_t)::value;
        const T hi = carry.hi, lo = carry.low();
        T loc = T(0);
        V4 o[N];
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const int u = unit_at(i + k);
            const V4 q = *reinterpret_cast<const V4 *>(buf + u * kUnit + (REV ? kUnit - 4 - 4 * lane : 4 * lane));
            const T x0 = REV ? q.w : q.x, x1 = REV ? q.z : q.y, x2 = REV ? q.y : q.z, x3 = REV ? q.x : q.w;
            const T s0 = x0, s1 = s0 + x1, s2 = s1 + x2, s3 = s2 + x3;
            const T wi = dev::warp_incl_scan_add(s3);
            T lex = __shfl_up_sync(0xffffffffu, wi, 1);
            if (lane == 0) lex = T(0);
            // the small parts first: one rounding at the prefix's magnitude
            const T b = lo + (loc + lex);
            const T y0 = hi + (INCL ? b + s0 : b), y1 = hi + (INCL ? b + s1 : b + s0), y2 = hi + (INCL ? b + s2 : b + s1),
                    y3 = hi + (INCL ? b + s3 : b + s2);
            if (REV) { o[k].x = y3; o[k].y = y2; o[k].z = y1; o[k].w = y0; }
            else { o[k].x = y0; o[k].y = y1; o[k].z = y2; o[k].w = y3; }
            loc = loc + __shfl_sync(0xffffffffu, wi, 31);
        }
        carry.add(loc);
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const int e0 = unit_at(i + k) * kUnit, e = e0 + (REV ? kUnit - 4 - 4 * lane : 4 * lane);
            if (vout && e0 + kUnit <= len) {
                dev::st_stream(reinterpret_cast<V4 *>(dst + e), o[k]);
            } else {                              // through the unit's own shared memory
                __syncwarp();
                *reinterpret_cast<V4 *>(buf + e) = o[k];
                __syncwarp();
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int q = e0 + 32 * m + lane;
                    if (q < len) dst[q] = buf[q];
                }
            }
        }
    };
    int i = 0;
    const int cnt = u1 - u0;
    for (; i + 4 <= cnt; i += 4) scan_units(i, std::integral_constant<int, 4>{});
    if (i + 2 <= cnt) {
        scan_units(i, std::integral_constant<int, 2>{});
        i += 2;
    }
    if (i < cnt) scan_units(i, std::integral_constant<int, 1>{});
}

template <class T, bool INCL, bool REV>
int launch_wave(const ScanLaunch &sc, cudaStream_t s)
{
    const bool rows = sc.seg > 0 && sc.seg < sc.n;
    WaveGeom g{};
    g.n = rows ? sc.seg : sc.n;
    g.rows = rows;
    if (rows) {
        g.blocks = sc.n / sc.seg;
        g.chunk = ceil_div(g.n, (int64_t)kUnit) * kUnit;
    } else {
        // one block per SM, but at least 2048 elements each
        const int64_t most = device_info().sms, want = ceil_div(sc.n, (int64_t)2048);
        g.blocks = want < most ? want : most;
        g.chunk = ceil_div(ceil_div(sc.n, g.blocks), (int64_t)kUnit) * kUnit;
        g.blocks = ceil_div(sc.n, g.chunk);
    }
    const int units = (int)(g.chunk / kUnit);
    const bool whole = !rows || g.n % 4 == 0;     // every block starts at a multiple of 4 elements
    g.vin = whole && aligned16(sc.in);
    g.vout = whole && aligned16(sc.out);
    int nw = (units + 1) / 2;                     // two units per warp and more
    if (nw > kWaveMaxWarps) nw = kWaveMaxWarps;
    if (rows) nw = (units + 3) / 4 < kWaveMaxWarps ? (units + 3) / 4 : kWaveMaxWarps;   // several blocks share an SM
    const int smem = units * kUnit * (int)sizeof(T);
    auto kern = scan_wave<T, INCL, REV>;
    if (kernel_occupancy(kern, 32 * nw, kWaveMaxUnits * kUnit * (int)sizeof(T)) < 1)
        return fail(SKEL_ERR_UNSUPPORTED, "scan wave: kernel does not fit an SM");
    Scratch scr{};
    int rc = get_scratch(s, 0, rows ? 0 : (size_t)g.blocks, &scr);
    if (rc) return rc;
    const DebugKnobs k = debug_knobs();
    launch_kernel(kern, (unsigned)g.blocks, 32 * nw, (size_t)smem, s, static_cast<const T *>(sc.in),
                  static_cast<T *>(sc.out), g, scr.words, scr.ctl, scr.epoch, k.scan_skip_publish_tile, k.wait_limit_ns);
    const cudaError_t e = cudaPeekAtLastError();
    return e == cudaSuccess ? SKEL_OK : fail_cuda(cudaGetLastError(), "scan wave launch");
}

template <class T>
int run_wave(const ScanLaunch &sc, cudaStream_t s)
{
    if (sc.inclusive) return sc.reverse ? launch_wave<T, true, true>(sc, s) : launch_wave<T, true, false>(sc, s);
    return sc.reverse ? launch_wave<T, false, true>(sc, s) : launch_wave<T, false, false>(sc, s);
}

}  // namespace

bool scan_wave_fits(const ScanLaunch &sc)
{
    constexpr int64_t most = (int64_t)kWaveMaxUnits * kUnit;
    if (sc.seg > 0 && sc.seg < sc.n) return sc.seg <= most && sc.n / sc.seg <= 0x7fffffffLL;
    return sc.n <= most * device_info().sms;
}

int scan_wave_launch(const ScanLaunch &sc, cudaStream_t s)
{
    if (!scan_wave_fits(sc))
        return fail(SKEL_ERR_UNSUPPORTED, "scan wave: the sequence exceeds the SMs' shared memory");
    if (sc.dtype == SKEL_F32) return run_wave<float>(sc, s);
    if (sc.dtype == SKEL_I32) return run_wave<uint32_t>(sc, s);
    return fail(SKEL_ERR_DTYPE, "scan: float32 or int32 only");
}

}  // namespace skel
