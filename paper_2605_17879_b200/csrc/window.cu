// Windowed per-series median: for every (rank, metric) series the exact median of its
// last n ring steps.
#include <math_constants.h>

#include <climits>
#include <mutex>

#include "colselect.cuh"
#include "kernels.h"
#include "thselect.cuh"
#include "warpselect.cuh"
#include "xrank_common.cuh"

namespace guard {

namespace {

// ---------------------------------------------------------------------------------------
// Warp-per-series path for windows of up to 256 steps: the window of one series lives in
// the registers of one warp (VPL keys per lane), so no shared-memory column limits the
// number of resident warps.  A CTA of 32 warps handles a tile of 32 adjacent series; tiles
// are staged into a double buffer with one bulk asynchronous copy (TMA) per ring row onto
// an mbarrier per buffer (plain cp.async when rows are not 16-byte aligned).  Rows are
// pitched 36 words apart: 16-byte aligned for the bulk copy, and a column read then costs
// four shared-memory wavefronts instead of thirty-two.
//
// Selection: every lane sorts its own keys (odd-even merge network).  The median of the
// lanes' middle keys (a 32-key bitonic sort over shuffles) is a pivot within a few ranks of
// the wanted one; every lane counts its keys below / not above the pivot and one
// __reduce_add_sync gives the pivot's global rank.  From there the warp walks rank by rank
// (each lane offers its next key, __reduce_min/max_sync picks the winner) until it passes
// the wanted rank; if the pivot turns out to be far off, further pivot rounds (middle key of
// the longest still-active run) narrow the distance first.  Every round removes at least its
// pivot from the active set, so the loop is bounded by the window length.
// ---------------------------------------------------------------------------------------
constexpr int kWarpTileCols = 32;
constexpr int kWarpPitch = 36;

__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// A first guess of the half-width the thread path should search around a series' smoothed
// median: 0.36 x the mean absolute deviation of the window about its median (for Gaussian
// noise that spans about +-0.29 sigma, some 3 standard errors of a 200-step median and ~22 %
// of the window).  Only a starting point: the thread path re-tunes it from its own counts.
template <int VPL>
__device__ __forceinline__ float warp_spread_guess(const uint32_t (&kv)[VPL], const int n, const float med) {
    float s = 0.0f;
#pragma unroll
    for (int i = 0; i < VPL; ++i)
        if (kv[i] != 0xFFFFFFFFu) s += fabsf(key2f(kv[i]) - med);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    return 0.36f * s / (float)n;
}

template <int VPL>
__global__ void __launch_bounds__(1024, 2) window_warp_kernel(const WindowArgs a, const int ntiles, const int use_bulk) {
    pdl_wait();
    extern __shared__ __align__(128) uint32_t wbuf[];   // 2 x [n][kWarpPitch]
    __shared__ __align__(8) uint64_t bar[2];
    const int tid = threadIdx.x, lane = lane_id(), w = warp_id();
    const int n = a.n;
    const int first = a.last_slot - (n - 1) + (a.last_slot < n - 1 ? a.capacity : 0);
    const int bufwords = n * kWarpPitch;

    auto stage = [&](int tile, int b) {
        uint32_t *buf = wbuf + b * bufwords;
        const int col0 = tile * kWarpTileCols;
        const int ncols = min(kWarpTileCols, a.series - col0);
        if (use_bulk) {
            if (tid == 0) mbar_arrive_expect_tx(&bar[b], (uint32_t)n * (uint32_t)ncols * 4u);
            __syncthreads();   // the expectation is registered before any copy can complete
            // lane l of warp w issues rows w + 32 l, w + 32 l + 1024, ...: a warp's bulk copies are
            // issued one lane after the other, so they are spread over all warps
            for (int row = w + 32 * lane; row < n; row += 1024) {
                int slot = first + row;
                if (slot >= a.capacity) slot -= a.capacity;
                bulk_g2s(buf + row * kWarpPitch, a.ring + (size_t)slot * a.row_stride + col0, (uint32_t)ncols * 4u, &bar[b]);
            }
        } else {
            for (int e = tid; e < n * kWarpTileCols; e += 1024) {
                const int row = e >> 5, c = e & 31;
                int slot = first + row;
                if (slot >= a.capacity) slot -= a.capacity;
                if (c < ncols) cp_async4(buf + row * kWarpPitch + c, a.ring + (size_t)slot * a.row_stride + col0 + c);
            }
            cp_async_commit();
        }
    };

    if (use_bulk && tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
    }
    __syncthreads();
    int cur = 0, it = 0;
    if ((int)blockIdx.x < ntiles) stage(blockIdx.x, 0);
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
        const int next = tile + gridDim.x;
        if (next < ntiles) stage(next, cur ^ 1);
        if (use_bulk) {
            // only this first wait takes the caller's (test) limit: the waits below, which let the copies
            // in flight land before the CTA leaves, always get the full one.  The CTA decides as one:
            // if the wait ran out for any thread, all of them leave.
            const bool arrived = mbar_wait_bounded(&bar[cur], (uint32_t)((it >> 1) & 1),
                                                   a.first_wait_cycles > 0 ? a.first_wait_cycles : kWaitLimitCycles);
            if (__syncthreads_or(!arrived)) {
                if (!arrived) atomicOr(a.status, kStatTimeout);
                mbar_wait_bounded(&bar[cur], (uint32_t)((it >> 1) & 1), kWaitLimitCycles);   // let copies in flight land
                if (next < ntiles) mbar_wait_bounded(&bar[cur ^ 1], (uint32_t)(((it + 1) >> 1) & 1), kWaitLimitCycles);
                return;
            }
        } else {
            if (next < ntiles) cp_async_wait<1>(); else cp_async_wait<0>();
            __syncthreads();
        }
        const uint32_t *buf = wbuf + cur * bufwords;
        const int series = tile * kWarpTileCols + w;
        if (series < a.series) {
            uint32_t kv[VPL];
            int nreal = 0;
#pragma unroll
            for (int i = 0; i < VPL; ++i) {
                const int row = lane + 32 * i;
                const bool real = row < n;
                kv[i] = real ? key_of_bits(buf[row * kWarpPitch + w]) : 0xFFFFFFFFu;
                nreal += real;
            }
            lane_sort<VPL>(kv);
            float med = 0.0f;
            const uint32_t hint = (a.use_hint && a.wmed_prev) ? f2key(a.wmed_prev[series]) : 0u;   // last evaluation's median
            const bool ok = warp_median<VPL>(kv, nreal, n, hint, med);
            const float h0 = warp_spread_guess<VPL>(kv, n, med);
            if (lane == 0) {
                if (!ok) atomicOr(a.status, kStatInternal);
                a.wmed[series] = med;
                if (a.spread) a.spread[series] = h0;
                if (a.centre) a.centre[series] = med;
            }
        }
        __syncthreads();   // every warp is done with this buffer before it is refilled
        cur ^= 1;
    }
}

// Function attributes are set once per device and kernel (the calls go to the driver: two of them
// per evaluation showed in the per-step latency of the streaming configuration).
struct AttrOnce {
    std::mutex mu;
    bool done[64] = {};
    int sms[64] = {};
    template <typename F>
    cudaError_t operator()(int &dev_out, F &&set) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        dev_out = dev & 63;
        std::lock_guard<std::mutex> lock(mu);
        if (!done[dev_out]) {
            e = set();
            if (e != cudaSuccess) return e;
            if (cudaDeviceGetAttribute(&sms[dev_out], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) sms[dev_out] = 148;
            done[dev_out] = true;
        }
        return cudaSuccess;
    }
};

template <int VPL>
cudaError_t launch_warp_path(const WindowArgs &a, int use_bulk, cudaStream_t st) {
    const size_t smem = 2 * (size_t)a.n * kWarpPitch * 4;
    static AttrOnce once;
    int dev = 0;
    cudaError_t e = once(dev, [] {
        return cudaFuncSetAttribute(window_warp_kernel<VPL>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * 32 * VPL * kWarpPitch * 4);
    });
    if (e != cudaSuccess) return e;
    const int sms = once.sms[dev];
    const int ntiles = (a.series + kWarpTileCols - 1) / kWarpTileCols;
    const int grid = ntiles < 2 * sms ? ntiles : 2 * sms;
    return launch_after_smem(window_warp_kernel<VPL>, grid, 1024, smem, st, a, ntiles, use_bulk);
}

// ---------------------------------------------------------------------------------------
// Thread path: from the second evaluation on, a series' smoothed median and a tuned half-width
// h give an interval [centre - h, centre + h] that almost always holds the new middle
// elements, so that counting the values below the interval and selecting among the few dozen
// inside it replaces sorting the window.  One thread per series reads its window
// straight from the ring (a warp reads 32 adjacent series of a row: one fully used 128-byte
// line per load, eight rows in flight per thread), counts the values below the interval and
// keeps those inside it in its own shared-memory column.  No thread ever waits
// for another one: there is no barrier in the kernel, CTAs are four warps, and with 60 kept
// slots per thread seven CTAs share an SM.  The interval is centred on a smoothed median (a
// single window's median carries its own sampling noise, which would add to the next one's).
//
// Selection among the kept values runs the same instruction stream in every lane (thselect.cuh):
// counting passes over the column (128-bit shared-memory accesses; a column is 60 words, 4 x an
// odd number, so the lanes' quads fall on different banks) with a pivot interpolated between the
// ends of a shrinking bracket, every third pass a bisection, run until t - 1, t or t + 1 values
// lie below the pivot: the two largest below it and the two smallest not below it then include
// ranks t - 1 and t.  If the bracket shrinks to one value, that value holds both ranks (ties).
// A series whose interval missed, overflowed, did not converge or ended on a zero goes on a list;
// the kernel behind this one gives each listed series a warp (window_finish_kernel).
// ---------------------------------------------------------------------------------------
constexpr int kThCols = 128;     // series per CTA = threads per CTA
constexpr int kThSlots = 60;     // kept keys per series
constexpr int kThTarget = 42;    // number of keys the interval is tuned to catch (windows that share few steps)
constexpr int kThRows = 8;       // rows in flight per thread
constexpr int kThMaxPasses = 12;
constexpr float kThSmooth = 0.3f;   // weight of the newest median in the interval's centre
// Part of the way the half-width goes towards the one that would have caught kThTarget: little while the count is
// within its noise (a third), so that it does not follow it (2.1 % of 131 072 series unserved with a half in any case,
// 1.6 % so), half of the way beyond (a small part in any case: slow to settle, 3 % unserved instead of 0.8 % at 24 000 x 8).
constexpr float kThNear = 0.33f, kThNearPart = 0.15f, kThFarPart = 0.5f;

template <int VPL>
__global__ void __launch_bounds__(kThCols, 9) window_thread_kernel(const WindowArgs a) {
    pdl_wait();
    extern __shared__ __align__(16) uint32_t tkept[];   // [kThCols][kThSlots]
    const int tid = threadIdx.x, lane = lane_id();
    const int n = a.n;
    const int c = blockIdx.x * kThCols + tid;
    const bool active = c < a.series;
    const int cc = active ? c : a.series - 1;           // idle lanes of the last CTA read a valid column
    const int first = a.last_slot - (n - 1) + (a.last_slot < n - 1 ? a.capacity : 0);
    const int n1 = min(n, a.capacity - first);          // rows before the ring wraps

    const float hint = a.centre[cc], h = a.spread[cc];
    const bool usable = active && th_usable(hint, h);
    const ThRange range = th_range(hint, h, usable);

    const uint32_t kbase = smem_u32(tkept + tid * kThSlots), klim = kbase + (uint32_t)(kThSlots * 4);
    uint32_t kaddr = kbase;
    float cltf = 0.0f;
    auto stream = [&](const float *__restrict__ p, const int rows) {
        int r = 0;
        for (; r + kThRows <= rows; r += kThRows) {
            float x[kThRows];
#pragma unroll
            for (int u = 0; u < kThRows; ++u) x[u] = __ldg(p + (size_t)(r + u) * a.row_stride);
#pragma unroll
            for (int u = 0; u < kThRows; ++u) th_cell(x[u], range, klim, cltf, kaddr);
        }
        for (; r < rows; ++r) th_cell(__ldg(p + (size_t)r * a.row_stride), range, klim, cltf, kaddr);
    };
    stream(a.ring + (size_t)first * a.row_stride + cc, n1);
    stream(a.ring + cc, n - n1);

    const bool even = !(n & 1);
    const int k1 = (n - 1) >> 1, k2 = n >> 1;
    const int nk = (int)((kaddr - kbase) >> 2);
    const int clt = (int)cltf;
    bool ok = usable && clt <= k1 && k2 < clt + nk && nk <= kThSlots;
    // ---- selection among the kept values: the same instruction stream in every lane -------------
    float vb = 0.0f, vu = 0.0f, med = 0.0f;
    th_select_pair<kThSlots, kThMaxPasses>(kbase, nk, ok, k2 - clt, range, vb, vu);   // (k2 - clt >= 1 when n is even)
    if (ok) med = even ? __fmul_rn(0.5f, __fadd_rn(vb, vu)) : vu;
    if (active && ok) {
        a.wmed[c] = med;
        // re-tune the half-width so that the interval catches about kThTarget keys next time
        const float target = (float)(a.target > 0 ? a.target : kThTarget);
        const float f = fminf(2.0f, fmaxf(0.5f, target / (float)max(nk, 1)));
        const float part = fabsf((float)nk - target) > kThNear * target ? kThFarPart : kThNearPart;
        a.spread[c] = h * (1.0f - part + part * f);
        a.centre[c] = hint + (a.smooth > 0.0f ? a.smooth : kThSmooth) * (med - hint);
    }
    // ---- series the interval did not serve go on the launch's list (window_finish_kernel follows) ------
    // why (diagnostic): 0 no usable interval, 1 more keys than slots, 2 median below the interval,
    // 3 above it, 4 selection did not converge
    const int why = !usable ? 0 : (nk > kThSlots ? 1 : (clt > k1 ? 2 : (k2 >= clt + nk ? 3 : 4)));
    const unsigned todo = __ballot_sync(0xFFFFFFFFu, active && !ok);
    if (todo) {
        uint32_t base = 0;
        if (lane == 0) base = atomicAdd(a.fb_list_count, (uint32_t)__popc(todo));
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        if ((todo >> lane) & 1u) a.fb_list[base + __popc(todo & ((1u << lane) - 1u))] = ((uint32_t)why << 28) | (uint32_t)c;
    }
}

// The series the thread path's interval did not serve (a few per thousand), one warp per listed series: the lanes
// fetch the window, sort their own keys and run the warp selection.  A kernel of its own, so that these series spread
// over the GPU instead of queueing behind one another at the end of the warp that found them.
// The interval starts afresh at the median.  One that the median left by less than its width was not too narrow for the
// noise, but a little: it keeps a quarter more than its width, where a width from the window's deviations would be as far
// off as the first one was (passes of 24 000 ranks x 8 x 100 in blocks of 50 166.2 us, 170.0 afresh, 167.0 with the width as
// it was; 16 384 x 8 x 200 251.9 in blocks of 100, 260.2, 257.2; windows of up to 64 steps, of noisier medians, 160.8 and
// 158.8 afresh).  Bound by the loads' cache lines, one for each step of a listed series, and the chain of the selection: all
// of 131 072 series of 200 steps 180 us.  (Looking for a median just outside of its interval among the values of the
// neighbouring stretch first: the same beside other kernels, and 8 % more where all series are listed.)
constexpr int kFinThreads = 128;
constexpr int kFinCtas = 148 * 4;
constexpr float kFinNear = 3.0f, kFinWiden = 1.25f;

template <int VPL>
__global__ void __launch_bounds__(kFinThreads) window_finish_kernel(const WindowArgs a) {
    pdl_wait();
    __shared__ int is_last;
    const int lane = lane_id();
    const int n = a.n;
    const int first = a.last_slot - (n - 1) + (a.last_slot < n - 1 ? a.capacity : 0);
    const uint32_t count = min(__ldcg(a.fb_list_count), (uint32_t)a.series);
    const uint32_t nwarps = gridDim.x * (kFinThreads / 32);
    for (uint32_t i = blockIdx.x * (kFinThreads / 32) + warp_id(); i < count; i += nwarps) {
        const uint32_t item = __ldcg(a.fb_list + i);
        const int series = (int)(item & 0x0FFFFFFFu), why_src = (int)(item >> 28);
        float h = -1.0f, c = 0.0f;                         // (in flight with the window)
        if (VPL > 2 && (why_src == 2 || why_src == 3)) {   // below or above the interval
            h = __ldcg(a.spread + series);
            c = __ldcg(a.centre + series);
        }
        uint32_t kv[VPL];
        int nreal = 0;
#pragma unroll
        for (int j = 0; j < VPL; ++j) {
            const int row = lane + 32 * j;
            kv[j] = 0xFFFFFFFFu;
            if (row < n) {
                int slot = first + row;
                if (slot >= a.capacity) slot -= a.capacity;
                kv[j] = f2key(__ldg(a.ring + (size_t)slot * a.row_stride + series));
                ++nreal;
            }
        }
        lane_sort<VPL>(kv);
        float med = 0.0f;
        const bool ok2 = warp_median<VPL>(kv, nreal, n, 0u, med);
        float spread = warp_spread_guess<VPL>(kv, n, med);
        if (fabsf(med - c) <= kFinNear * h) spread = kFinWiden * h;
        if (lane == 0) {
            if (!ok2) atomicOr(a.status, kStatInternal);
            a.wmed[series] = med;
            a.spread[series] = spread;
            a.centre[series] = med;
            if (a.fb_count) { atomicAdd(a.fb_count, 1u); atomicAdd(a.fb_count + 1 + why_src, 1u); }
        }
    }
    // the CTA that finishes last clears the list for the next launch
    __syncthreads();
    if (threadIdx.x == 0) is_last = (atomicAdd(a.fb_list_count + 1, 1u) == gridDim.x - 1u) ? 1 : 0;
    __syncthreads();
    if (is_last && threadIdx.x == 0) {
        a.fb_list_count[0] = 0u;
        a.fb_list_count[1] = 0u;
    }
}

template <int VPL>
cudaError_t launch_thread_path(const WindowArgs &a, cudaStream_t st) {
    const size_t smem = (size_t)kThSlots * kThCols * 4;
    static AttrOnce once;
    int dev = 0;
    cudaError_t e = once(dev, [] {
        cudaError_t e2 = cudaFuncSetAttribute(window_thread_kernel<VPL>, cudaFuncAttributeMaxDynamicSharedMemorySize, kThSlots * kThCols * 4);
        if (e2 == cudaSuccess)
            e2 = cudaFuncSetAttribute(window_thread_kernel<VPL>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        return e2;
    });
    if (e != cudaSuccess) return e;
    e = launch_after_smem(window_thread_kernel<VPL>, (a.series + kThCols - 1) / kThCols, kThCols, smem, st, a);
    if (e != cudaSuccess) return e;
    const int fgrid = min(kFinCtas, (a.series + kFinThreads / 32 - 1) / (kFinThreads / 32));
    return launch_after(window_finish_kernel<VPL>, fgrid, kFinThreads, st, a);
}

// ---------------------------------------------------------------------------------------
// Sliding-window path: evaluations that follow one another by a few steps (streaming: one step)
// share all but a few steps of their windows, so a series' median moves by a rank or two.  Each
// series keeps, across evaluations, an interval [lo, hi] around its median, the number of window
// values below lo, and the handful of values inside the interval (global memory, each series' sorted
// list contiguous).  An evaluation reads only the steps that entered and left the window, one thread
// per series: a value below lo moves the count; a value inside the interval is inserted into /
// removed from the series' list by eight lanes, four series of the warp at a time; the median is then
// position (middle - count) of the list.
// A series whose median has left its interval, whose list is full, or that has no state yet is
// rebuilt from its whole window by a warp of the same CTA.  Exact either way: the interval only decides which values are
// listed.  The CTA's four warps share its rebuilds (of 128 series of continuous values one CTA in two has one): queued inside
// the warp that found them they make the kernel as slow as its unluckiest warp, and a kernel of their own costs the next
// step's update a launch and a scan of lists (an eighth of a single step of 2 048 ranks x 8, with node verdicts).
// ---------------------------------------------------------------------------------------
constexpr int kIncThreads = 128;
constexpr int kIncLanes = 8, kIncPer = kIncSlots / kIncLanes;   // lanes that hold a list, and slots per lane
static_assert(kIncPer * kIncLanes == kIncSlots, "a list is spread evenly");
constexpr int kIncNone = INT_MAX;   // above the keys of all numbers

// Signed integers in the total order of the floats, and back.
__device__ __forceinline__ int inc_key(const float x) { const int b = __float_as_int(x); return b ^ ((b >> 31) & 0x7FFFFFFF); }
__device__ __forceinline__ float inc_float(const int k) { return __int_as_float(k ^ ((k >> 31) & 0x7FFFFFFF)); }

// Median and state of a series from P sorted values per lane (element e in lane e / P, register e % P; m of them): those of
// ranks `base` and on of its window.
template <int P>
__device__ __forceinline__ void inc_store(const WindowArgs &a, const IncArgs &s, const int series, const uint32_t (&kv)[P], const int m, const int base) {
    const int lane = lane_id(), n = a.n;
    const bool even = !(n & 1);
    const int k1 = (n - 1) >> 1, k2 = n >> 1;
    auto pick = [&](int r) -> uint32_t {
        r -= base;
        uint32_t mine = kv[0];
#pragma unroll
        for (int j = 1; j < P; ++j) mine = ((r % P) == j) ? kv[j] : mine;
        return __shfl_sync(0xFFFFFFFFu, mine, r / P);
    };
    const float med = median_from_keys(pick(k1), pick(k2), even);
    const float flo = key2f(pick(max(0, k1 - kIncHalf))), fhi = key2f(pick(min(n - 1, k2 + kIncHalf)));
    // values below / inside the interval, by the same float comparisons the sliding update uses
    int below = 0, in = 0;
#pragma unroll
    for (int j = 0; j < P; ++j) {
        const bool real = lane * P + j < m;
        const float x = key2f(kv[j]);
        below += real && (x < flo);
        in += real && !(x < flo) && (x <= fhi);
    }
    int incl = in;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int u = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= d) incl += u;
    }
    const int nin = __shfl_sync(0xFFFFFFFFu, incl, 31);
    const int cb = base + (int)__reduce_add_sync(0xFFFFFFFFu, (uint32_t)below);
    const bool fits = nin <= kIncSlots;
    if (fits) {
        int pos = incl - in;
#pragma unroll
        for (int j = 0; j < P; ++j) {
            const bool real = lane * P + j < m;
            const float x = key2f(kv[j]);
            if (real && !(x < flo) && (x <= fhi)) { s.val[(size_t)series * kIncSlots + pos] = x; ++pos; }
        }
    }
    if (lane == 0) {
        a.wmed[series] = med;
        s.lo[series] = flo;
        s.hi[series] = fhi;
        // an interval with more (tied) values than a list holds stays without state: it rebuilds every time
        s.cnt[series] = fits ? (0x80000000u | ((uint32_t)nin << 16) | (uint32_t)cb) : 0u;
        if (s.rebuilds) atomicAdd(s.rebuilds, 1u);
    }
}

// The state of one series from its whole window, by a warp: the lanes fetch the window and sort it (bitonic network over
// registers and shuffles) for the median, the interval ends kIncHalf ranks beyond the middle ranks, and the values inside.
// A median that has left its interval has not gone far: where the values within a width of the interval hold all of these
// ranks (counted), only they are sorted, two per lane (`list`: room for 64 of them).
template <int VPL>
__device__ __forceinline__ void inc_rebuild(const WindowArgs &a, const IncArgs &s, const int series, const int first, float *list) {
    const int lane = lane_id(), n = a.n;
    float x[VPL];
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
        const int row = lane + 32 * j;
        x[j] = 0.0f;
        if (row < n) {
            int slot = first + row;
            if (slot >= a.capacity) slot -= a.capacity;
            x[j] = __ldg(a.ring + (size_t)slot * a.row_stride + series);
        }
    }
    if (VPL > 2 && !s.rebuild_all && (s.cnt[series] >> 31)) {
        const float l0 = s.lo[series], h0 = s.hi[series], d = h0 - l0, lo = l0 - d, hi = h0 + d;
        int below = 0, kept = 0;
#pragma unroll
        for (int j = 0; j < VPL; ++j) {
            const bool real = lane + 32 * j < n;
            below += real && x[j] < lo;
            const bool in = real && x[j] >= lo && x[j] <= hi;
            const uint32_t who = __ballot_sync(0xFFFFFFFFu, in);
            const int at = kept + __popc(who & ((1u << lane) - 1u));
            if (in && at < 64) list[at] = x[j];
            kept += __popc(who);
        }
        const int base = (int)__reduce_add_sync(0xFFFFFFFFu, (uint32_t)below);
        const int r0 = max(0, ((n - 1) >> 1) - kIncHalf), r1 = min(n - 1, (n >> 1) + kIncHalf);
        if (kept <= 64 && base <= r0 && r1 < base + kept) {   // (the same for the whole warp)
            __syncwarp();
            uint32_t kv[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) kv[j] = 2 * lane + j < kept ? f2key(list[2 * lane + j]) : 0xFFFFFFFFu;
            warp_bitonic_sort<2>(kv, lane);
            inc_store<2>(a, s, series, kv, kept, base);
            __syncwarp();
            return;
        }
        __syncwarp();
    }
    uint32_t kv[VPL];
#pragma unroll
    for (int j = 0; j < VPL; ++j) kv[j] = lane + 32 * j < n ? f2key(x[j]) : 0xFFFFFFFFu;   // padding sorts behind every finite value
    warp_bitonic_sort<VPL>(kv, lane);
    inc_store<VPL>(a, s, series, kv, n, 0);
}

// A series whose list is edited: what eight lanes need of it.
template <int NEW>
struct IncEdit {
    int c, cb, nin;
    uint32_t in_l, in_e;         // which of the steps lie inside the interval
    float xl[NEW], xe[NEW];
};

// NEW: the most steps that entered / left (1 for an evaluation after every step, else kIncMaxNew); VPL: values per lane of
// a rebuild.  (Two series per thread, all of 262 144 resident at once: the same alone, and beside the cluster kernels of
// other evaluations, which then wait for room, six deferred steps of 32 768 x 8 take 6 % longer.)
template <int NEW, int VPL>
__global__ void __launch_bounds__(kIncThreads, 8) window_inc_kernel(const WindowArgs a, const IncArgs s, const int per) {
    pdl_wait();
    __shared__ float sh_list[kIncThreads / 32][32 / kIncLanes][kIncSlots];   // per warp: the edited lists
    __shared__ IncEdit<NEW> sh_edit[kIncThreads / 32][32];                   // ... and what is edited
    __shared__ uint32_t rb_n, rb_list[kIncThreads];                          // series of this CTA to rebuild
    if (threadIdx.x == 0) rb_n = 0u;
    __syncthreads();
    const int lane = lane_id(), wid = warp_id();
    const int n = a.n;
    const int first = a.last_slot - (n - 1) + (a.last_slot < n - 1 ? a.capacity : 0);   // slot of the window's oldest step
    const bool even = !(n & 1);
    const int k1 = (n - 1) >> 1, k2 = n >> 1;
    const int c = blockIdx.x * per + threadIdx.x;        // (the other threads take part in the rebuilds)
    const bool mine = (int)threadIdx.x < per && c < a.series;

    // The steps that left the window (the ones right before its oldest step) and the steps that entered it (the
    // newest ones), all fetched up front.
    const uint32_t w = mine ? s.cnt[c] : 0u;
    const float lo = mine ? s.lo[c] : 0.0f, hi = mine ? s.hi[c] : 0.0f;
    float xl[NEW], xe[NEW];
#pragma unroll
    for (int i = 0; i < NEW; ++i) {
        xl[i] = 0.0f;
        xe[i] = 0.0f;
        if (mine && i < s.leaving) {
            int slot = first - s.leaving + i;
            if (slot < 0) slot += a.capacity;
            xl[i] = __ldg(a.ring + (size_t)slot * a.row_stride + c);
        }
        if (mine && i < s.entering) {
            int slot = a.last_slot - (s.entering - 1 - i);
            if (slot < 0) slot += a.capacity;
            xe[i] = __ldg(a.ring + (size_t)slot * a.row_stride + c);
        }
    }
    // A value below lo moves the count; a value inside the interval changes the series' sorted list, which eight lanes
    // then edit (below).  A list that stays as it is has the middle ranks of the window at positions k1 - cb and k2 - cb.
    const bool ok = mine && (w >> 31) && !s.rebuild_all;
    int cb = (int)(w & 0xFFFFu);
    const int nin = (int)((w >> 16) & 0xFFu);
    uint32_t in_l = 0, in_e = 0;
#pragma unroll
    for (int i = 0; i < NEW; ++i) {
        if (i < s.leaving) {
            if (xl[i] < lo) --cb;
            else if (xl[i] <= hi) in_l |= 1u << i;
        }
        if (i < s.entering) {
            if (xe[i] < lo) ++cb;
            else if (xe[i] <= hi) in_e |= 1u << i;
        }
    }
    const bool edits = ok && (in_l | in_e) != 0u;
    const bool plain = ok && !edits && cb >= 0 && cb <= k1 && k2 < cb + nin;
    float f1 = 0.0f, f2 = 0.0f;
    uint32_t cnt = 0;
    if (plain) {
        f1 = s.val[(size_t)c * kIncSlots + (k1 - cb)];
        f2 = s.val[(size_t)c * kIncSlots + (k2 - cb)];
        cnt = 0x80000000u | ((uint32_t)nin << 16) | (uint32_t)cb;
    }
    const unsigned upd = __ballot_sync(0xFFFFFFFFu, edits);
    if (edits) {
        IncEdit<NEW> &e = sh_edit[wid][__popc(upd & ((1u << lane) - 1u))];
        e.c = c;
        e.cb = cb;
        e.nin = nin;
        e.in_l = in_l;
        e.in_e = in_e;
#pragma unroll
        for (int i = 0; i < NEW; ++i) { e.xl[i] = xl[i]; e.xe[i] = xe[i]; }
    }
    const int nedit = __popc(upd);
    if (mine && !plain && !edits) rb_list[atomicAdd(&rb_n, 1u)] = (uint32_t)c;
    __syncwarp();
    // ---- list updates, four series at a time: eight lanes hold a list, kIncPer neighbouring slots each ----
    const int grp = lane / kIncLanes, gl = lane % kIncLanes;
    float ahead[kIncPer];
    auto fetch = [&](const int i) {              // (the next lists are on their way while these are edited)
        if (i < nedit) {
            const float *list = s.val + (size_t)sh_edit[wid][i].c * kIncSlots + gl * kIncPer;
            const int ns = sh_edit[wid][i].nin;
#pragma unroll
            for (int j = 0; j < kIncPer; ++j)
                if (gl * kIncPer + j < ns) ahead[j] = list[j];
        }
    };
    fetch(grp);
    for (int i0 = 0; i0 < nedit; i0 += 32 / kIncLanes) {
        const bool act = i0 + grp < nedit;
        const IncEdit<NEW> &e = sh_edit[wid][act ? i0 + grp : 0];
        int ns = act ? e.nin : 0;
        const int ce = e.c, cbe = e.cb;
        const uint32_t ml = act ? e.in_l : 0u, me = act ? e.in_e : 0u;
        int old[kIncPer], v[kIncPer];            // slots without a value lie above everything
#pragma unroll
        for (int j = 0; j < kIncPer; ++j) old[j] = v[j] = gl * kIncPer + j < ns ? inc_key(ahead[j]) : kIncNone;
        fetch(i0 + 32 / kIncLanes + grp);
        bool good = act;
#pragma unroll
        for (int i = 0; i < NEW; ++i) {
            const bool here = (ml >> i) & 1u;
            if (!__any_sync(0xFFFFFFFFu, here)) continue;
            const int kx = here ? inc_key(e.xl[i]) : kIncNone;
            // values from the first one not below x on move down by one; that one has to be x
            int next = __shfl_down_sync(0xFFFFFFFFu, v[0], 1, kIncLanes);
            if (gl == kIncLanes - 1) next = kIncNone;
            bool found = false;
#pragma unroll
            for (int j = 0; j < kIncPer; ++j) {
                found |= v[j] == kx;
                v[j] = v[j] < kx ? v[j] : (j + 1 < kIncPer ? v[j + 1] : next);
            }
            const uint32_t hit = (__ballot_sync(0xFFFFFFFFu, found) >> (grp * kIncLanes)) & ((1u << kIncLanes) - 1u);
            if (here) { good = good && hit != 0u; --ns; }   // (else the books do not balance: rebuild)
        }
#pragma unroll
        for (int i = 0; i < NEW; ++i) {
            const bool here = (me >> i) & 1u;
            if (!__any_sync(0xFFFFFFFFu, here)) continue;
            const int kx = here ? inc_key(e.xe[i]) : kIncNone;
            int prev = __shfl_up_sync(0xFFFFFFFFu, v[kIncPer - 1], 1, kIncLanes);
            if (gl == 0) prev = INT_MIN;
#pragma unroll
            for (int j = kIncPer - 1; j >= 0; --j) v[j] = max(j ? v[j - 1] : prev, min(v[j], kx));
            if (here) { good = good && ns < kIncSlots; ++ns; }
        }
        good = good && cbe >= 0 && cbe <= k1 && k2 < cbe + ns;
        float *list = s.val + (size_t)ce * kIncSlots + gl * kIncPer;
#pragma unroll
        for (int j = 0; j < kIncPer; ++j) {
            const int slot = gl * kIncPer + j;
            sh_list[wid][grp][slot] = inc_float(v[j]);
            if (good && slot < ns && v[j] != old[j]) list[j] = inc_float(v[j]);
        }
        __syncwarp();
        if (gl == 0 && act) {
            if (good) {
                a.wmed[ce] = median_from_keys(f2key(sh_list[wid][grp][k1 - cbe]), f2key(sh_list[wid][grp][k2 - cbe]), even);
                s.cnt[ce] = 0x80000000u | ((uint32_t)ns << 16) | (uint32_t)cbe;
            } else {
                rb_list[atomicAdd(&rb_n, 1u)] = (uint32_t)ce;
            }
        }
        __syncwarp();
    }
    if (plain) {
        a.wmed[c] = median_from_keys(f2key(f1), f2key(f2), even);
        s.cnt[c] = cnt;
    }
    // ---- series without a usable state: the CTA's warps share them ----
    __syncthreads();
    const uint32_t count = rb_n;
    for (uint32_t i = (uint32_t)wid; i < count; i += kIncThreads / 32) inc_rebuild<VPL>(a, s, (int)rb_list[i], first, &sh_list[wid][0][0]);
}

}  // namespace

// Which whole-window path an evaluation takes.  Many series of a short window with an earlier result: one thread per
// series (21 + 5 us at 131 072 series of 100 steps, 36 + 10 at 200, against 56 and 86 with a tile per 32 series).  Up to
// 65 536 series the threads are too few to hide their own latency, and a launch less counts (8 192 series of
// 100 / 200 steps: 14 + 5 / 21 + 8 us against 11 / 16; 32 768: 16 + 5 / 24 + 8 against 14 / 25).  First evaluations:
// a warp per series while there are few (9.2 us against 12 at 8 192 series of 100 steps; at 32 768 series 28 against
// 18, at 131 072 series of 200 steps 196 against 101).
enum WindowPath { kPathThread, kPathWarp, kPathBins };
static WindowPath window_path(const WindowArgs &a) {
    if (a.n > 256) return kPathBins;
    if (!a.use_hint) return a.series <= 16384 ? kPathWarp : kPathBins;
    return a.series > 65536 && a.spread && a.centre && a.fb_list && a.series < (1 << 28) ? kPathThread : kPathBins;
}

int window_launch_count(const WindowArgs &a) { return window_path(a) == kPathThread ? 2 : 1; }

size_t window_inc_bytes(int series) { return (size_t)series * sizeof(float); }

bool window_inc_supported(const WindowArgs &a) { return a.n >= 1 && a.n <= 256; }

// Series of a CTA of the sliding update: its warps share its rebuilds, so that few series to a CTA spread the rebuilds over
// the whole chip.  Where many series keep no list (constant or coarse values) or all leave theirs at a time (a common shift of
// level), 128 series to a CTA take an evaluation of 64 ranks x 4 x 50 steps from 17.9 us to 73.3 (all series constant), of
// 2 048 x 8 x 200 from 41.3 to 69.9 and of 8 192 x 8 x 200 from 95.5 to 133.4 (two metrics of eight constant).  1 024 CTAs at
// most: the more there are, the fewer find room beside the cross-rank clusters (continuous values of 8 192 x 8 x 200 33.7 us,
// with 128 series to a CTA 33.4, with the 1 184 CTAs that an idle chip holds 34.1 and, of constant ones, 87).
static int inc_series_per_cta(const int series) {
    constexpr int kMost = 1024;
    return min(kIncThreads, max(8, ((series + kMost - 1) / kMost + 7) & ~7));
}

template <int VPL>
static cudaError_t launch_inc(const WindowArgs &a, const IncArgs &inc, cudaStream_t st) {
    const int per = inc_series_per_cta(a.series), grid = (a.series + per - 1) / per;
    return inc.entering <= 1 && inc.leaving <= 1 ? launch_after(window_inc_kernel<1, VPL>, grid, kIncThreads, st, a, inc, per)
                                                 : launch_after(window_inc_kernel<kIncMaxNew, VPL>, grid, kIncThreads, st, a, inc, per);
}

cudaError_t launch_window_incremental(const WindowArgs &a, const IncArgs &inc, cudaStream_t st) {
    if (a.n <= 64) return launch_inc<2>(a, inc, st);
    if (a.n <= 128) return launch_inc<4>(a, inc, st);
    return launch_inc<8>(a, inc, st);
}

cudaError_t launch_window_select(const WindowArgs &a, cudaStream_t st) {
    const WindowPath path = window_path(a);
    if (path == kPathThread) {
        if (a.n <= 64) return launch_thread_path<2>(a, st);
        if (a.n <= 128) return launch_thread_path<4>(a, st);
        return launch_thread_path<8>(a, st);
    }
    if (path == kPathBins) {
        WindowArgs b = a;
        // the thread path takes over from the next evaluation on: its interval has fewer slots
        b.target = a.n <= 256 && a.series > 65536 ? kThTarget : 0;
        return launch_window_bins(b, st);
    }
    // bulk copies need 16-byte aligned sources and sizes
    const int use_bulk = (a.series % 4 == 0) && (((uintptr_t)a.ring & 15) == 0);
    if (a.n <= 64) return launch_warp_path<2>(a, use_bulk, st);
    if (a.n <= 128) return launch_warp_path<4>(a, use_bulk, st);
    return launch_warp_path<8>(a, use_bulk, st);
}

}  // namespace guard
