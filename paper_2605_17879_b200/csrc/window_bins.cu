// Windowed medians, tile path: a CTA takes 32 adjacent series (lane = series) and splits the window's steps over its
// warps, the values in registers (windows of up to 1 024 steps) or read again in every pass (longer ones).
//   1. a value range that should hold the middle ranks: around the series' smoothed median where an earlier
//      evaluation left one, else between two of sixteen values of the window;
//   2. one pass bins all values (32 bins per series, the first and the last for what lies below and beyond the range; a
//      bin's counters of the 32 series are 32 adjacent words, so that the shared-memory reductions of a warp never meet in
//      a bank); one warp scans the bins for the middle ranks;
//   3. a second pass notes the values of those one or two bins, a few per thread, and they are ranked.
// The counts prove the range; one that misses is moved, and a bin with too many values becomes the next range
// (or the answer, if they are all the same), so any values come out exactly; what is still open after a few rounds
// is settled bit by bit.  A value's bin is the low mantissa bits of two chained multiply-adds, the first saturated to
// [0, 1]: monotone in x whatever the rounding, and both full rate (compares and integer adds run at half rate).
// Bound by instruction issue: some 900 instructions a warp for 24 to 28 values, a third of them not per value (the hits of
// its luckiest lane, ranking, barriers, its share of the scan).  What cost most before: three compares a value where the
// saturation does, a scan shared by all warps, selecting noted values from registers by their index (a chain over all of
// them per hit), and 20 to 236 bytes of spills; now none up to 28 values a thread.
// Measured, kernel alone: 98 760 first windows of 180 steps 45 us (68 with those), 65 536 of 100 steps with ties 22 (33),
// 65 536 of 120 beside the cross-rank kernel 19 (38), 8 192 of 1 000 steps 19 (24; half as many warps that read the
// window again 60), 8 192 of 100 8.5 (10.9).  131 072 of 200 steps 64 to 80 beside other kernels: a thread per series
// (window.cu) takes 7 instructions a value and one warp's selection for 32 series, 37 + 10.
#include <math_constants.h>

#include "binmap.cuh"
#include "kernels.h"

namespace guard {

namespace {

constexpr int kWbBins = 32;
constexpr int kWbSample = 16;
// Values of a bin that are ranked directly (sixteen to 32 of them take eight warps longer than another round)
__host__ __device__ constexpr int wb_list(const int G) { return G <= 8 ? 16 : 32; }
__host__ __device__ constexpr int wb_hits(const int G) { return G <= 8 ? 10 : 6; }   // wanted values that a thread notes (more than that: ties)
constexpr int kWbRounds = 6;       // rounds of ranges before the bit-by-bit selection
constexpr float kWbSmooth = 0.3f;  // weight of the newest median in the range's centre
constexpr float kWbMagic = 12582912.0f;   // 1.5 * 2^23: adding it leaves an integer in the low mantissa bits
constexpr float kWbMax = 3.402823466e+38f;

template <int G>
struct WbShared {
    __align__(16) uint32_t hist[kWbBins][32];
    float hit[G][wb_hits(G)][32];  // wanted values, by thread
    float f0[32], f1[32];          // values to fetch: those of bins f0 to f1
    uint32_t how[32];              // 0 nothing, 1 list and rank, 2 largest of bin f0 / smallest of bin f1, 3 smallest and largest
    uint32_t q1[32], nl[32], mx[32], mn[32], v1[32], v2[32];
    float lo[32], hi[32];          // the next range
    float width[32];               // of the first range its width, the values inside, and why it did not serve, if so
    uint32_t inside[32];           // (diagnostic): 1 too many values in a bin, 2 the median lies below it, 3 above it
    int why[32];
    uint32_t list[wb_list(G)][32];
    uint32_t prefix[32], krem[32], cnt[32];   // bit-by-bit selection
};

// A value's bin: t = fma(sat(fma(x, scale, off)), bins - 1, magic), bits of the first bin's t plus the bin.
// (Inside the assembly of each use: the compiler would otherwise keep the results of one pass for the next and spill.)
#define WB_T(x, scale, off) "fma.rn.sat.f32 t, " x ", " scale ", " off ";\n\tfma.rn.f32 t, t, 0f41F80000, 0f4B400000;\n\t"
static_assert(kWbBins == 32, "31.0f is part of WB_T");
// hist[bin] += 1
__device__ __forceinline__ void wb_bin(const float x, const float scale, const float off, const uint32_t base) {
    asm volatile(
        "{\n\t.reg .u32 a, b;\n\t.reg .f32 t;\n\t" WB_T("%0", "%1", "%2")
        "mov.b32 b, t;\n\t"
        "mad.lo.u32 a, b, 128, %3;\n\t"
        "red.shared.add.u32 [a], 1;\n\t}"
        :
        : "f"(x), "f"(scale), "f"(off), "r"(base)
        : "memory");
}
// if (f0 <= t <= f1) { if (addr < lim) shared[addr] = x; addr += 128; }
__device__ __forceinline__ void wb_note(const float x, const float scale, const float off, const float f0, const float f1, const uint32_t lim,
                                        uint32_t &addr) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .f32 t;\n\t" WB_T("%1", "%2", "%3")
        "setp.ge.f32 p, t, %4;\n\t"
        "setp.le.and.f32 p, t, %5, p;\n\t"
        "setp.lt.and.u32 q, %0, %6, p;\n\t"
        "@q st.shared.f32 [%0], %1;\n\t"
        "@p add.u32 %0, %0, 128;\n\t}"
        : "+r"(addr)
        : "f"(x), "f"(scale), "f"(off), "f"(f0), "f"(f1), "r"(lim)
        : "memory");
}
__device__ __forceinline__ float wb_t(const float x, const float scale, const float off) {
    float t;
    asm volatile("{\n\t.reg .f32 t;\n\t" WB_T("%1", "%2", "%3") "mov.f32 %0, t;\n\t}" : "=f"(t) : "f"(x), "f"(scale), "f"(off));
    return t;
}
// G warps of V values per thread; RELOAD: the window is longer than that, V values at a time are read again.
template <int V, int G, bool RELOAD>
__global__ void __launch_bounds__(32 * G, G <= 8 ? 4 : (G <= 16 ? 2 : 1)) window_bins_kernel(const WindowArgs a) {
    pdl_wait();
    constexpr int H = wb_hits(G), kWbList = wb_list(G);
    __shared__ WbShared<G> sh;
    const int lane = lane_id(), w = __shfl_sync(0xFFFFFFFFu, warp_id(), 0), n = a.n;   // (w in a uniform register: so are the rows' numbers)
    const int c = blockIdx.x * 32 + lane;
    const bool active = c < a.series;
    const int cc = active ? c : a.series - 1;
    const int first = a.last_slot - (n - 1) + (a.last_slot < n - 1 ? a.capacity : 0);
    const bool even = !(n & 1);
    const uint32_t k1 = (uint32_t)((n - 1) >> 1), k2 = (uint32_t)(n >> 1);
    const float *colp = a.ring + cc;
    auto load = [&](const int r) -> float {   // step r of the window; beyond its end the largest number (ranks are counted from below)
        int slot = first + r;
        if (slot >= a.capacity) slot -= a.capacity;
        return r < n ? __ldg(colp + (size_t)slot * a.row_stride) : kWbMax;
    };
    float x[V];
    if (!RELOAD) {
        if (first + n <= a.capacity) {       // (an addition per row)
            const float *q = colp + (size_t)(first + w) * a.row_stride;
            const size_t step = (size_t)G * a.row_stride;
#pragma unroll
            for (int i = 0; i < V; ++i, q += step) x[i] = w + i * G < n ? __ldg(q) : kWbMax;
        } else {
#pragma unroll
            for (int i = 0; i < V; ++i) x[i] = load(w + i * G);
        }
    }
    // f(), for each batch of V values of this thread (steps r0, r0 + G, ...)
    auto batches = [&](auto &&f) {
        if (!RELOAD) {
            f(w);
        } else {
#pragma unroll 1
            for (int r0 = w; r0 < n; r0 += V * G) {
#pragma unroll
                for (int i = 0; i < V; ++i) x[i] = load(r0 + i * G);
                f(r0);
            }
        }
    };
    float lo = 0.0f, hi = 0.0f;
    bool hinted = false;
    if (a.use_hint) {
        const float centre = a.centre[cc], spread = a.spread[cc];
        hinted = spread > 0.0f && spread < 1.0e37f && fabsf(centre) < 1.0e37f;
        lo = centre - spread;
        hi = centre + spread;
    }
    auto clear = [&] {
        for (int i = threadIdx.x; i < kWbBins * 8; i += 32 * G) reinterpret_cast<uint4 *>(&sh.hist[0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
    };
    clear();
    // series without an earlier result: from sixteen values of the window, each warp's share of them from its registers: its
    // first, and with eight warps one from the middle of its values.  (Values of long windows that are read again are spread over
    // the window; the sixteen oldest steps of a window of 257 to 1 024 say less about one that drifts: first evaluations of
    // 1 024 x 8 series of 1 000 steps that grow by half over the window take 50 us instead of 39.)  The second smallest of the
    // smaller ones of eight pairs and the second largest of the larger ones (of values without order one in a thousand medians
    // lies outside, and an outlier at either end does not stretch the range); of all sixteen where a warp has one; the ends of a
    // window too short for that.
    if (__any_sync(0xFFFFFFFFu, !hinted)) {   // (the same for every warp of the CTA)
        constexpr bool kPairs = G < kWbSample;
        constexpr int N = kPairs ? G : kWbSample;
        static_assert(!kPairs || 2 * G == kWbSample, "two values per warp");
        if (w < N) {
            auto at = [&](const int q) -> float {
                return RELOAD ? load((int)(((2 * (q * G + w) + 1) * (long long)n) / (2 * kWbSample))) : x[q * V / 2];
            };
            const float u = at(0), v = kPairs ? at(1) : u;
            const bool two = RELOAD || w + (V / 2) * G < n;   // (beyond the window: the largest number)
            sh.list[w][lane] = __float_as_uint(fminf(u, v));
            sh.hit[0][0][w * 32 + lane] = RELOAD || w < n ? (kPairs && two ? fmaxf(u, v) : u) : -kWbMax;
        }
        __syncthreads();
        float l1 = kWbMax, l2 = kWbMax, h1 = -kWbMax, h2 = -kWbMax;   // two smallest, two largest
#pragma unroll 4
        for (int i = 0; i < N; ++i) {
            const float u = __uint_as_float(sh.list[i][lane]), v = sh.hit[0][0][i * 32 + lane];
            l2 = fminf(l2, fmaxf(l1, u));
            l1 = fminf(l1, u);
            h2 = fmaxf(h2, fminf(h1, v));
            h1 = fmaxf(h1, v);
        }
        if (!hinted) { lo = n >= 3 * kWbSample ? l2 : l1; hi = n >= 3 * kWbSample ? h2 : h1; }
    }
    if (w == 0) { sh.width[lane] = hi - lo; sh.why[lane] = hinted ? -1 : 0; }
    constexpr float T0 = kWbMagic;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(&sh.hist[0][lane]) - (uint32_t)(0x4B400000ull * 128ull);   // bits of T0
    const uint32_t hit0 = (uint32_t)__cvta_generic_to_shared(&sh.hit[w][0][lane]);
    bool live = true;
    int round = 0;
#pragma unroll 1
    for (;; ++round) {
        // ---- bin: the range (a little wider: binmap.cuh) from the middle of the second bin to that of the last but one; the
        // first and the last take all values below and beyond ----
        const BinMap map = bin_map<kWbBins - 1>(lo, hi);
        float scale = map.scale, off = map.off;
        if (hi - lo > kWbMax) { scale = 0.0f; off = 0.5f; }   // (a range wider than the largest number: all values share a bin)
        if (!live) { scale = 0.0f; off = 0.0f; }              // (settled series count nothing that matters)
        __syncthreads();           // bins are zero
        if (round >= kWbRounds) break;
        batches([&](int) {
#pragma unroll
            for (int i = 0; i < V; ++i) wb_bin(x[i], scale, off, base);
        });
        __syncthreads();
        // ---- scan, by one warp: where the middle ranks lie ----
        if (w == 0) {
            uint32_t r = 0, start = 0, size = 0, b1 = 0, b2 = 0;
#pragma unroll 8
            for (uint32_t b = 0; b < kWbBins; ++b) {
                const uint32_t h = sh.hist[b][lane];
                if (r <= k1) { start = r; size = h; b1 = b; }
                if (r <= k2) b2 = b;
                r += h;
            }
            const bool served = live && b1 > 0u && b2 < kWbBins - 1;
            sh.f0[lane] = served ? T0 + (float)b1 : CUDART_INF_F;
            sh.f1[lane] = served ? T0 + (float)b2 : -CUDART_INF_F;
            sh.q1[lane] = k1 - start;
            sh.how[lane] = !served ? 0u : (b1 != b2 ? 2u : (size <= (uint32_t)kWbList ? 1u : 3u));
            sh.nl[lane] = 0u;
            sh.mx[lane] = 0u;
            sh.mn[lane] = 0xFFFFFFFFu;
            if (live && !served) {     // move or stretch the range: a little (a level that shifts or drifts), far, to everything
                const float wd = map.span, edge = 0.0625f * wd, step = round < 2 ? (round == 0 ? 4.0f : 64.0f) * wd + 1.0e-30f : kWbMax;
                float nlo = lo, nhi = hi;
                if (b1 == 0u) { nlo = fmaxf(lo - step, -kWbMax); if (b2 == 0u) nhi = lo + edge; }
                if (b2 == kWbBins - 1) { nhi = fminf(hi + step, kWbMax); if (b1 == kWbBins - 1) nlo = hi - edge; }
                sh.lo[lane] = nlo;
                sh.hi[lane] = nhi;
            }
            if (round == 0) {
                sh.inside[lane] = r - sh.hist[0][lane] - sh.hist[kWbBins - 1][lane];
                if (hinted && !served) sh.why[lane] = b1 == 0u ? 2 : 3;
            }
        }
        __syncthreads();
        // ---- fetch the values of those bins (a few) ----
        {
            const float f0 = sh.f0[lane], f1 = sh.f1[lane];
            batches([&](const int r0) {
                uint32_t addr = hit0;
#pragma unroll
                for (int i = 0; i < V; ++i) wb_note(x[i], scale, off, f0, f1, hit0 + 128u * H, addr);
                const int hits = (int)((addr - hit0) >> 7);
                if (hits) {
                    const uint32_t how = sh.how[lane];
                    uint32_t pos = 0, mx = 0u, mn = 0xFFFFFFFFu;
                    if (how == 1u) pos = atomicAdd(&sh.nl[lane], (uint32_t)hits);
                    auto take = [&](const float v) {
                        const uint32_t key = f2key(v);
                        if (how == 1u) {   // (the bin's count says that they fit)
                            sh.list[pos++][lane] = key;
                        } else {
                            const bool low = how == 3u || wb_t(v, scale, off) <= f0;
                            if (low) mx = max(mx, key);
                            if (how == 3u || !low) mn = min(mn, key);
                        }
                    };
                    if (hits <= H) {
                        for (int i = 0; i < hits; ++i) take(sh.hit[w][i][lane]);
                    } else {       // (read again: the registers cannot be indexed)
#pragma unroll 1
                        for (int i = 0; i < V; i += 4) {
                            float v[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) v[j] = load(r0 + (i + j) * G);
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const float t = wb_t(v[j], scale, off);
                                if (t >= f0 && t <= f1) take(v[j]);
                            }
                        }
                    }
                    if (how >= 2u) {
                        if (mx != 0u) atomicMax(&sh.mx[lane], mx);
                        if (mn != 0xFFFFFFFFu) atomicMin(&sh.mn[lane], mn);
                    }
                }
            });
        }
        __syncthreads();
        // ---- settle ----
        const uint32_t how = sh.how[lane];
        if (how == 1u) {
            const uint32_t m = min(sh.nl[lane], (uint32_t)kWbList), q1 = sh.q1[lane], q2 = even ? q1 + 1u : q1;
            for (uint32_t j = (uint32_t)w; j < m; j += (uint32_t)G) {
                const uint32_t mk = sh.list[j][lane];
                uint32_t lt = 0, le = 0;
#pragma unroll 4
                for (uint32_t i = 0; i < m; ++i) {
                    const uint32_t o = sh.list[i][lane];
                    lt += o < mk;
                    le += o <= mk;
                }
                if (q1 >= lt && q1 < le) sh.v1[lane] = mk;
                if (q2 >= lt && q2 < le) sh.v2[lane] = mk;
            }
        } else if (how >= 2u && w == 0) {
            const uint32_t mx = sh.mx[lane], mn = sh.mn[lane];
            if (how == 2u || mx == mn) {
                sh.v1[lane] = mx;
                sh.v2[lane] = mn;
            } else {               // a full bin of different values becomes the range
                sh.lo[lane] = key2f(mn);
                sh.hi[lane] = key2f(mx);
                if (round == 0 && hinted) sh.why[lane] = 1;
            }
        }
        const bool settled = !live || how == 1u || how == 2u || (how == 3u && sh.mx[lane] == sh.mn[lane]);
        const uint32_t still = __ballot_sync(0xFFFFFFFFu, !settled);   // (the same for every warp of the CTA)
        live = live && !settled;
        if (still == 0u) break;
        __syncthreads();           // ranges and results are written
        if (live) { lo = sh.lo[lane]; hi = sh.hi[lane]; }
        clear();
    }
    if (round >= kWbRounds) {      // denormal ranges and the like: one key bit after the other, the values read again
        if (w == 0) { sh.prefix[lane] = 0u; sh.krem[lane] = k1; sh.cnt[lane] = 0u; sh.mn[lane] = 0xFFFFFFFFu; sh.nl[lane] = 0u; }
        __syncthreads();
#pragma unroll 1
        for (int bit = 31; bit >= 0; --bit) {
            const uint32_t prefix = sh.prefix[lane];
            uint32_t zeros = 0;
#pragma unroll 4
            for (int r = w; r < n; r += G) {
                const uint32_t key = f2key(load(r));
                const bool match = bit == 31 || ((key ^ prefix) >> (bit + 1)) == 0u;
                zeros += match && !((key >> bit) & 1u);
            }
            atomicAdd(&sh.cnt[lane], zeros);
            __syncthreads();
            if (w == 0) {
                const uint32_t z = sh.cnt[lane], k = sh.krem[lane];
                if (k >= z) { sh.prefix[lane] |= 1u << bit; sh.krem[lane] = k - z; }
                sh.cnt[lane] = 0u;
            }
            __syncthreads();
        }
        const uint32_t key1 = sh.prefix[lane];
        uint32_t le = 0, above = 0xFFFFFFFFu;
#pragma unroll 4
        for (int r = w; r < n; r += G) {
            const uint32_t key = f2key(load(r));
            le += key <= key1;
            if (key > key1) above = min(above, key);
        }
        atomicAdd(&sh.nl[lane], le);
        atomicMin(&sh.mn[lane], above);
        __syncthreads();
        if (w == 0 && live) {
            sh.v1[lane] = key1;
            sh.v2[lane] = sh.nl[lane] > k2 ? key1 : sh.mn[lane];
        }
    }
    __syncthreads();
    if (w == 0 && active) {
        const uint32_t v1 = sh.v1[lane], v2 = sh.v2[lane];
        const float med = median_from_keys(even ? v1 : v2, v2, even);
        a.wmed[c] = med;
        if (a.spread && a.centre) {
            // the range is tuned to catch 5 sqrt(n) values (or what the caller asks for) next time (four standard errors of the difference between the
            // smoothed median and the next window's): half of the way, one window's count is a noisy estimate of the density
            const float target = a.target > 0 ? (float)a.target : 5.0f * sqrtf((float)n);
            if (hinted && sh.why[lane] < 0) {
                const float centre = a.centre[c], spread = a.spread[c];
                const float f = fminf(2.0f, fmaxf(0.5f, target / (float)max(sh.inside[lane], 1u)));
                a.spread[c] = spread * (0.5f + 0.5f * f);
                a.centre[c] = centre + (a.smooth > 0.0f ? a.smooth : kWbSmooth) * (med - centre);
            } else {
                // start afresh: from the density inside the first range, which for values that crowd about their median is
                // some 0.7 of the density there (a path that holds few values asked for a target; misses are cheap here,
                // so ours stays wide); hinted ones have missed: half as wide again
                a.spread[c] = hinted ? 1.5f * a.spread[c] : (a.target > 0 ? 0.35f : 0.5f) * sh.width[lane] * target / (float)max(sh.inside[lane], 1u);
                a.centre[c] = med;
            }
        }
        if (hinted && sh.why[lane] >= 0 && a.fb_count) { atomicAdd(a.fb_count, 1u); atomicAdd(a.fb_count + 1 + sh.why[lane], 1u); }
    }
}

}  // namespace

// Windows of up to 1 024 steps in registers.
cudaError_t launch_window_bins(const WindowArgs &a, cudaStream_t st) {
    const int grid = (a.series + 31) / 32;
    if (a.n <= 64) return launch_after(window_bins_kernel<8, 8, false>, grid, 256, st, a);
    if (a.n <= 96) return launch_after(window_bins_kernel<12, 8, false>, grid, 256, st, a);
    if (a.n <= 128) return launch_after(window_bins_kernel<16, 8, false>, grid, 256, st, a);
    if (a.n <= 160) return launch_after(window_bins_kernel<20, 8, false>, grid, 256, st, a);
    if (a.n <= 192) return launch_after(window_bins_kernel<24, 8, false>, grid, 256, st, a);
    if (a.n <= 224) return launch_after(window_bins_kernel<28, 8, false>, grid, 256, st, a);
    if (a.n <= 256) return launch_after(window_bins_kernel<32, 8, false>, grid, 256, st, a);
    if (a.n <= 512) return launch_after(window_bins_kernel<32, 16, false>, grid, 512, st, a);
    if (a.n <= 1024) return launch_after(window_bins_kernel<32, 32, false>, grid, 1024, st, a);
    return launch_after(window_bins_kernel<16, 16, true>, grid, 512, st, a);
}

}  // namespace guard
