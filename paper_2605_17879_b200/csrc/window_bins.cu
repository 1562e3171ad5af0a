// Windowed medians, tile path: a CTA takes 32 adjacent series (lane = series) and splits the window's steps over its
// warps, the values in registers (windows of up to 1 024 steps) or read again in every pass (longer ones).
//   1. a value range that should hold the middle ranks: around the series' smoothed median where an earlier
//      evaluation left one, else between two of 32 spread values of the window;
//   2. one pass counts the values below the range and bins those inside (32 or 64 bins per series; a bin's counters of the
//      32 series are 32 adjacent words, so that the shared-memory reductions of a warp never meet in a bank);
//   3. the bins are scanned for the middle ranks, a second pass fetches the values of those one or two bins, and
//      they are ranked.
// The counts prove the range; one that misses is moved, and a bin with too many values becomes the next range
// (or the answer, if they are all the same), so any values come out exactly; what is still open after a few rounds
// is settled bit by bit.  A value's bin is the low mantissa bits of fma(x, scale, offset): monotone in x whatever
// the rounding, and one full-rate instruction (integer compares and adds run at half rate, conversions slower still).
// Bound by instruction issue, most of it not per value (scan, ranking, barriers: 16 000 cycles a tile, four tiles on an
// SM).  At 64 registers a thread the instances with 16 values or more spill (20 to 236 bytes of stores a thread), outside
// of the passes over the values: 0.8 % of the warp instructions (1 000 steps: 0.10 M of 13.2 M; 180 steps: 0.39 M of 50 M).
// Measured, kernel alone, against what it replaces: 8 192 series of 1 000 steps 24 us (three-way quickselect per thread in
// shared memory: 805), 98 760 first windows of 180 steps 63 us (sort per warp: 135), 8 192 of 100 steps 9.6 us (one
// thread per series: 12 + 5).
#include <math_constants.h>

#include "kernels.h"

namespace guard {

namespace {

constexpr int kWbSample = 16;
constexpr int kWbList = 16;        // values of a bin that are ranked directly
constexpr int kWbRounds = 6;       // rounds of ranges before the bit-by-bit selection
constexpr float kWbSmooth = 0.3f;  // weight of the newest median in the range's centre
constexpr float kWbMagic = 12582912.0f;   // 1.5 * 2^23: adding it leaves an integer in the low mantissa bits
constexpr float kWbMax = 3.402823466e+38f;

template <int BINS>
struct WbShared {
    uint32_t hist[BINS][32];
    uint32_t part[32][32];         // a warp's bins, summed
    uint32_t below[32];            // values below the range
    float f0[32], f1[32];          // values to fetch: those whose fma result lies in [f0, f1]
    float cut[32];                 // last fma result of the lower middle rank's bin
    uint32_t how[32];              // 0 nothing, 1 list and rank, 2 largest up to / smallest beyond `cut`, 3 smallest and largest
    uint32_t q1[32], nl[32], mx[32], mn[32], v1[32], v2[32];
    float lo[32], hi[32];          // the next range
    float list[kWbList][32];
    uint32_t prefix[32], krem[32], cnt[32];   // bit-by-bit selection
};

// t = fma(x, scale, off).  (Inside the assembly of each use: the compiler would otherwise keep the products of one pass
// for the next and spill.)
#define WB_T(x) "fma.rn.f32 t, " x ";\n\t"
// below += (t < T0); if (T0 <= t <= T1) hist[t - T0] += 1
__device__ __forceinline__ void wb_bin(const float x, const float scale, const float off, const float T0, const float T1,
                                       const uint32_t base, uint32_t &below) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .u32 a, b;\n\t.reg .f32 t;\n\t" WB_T("%1, %2, %3")
        "setp.lt.f32 p, t, %4;\n\t"
        "setp.le.and.f32 q, t, %5, !p;\n\t"
        "@p add.u32 %0, %0, 1;\n\t"
        "mov.b32 b, t;\n\t"
        "mad.lo.u32 a, b, 128, %6;\n\t"
        "@q red.shared.add.u32 [a], 1;\n\t}"
        : "+r"(below)
        : "f"(x), "f"(scale), "f"(off), "f"(T0), "f"(T1), "r"(base)
        : "memory");
}
// if (f0 <= t <= f1) hits |= bit
__device__ __forceinline__ void wb_hit(const float x, const float scale, const float off, const float f0, const float f1, const uint32_t bit,
                                       uint32_t &hits) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .f32 t;\n\t" WB_T("%1, %2, %3")
        "setp.ge.f32 p, t, %4;\n\tsetp.le.and.f32 q, t, %5, p;\n\t@q or.b32 %0, %0, %6;\n\t}"
        : "+r"(hits)
        : "f"(x), "f"(scale), "f"(off), "f"(f0), "f"(f1), "r"(bit));
}
// f2key, computed anew at every use (the compiler would keep the keys beside the values and spill)
__device__ __forceinline__ uint32_t wb_key(const float x) {
    uint32_t k;
    asm volatile("{\n\t.reg .s32 s;\n\tshr.s32 s, %1, 31;\n\tor.b32 s, s, 0x80000000;\n\txor.b32 %0, %1, s;\n\t}" : "=r"(k) : "r"(__float_as_uint(x)));
    return k;
}
// G warps of V values per thread; RELOAD: the window is longer than that, V values at a time are read again.
template <int V, int G, int BINS, bool RELOAD>
__global__ void __launch_bounds__(32 * G, G <= 8 ? 4 : (G <= 16 ? 2 : 1)) window_bins_kernel(const WindowArgs a) {
    pdl_wait();
    static_assert(BINS % G == 0 && 32 % G == 0, "warps share the bins and the spread values evenly");
    __shared__ WbShared<BINS> sh;
    const int lane = lane_id(), w = warp_id(), n = a.n;
    const int c = blockIdx.x * 32 + lane;
    const bool active = c < a.series;
    const int cc = active ? c : a.series - 1;
    const int first = a.last_slot - (n - 1) + (a.last_slot < n - 1 ? a.capacity : 0);
    const bool even = !(n & 1);
    const uint32_t k1 = (uint32_t)((n - 1) >> 1), k2 = (uint32_t)(n >> 1);
    const float *colp = a.ring + cc;
    auto load = [&](const int r) -> float {   // step r of the window; beyond its end +inf: above every range
        int slot = first + r;
        if (slot >= a.capacity) slot -= a.capacity;
        return r < n ? __ldg(colp + (size_t)slot * a.row_stride) : CUDART_INF_F;
    };
    float x[V];
    if (!RELOAD) {
#pragma unroll
        for (int i = 0; i < V; ++i) x[i] = load(w + i * G);
    }
    // f(), for each batch of V values of this thread
    auto batches = [&](auto &&f) {
        if (!RELOAD) {
            f();
        } else {
#pragma unroll 1
            for (int r0 = w; r0 < n; r0 += V * G) {
#pragma unroll
                for (int i = 0; i < V; ++i) x[i] = load(r0 + i * G);
                f();
            }
        }
    };
    float centre = 0.0f, spread = 0.0f;
    if (a.use_hint) { centre = a.centre[cc]; spread = a.spread[cc]; }
    const bool hinted = a.use_hint && spread > 0.0f && spread < 1.0e37f && fabsf(centre) < 1.0e37f;
    for (int i = threadIdx.x; i < BINS * 32; i += blockDim.x) (&sh.hist[0][0])[i] = 0u;
    if (w == 0) sh.below[lane] = 0u;
    float lo = centre - spread, hi = centre + spread;
    // series without an earlier result: between the second and the last but one of sixteen spread values of the window
    // (three and a half standard deviations of a sample's rank to either side, and an outlier at either end does not
    // stretch the range), each warp's share of them from its registers
    if (__any_sync(0xFFFFFFFFu, !hinted)) {   // (the same for every warp of the CTA)
        constexpr int J = G < kWbSample ? kWbSample / G : 1;
        uint32_t mine[J];
        int real = 0, rank[J] = {};
        if (w < kWbSample) {
#pragma unroll
            for (int q = 0; q < J; ++q) {
                mine[q] = f2key(RELOAD ? load((int)(((2 * (q * G + w) + 1) * (long long)n) / (2 * kWbSample))) : x[(q * V) / J]);
                sh.part[q * G + w][lane] = mine[q];
            }
        }
#pragma unroll
        for (int q = 0; q < J; ++q) real += RELOAD ? G : min(max(n - ((q * V) / J) * G, 0), min(G, kWbSample));   // (the others are +inf)
        __syncthreads();
        if (w < kWbSample) {
#pragma unroll 8
            for (int i = 0; i < kWbSample; ++i) {
                const uint32_t o = sh.part[i][lane];
#pragma unroll
                for (int q = 0; q < J; ++q) rank[q] += (o < mine[q] || (o == mine[q] && i < q * G + w)) ? 1 : 0;
            }
            const int r_lo = real >> 4, r_hi = real - 1 - (real >> 4);
#pragma unroll
            for (int q = 0; q < J; ++q) {
                if (rank[q] == r_lo) sh.lo[lane] = key2f(mine[q]);
                if (rank[q] == r_hi) sh.hi[lane] = key2f(mine[q]);
            }
        }
        __syncthreads();
        if (!hinted) { lo = sh.lo[lane]; hi = sh.hi[lane]; }
    }
    const float first_width = hi - lo;
    constexpr float T0 = kWbMagic, T1 = kWbMagic + (float)(BINS - 1);
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(&sh.hist[0][lane]) - (uint32_t)(0x4B400000ull * 128ull);   // bits of T0
    uint32_t nin0 = 0;             // values inside the first range (warp 0)
    int why = hinted ? -1 : 0;     // (diagnostic) the first range did not serve: 1 too many values in a bin, 2 below it, 3 above it
    bool live = true;
    int round = 0;
#pragma unroll 1
    for (;; ++round) {
        // ---- count and bin ----
        float scale = hi > lo ? fminf((float)(BINS - 1) / (hi - lo), 1.0e37f) : 1.0f;
        if (hi - lo > kWbMax) scale = 0.0f;             // (a range wider than the largest number: all its values share a bin)
        const float off = live ? __fmaf_rn(-lo, scale, kWbMagic) : -CUDART_INF_F;   // settled series count nothing that matters
        __syncthreads();           // bins are zero
        if (round < kWbRounds) {
            uint32_t below = 0;
            batches([&] {
#pragma unroll
                for (int i = 0; i < V; ++i) wb_bin(x[i], scale, off, T0, T1, base, below);
            });
            atomicAdd(&sh.below[lane], below);
        }
        __syncthreads();
        if (round >= kWbRounds) break;
        // ---- scan: this warp's bins, then where the middle ranks lie ----
        constexpr int NB = BINS / G;
        uint32_t h[NB], mine = 0;
#pragma unroll
        for (int b = 0; b < NB; ++b) h[b] = sh.hist[w * NB + b][lane];
#pragma unroll
        for (int b = 0; b < NB; ++b) { mine += h[b]; sh.hist[w * NB + b][lane] = 0u; }
        sh.part[w][lane] = mine;
        __syncthreads();
        uint32_t r = sh.below[lane], total = 0;
        const uint32_t bel = r;
#pragma unroll
        for (int i = 0; i < G; ++i) {
            const uint32_t p = sh.part[i][lane];
            if (i < w) r += p;
            total += p;
        }
        const bool served = live && bel <= k1 && k2 < bel + total;
        if (served && k2 >= r && k1 < r + mine) {   // (a middle rank, or the gap between them, in this warp's bins)
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const float t = T0 + (float)(w * NB + b);
                if (k1 >= r && k1 - r < h[b]) {
                    sh.f0[lane] = t;
                    sh.cut[lane] = t;
                    sh.q1[lane] = k1 - r;
                    sh.how[lane] = k2 - r < h[b] ? (h[b] <= (uint32_t)kWbList ? 1u : 3u) : 2u;
                }
                if (k2 >= r && k2 - r < h[b]) sh.f1[lane] = t;
                r += h[b];
            }
        }
        if (w == 0) {
            sh.nl[lane] = 0u;
            sh.mx[lane] = 0u;
            sh.mn[lane] = 0xFFFFFFFFu;
            if (!served) {
                sh.how[lane] = 0u;
                sh.f0[lane] = CUDART_INF_F;
                sh.f1[lane] = -CUDART_INF_F;
                if (live) {        // move or stretch the range sixteenfold, from the second time on to everything
                    const float wd = hi - lo, step = round == 0 ? 16.0f * wd + 1.0e-30f : kWbMax;
                    float nlo = lo, nhi = hi;
                    if (bel > k1) { nlo = fmaxf(lo - step, -kWbMax); if (bel > k2) nhi = lo; }
                    if (k2 >= bel + total) { nhi = fminf(hi + step, kWbMax); if (k1 >= bel + total) nlo = hi; }
                    sh.lo[lane] = nlo;
                    sh.hi[lane] = nhi;
                }
            }
            if (round == 0) {
                nin0 = total;
                if (why < 0 && live && !served) why = bel > k1 ? 2 : 3;
            }
        }
        __syncthreads();
        // ---- fetch ----
        {
            const float f0 = sh.f0[lane], f1 = sh.f1[lane];
            batches([&] {
                uint32_t hits = 0;
#pragma unroll
                for (int i = 0; i < V; ++i) wb_hit(x[i], scale, off, f0, f1, 1u << i, hits);
                if (hits) {        // a value or two
                    const uint32_t how = sh.how[lane];
                    const float cut = sh.cut[lane];
                    uint32_t pos = 0;
                    if (how == 1u) pos = atomicAdd(&sh.nl[lane], (uint32_t)__popc(hits));
#pragma unroll 1
                    for (; hits; hits &= hits - 1u) {
                        const int at = __ffs(hits) - 1;
                        float v = x[0];
#pragma unroll
                        for (int i = 1; i < V; ++i) v = at == i ? x[i] : v;
                        if (how == 1u) {   // (the bin's count says that they fit)
                            sh.list[pos++][lane] = v;
                        } else {
                            const uint32_t key = f2key(v);
                            const bool low = how == 3u || __fmaf_rn(v, scale, off) <= cut, high = how == 3u || !low;
                            if (low) atomicMax(&sh.mx[lane], key);
                            if (high) atomicMin(&sh.mn[lane], key);
                        }
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
                const uint32_t mk = f2key(sh.list[j][lane]);
                uint32_t lt = 0, le = 0;
#pragma unroll 4
                for (uint32_t i = 0; i < m; ++i) {
                    const uint32_t o = f2key(sh.list[i][lane]);
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
                if (round == 0 && why < 0) why = 1;
            }
        }
        const bool settled = !live || how == 1u || how == 2u || (how == 3u && sh.mx[lane] == sh.mn[lane]);
        const uint32_t still = __ballot_sync(0xFFFFFFFFu, !settled);   // (the same for every warp of the CTA)
        live = live && !settled;
        if (still == 0u) break;
        __syncthreads();           // ranges and results are written
        if (live) { lo = sh.lo[lane]; hi = sh.hi[lane]; }
        if (w == 0) sh.below[lane] = 0u;
    }
    if (round >= kWbRounds) {      // denormal ranges and the like: one key bit after the other
        if (w == 0) { sh.prefix[lane] = 0u; sh.krem[lane] = k1; sh.cnt[lane] = 0u; sh.mn[lane] = 0xFFFFFFFFu; sh.nl[lane] = 0u; }
        __syncthreads();
#pragma unroll 1
        for (int bit = 31; bit >= 0; --bit) {
            const uint32_t prefix = sh.prefix[lane];
            uint32_t zeros = 0;
            batches([&] {
#pragma unroll
                for (int i = 0; i < V; ++i) {
                    const uint32_t key = wb_key(x[i]);
                    const bool match = bit == 31 || ((key ^ prefix) >> (bit + 1)) == 0u;
                    zeros += match && !((key >> bit) & 1u);
                }
            });
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
        batches([&] {
#pragma unroll
            for (int i = 0; i < V; ++i) {
                const uint32_t key = wb_key(x[i]);
                le += key <= key1;
                if (key > key1) above = min(above, key);
            }
        });
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
            if (hinted && why < 0) {
                const float f = fminf(2.0f, fmaxf(0.5f, target / (float)max(nin0, 1u)));
                a.spread[c] = spread * (0.5f + 0.5f * f);
                a.centre[c] = centre + (a.smooth > 0.0f ? a.smooth : kWbSmooth) * (med - centre);
            } else {
                // start afresh: from the density inside the first range, which for values that crowd about their median is
                // some 0.7 of the density there (a path that holds few values asked for a target; misses are cheap here,
                // so ours stays wide); hinted ones have missed: half as wide again
                a.spread[c] = hinted ? 1.5f * spread : (a.target > 0 ? 0.35f : 0.5f) * first_width * target / (float)max(nin0, 1u);
                a.centre[c] = med;
            }
        }
        if (hinted && why >= 0 && a.fb_count) { atomicAdd(a.fb_count, 1u); atomicAdd(a.fb_count + 1 + why, 1u); }
    }
}

}  // namespace

// Windows of up to 1 024 steps in registers.
cudaError_t launch_window_bins(const WindowArgs &a, cudaStream_t st) {
    const int grid = (a.series + 31) / 32;
    if (a.n <= 64) return launch_after(window_bins_kernel<8, 8, 32, false>, grid, 256, st, a);
    if (a.n <= 128) return launch_after(window_bins_kernel<16, 8, 32, false>, grid, 256, st, a);
    if (a.n <= 192) return launch_after(window_bins_kernel<24, 8, 32, false>, grid, 256, st, a);
    if (a.n <= 256) return launch_after(window_bins_kernel<32, 8, 32, false>, grid, 256, st, a);
    if (a.n <= 512) return launch_after(window_bins_kernel<32, 16, 64, false>, grid, 512, st, a);
    if (a.n <= 1024) return launch_after(window_bins_kernel<32, 32, 64, false>, grid, 1024, st, a);
    return launch_after(window_bins_kernel<16, 16, 64, true>, grid, 512, st, a);
}

}  // namespace guard
