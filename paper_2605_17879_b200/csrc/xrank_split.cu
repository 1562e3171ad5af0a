// Cross-rank selection, split path: blocks of fleets of some thousand to 32 768 ranks with 4 or 8 metrics, one pass
// over the telemetry.  What makes one pass enough is an estimate (c, a) of a column's median and MAD: the running
// mean of the results at the same step position of earlier blocks (consecutive blocks of a fleet have almost the same per-step
// statistics), or, where there is none, a histogram of a sample.
//
//   0. sample   (where there is no estimate from earlier blocks, or it missed lately) one CTA per (step, four metrics):
//               some thousand ranks are binned; the histogram's median, and the half-width about it that holds half of the mass;
//   1. sweep    one warp per (step, strip of ranks): with d = x - c, counts the values below the median's band
//               |d| <= hm and inside the MAD's band | |d| - a | <= ha, and keeps those in either band (8 % of a column
//               of 32 768 ranks, 11 % of 16 384, 22 % of 4 096; 15 to 20 % with estimates from a sample) in shared-memory lists, then in the column's list in global scratch; values that might exceed
//               the threshold are rare: those clear of its possible range set their exceedance bit at once, the
//               others are deferred to a per-step list;
//   2. select   one CTA per column: the median among the kept values of its band, then the MAD among the exact
//               deviations of the kept values of the other; the counts prove the median, and for the MAD that the
//               median did not move the band's ends across it;
//   3. finish   settles the deferred values, and recomputes with the values in registers (xrank_count.cuh) the columns
//               that were not proven, had no estimate, or whose lists overflowed (ties): exact either way.
//
// The sweep is bound by instruction issue, not by memory, and the arithmetic is chosen for the pipe it runs on:
// compares, integer adds and logic go to a half-rate pipe, float adds and multiply-adds do not.  The values are
// scaled by a power of two so that hm and ha are at least 2^24: a difference of two such numbers is then 0 or at least 1
// in magnitude, and a saturating subtraction IS the outcome of a compare, ready to be added.
// Measured, kernels alone, block of 200 steps x 16 384 ranks x 8 metrics: sweep 36 us, select 20, finish 4 (two sweeps,
// two selections, estimates and finish of the two-pass form: 36 + 40 + 9 + 9 + 3 + 4); 50 steps of 24 000 ranks:
// 19 + 10 + 3 (a cluster of four CTAs per step: 77).  What mattered in the sweep: exceedances listed and settled after
// the loop (settled where they are found: + 11 us), lists copied out by the bulk engine (by the warp: + 6), 80 registers
// (64 spill: + 12; prefetching the next batch costs registers and gains nothing).
#include <math_constants.h>

#include <mutex>
#include <type_traits>

#include "xrank_common.cuh"
#include "xrank_count.cuh"

namespace guard {

namespace {

constexpr int kSpThreads = 256;      // CTA of the sample kernel
constexpr int kSpU = 4;              // ranks per thread and sweep batch
constexpr int kSpWarps = 4;          // warps of a sweep CTA (they share nothing but the columns' bands)
constexpr int kSpSlack = 32;         // words behind each shared-memory list that absorb the stores of a full list
constexpr int kSpSlow = 64;          // ranks with a possible exceedance a sweep warp lists
constexpr int kSpAmb = 1024;         // deferred exceedance decisions per step
constexpr int kSpSBins = 2048;       // sample histogram bins
constexpr int kSpMaxM = 8;
constexpr int kSpMaxRanks = 32768;
constexpr int kSpRest = 8;           // blocks a column whose list overflowed (ties) stays away from the sweep,
                                     // or whose estimate missed takes a sample instead of the blocks before
constexpr float kSpSmooth = 0.3f;    // weight of the newest result in the estimate
constexpr float kFltMax = 3.402823466e+38f;
// half-widths of the bands, in units of MAD / sqrt(n) for an estimate whose variance is that of n values (4.6 standard
// errors; normal data: 1.858 MAD / sqrt(n) for a median, 1.167 for a MAD, 2.194 for both together)
constexpr float kSpMed = 8.55f, kSpMad = 5.37f, kSpBoth = 10.1f;

struct SpGeom {
    int chunks;     // sweep CTAs per step
    int strip;      // ranks per sweep warp
    int cap;        // values per metric a sweep warp can keep
    int col_cap;    // ... and a column's list
    int s;          // sampled ranks
    int period;     // one run of four consecutive ranks is sampled out of every `period`
    float q_sample; // a sample's standard error is that of 1 / q_sample^2 values
};

// Per-column record in global scratch.
struct SpCol {
    float c, a;          // estimates of the median and the MAD
    float q, extra;      // their standard error is that of 1 / q^2 values; relative widening of the bands
    float v;             // variance of an estimate from earlier blocks, in units of a single block's (0: from a sample)
    uint32_t epoch;      // SpScratch::epoch: the record holds an estimate
    uint16_t rest;       // blocks left before the column is swept again
    uint16_t resample;   // blocks left that take a sample
    uint32_t nk;         // kept values
    uint32_t below, inner;
    float med, rhs;      // the median and the exact threshold
};

// The estimate after an exact result: a running mean (its error adds to the next result's own), or the result itself
// where there was none from earlier blocks.
__device__ __forceinline__ void sp_learn(SpCol &col, const float med, const float mad, const bool afresh, const int R) {
    const bool first = afresh || col.v == 0.0f;
    col.c = first ? med : col.c + kSpSmooth * (med - col.c);
    col.a = first ? mad : col.a + kSpSmooth * (mad - col.a);
    col.v = first ? 1.0f : (1.0f - kSpSmooth) * (1.0f - kSpSmooth) * col.v + kSpSmooth * kSpSmooth;
    col.q = sqrtf((1.0f + col.v) / (float)R);
    col.extra = 0.0f;
}

struct SpScratch {
    SpCol *col;          // [S_max][M]
    uint32_t *fail;      // [S_max] metrics to be recomputed (a bit each); bit 31: one of them had been swept
    uint32_t *namb;      // [S_max] deferred exceedance decisions
    uint32_t *amb;       // [S_max][kSpAmb] (rank << 5 | metric)
    float *list;         // [S_max][M][col_cap] kept values
    uint32_t epoch;
};

// What the sweep and the selection derive from a column's estimate.  sc * (x - c) is what the bands are compared with.
struct SpBands {
    float c, sc, hm, a, ha, rlo, rhi;   // hm, a, ha, rlo, rhi in units of 1 / sc
    float hd;                           // how far the MAD may be from its estimate for rlo, rhi to hold (unscaled)
    float inv;                          // 1 / sc
    bool ok;
};

__device__ __forceinline__ SpBands sp_bands(const SpCol &col, const uint32_t epoch, const MetricParams &p, const int m) {
    SpBands b;
    const float med = col.c, mad = col.a, w = mad * col.q, x = mad * col.extra;
    const float hm = kSpMed * w + x, ha = kSpBoth * w + 1.5f * x, hd = kSpMad * w + x;
    const float rel = p.floor_rel[m];
    const float lo = fmaxf(fmaxf(mad - hd, rel * fmaxf(fabsf(med) - hm, 0.0f)), p.floor_abs[m]);
    const float hi = fmaxf(fmaxf(mad + hd, rel * (fabsf(med) + hm)), p.floor_abs[m]);
    const float rlo = p.thrp[m] * lo * 0.99999f - 1.00001f * hm, rhi = p.thrp[m] * hi * 1.00001f + 1.00001f * hm;
    // the power of two that lifts hm (the smaller half-width) to 2^24 .. 2^25
    const int e = (int)(__float_as_uint(hm) >> 23) - 127;
    b.ok = col.epoch == epoch && col.rest == 0 && mad > 0.0f && mad < 1.0e36f && fabsf(med) < 1.0e36f && e >= -100 && e <= 100 && rlo > mad;
    const float sc = __uint_as_float((uint32_t)(127 + 24 - e) << 23);
    b.ok = b.ok && fabsf(med) * sc < 1.0e37f && mad * sc < 1.0e37f;
    b.c = b.ok ? med : 0.0f;
    b.sc = b.ok ? sc : 0.0f;
    b.hm = b.ok ? hm * sc : -1.0f;
    b.a = b.ok ? mad * sc : 0.0f;
    b.ha = b.ok ? ha * sc : -1.0f;
    b.rlo = b.ok ? rlo * sc : CUDART_INF_F;
    b.rhi = b.ok ? rhi * sc : CUDART_INF_F;
    b.hd = hd;
    b.inv = __uint_as_float((uint32_t)(127 - 24 + e) << 23);
    return b;
}

// ---- 0. sample ---------------------------------------------------------------------------------
constexpr int kSpSmpG = kSpThreads / 4;                 // threads per metric in the scan
constexpr int kSpSmpBatch = 16;                         // sampled ranks in flight per thread

struct SpSampleShared {
    uint32_t hist[4][kSpSBins / 2 + 1];   // 16-bit bins, two per word; then the values in the bins before each
    uint32_t warp_tot[4][2];
    float inv_bw[4], off[4], pos[4];
    int ok[4];
    uint32_t half[4], keep[4], again[4];
};

// The sample of a step: runs of four consecutive ranks, so that a warp's 128-bit loads use whole cache lines.  One
// CTA handles four metrics: every thread bins the four components of its float4; then 64 threads per metric
// scan their histogram.
__global__ void __launch_bounds__(kSpThreads, 3) xsplit_sample_kernel(const XrankArgs a, const SpGeom g, const SpScratch sc, const int rows) {
    pdl_wait();
    __shared__ SpSampleShared sh;
    const int q = blockIdx.x, t = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int R = a.R, M = a.M;
    const int slot = a.first_slot + t - (t >= a.capacity - a.first_slot ? a.capacity : 0);
    const float *row = a.base + (size_t)slot * a.row_stride;
    SpCol *cols = sc.col + (size_t)t * M + 4 * q;
    const bool reuse = t < rows;   // the scratch has held this step position before
    if (tid == 0 && q == 0) { sc.fail[t] = 0u; sc.namb[t] = 0u; }
    if (tid < 4) { cols[tid].nk = 0u; cols[tid].below = 0u; cols[tid].inner = 0u; }
    // columns with an estimate from earlier blocks need no sample
    const bool known = reuse && cols[tid & 3].epoch == sc.epoch;
    const uint32_t again = known ? cols[tid & 3].resample : 0u;   // (thread c < 4 speaks for column c)
    if (__syncthreads_and(known && again == 0u)) return;

    const int first = (g.period - 4) >> 1;
    float xpre = 0.0f;   // (warps 0..3) the 32 spread values that fix a metric's bin map
    if (warp < 4) xpre = __ldg(row + (size_t)min(R - 1, (int)(((long long)(2 * lane + 1) * R) >> 6)) * M + 4 * q + warp);
    for (int i = tid; i < 4 * (kSpSBins / 2 + 1); i += kSpThreads) (&sh.hist[0][0])[i] = 0u;
    if (tid < 4) {
        sh.half[tid] = 0xFFFFFFFFu;
        sh.keep[tid] = known && again == 0u;
        sh.again[tid] = again ? again - 1u : 0u;
        if (!known) cols[tid].rest = 0;
    }
    if (warp < 4) {
        const uint32_t key = ct_warp_sort(f2key(xpre), lane);
        const float c50 = key2f(__shfl_sync(0xFFFFFFFFu, key, 16));
        const float c25 = key2f(__shfl_sync(0xFFFFFFFFu, key, 8)), c75 = key2f(__shfl_sync(0xFFFFFFFFu, key, 23));
        if (lane == 0) {
            const float sig = (c75 - c25) / 1.35f;
            const float inv_bw = 64.0f / sig;     // 2048 bins over +-16 sigma
            const float off = (float)(1024.0 - (double)c50 * (double)inv_bw);
            sh.ok[warp] = (sig > 0.0f) && (inv_bw < kFltMax) && (fabsf(off) < kFltMax);
            sh.inv_bw[warp] = sh.ok[warp] ? inv_bw : 0.0f;
            sh.off[warp] = sh.ok[warp] ? off : 0.0f;
        }
    }
    __syncthreads();
    for (int i0 = 0; i0 < g.s; i0 += kSpSmpBatch * kSpThreads) {
        float4 xs[kSpSmpBatch];
#pragma unroll
        for (int j = 0; j < kSpSmpBatch; ++j) {
            const int i = i0 + tid + j * kSpThreads;   // index into the sample
            xs[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (i < g.s) xs[j] = __ldg(reinterpret_cast<const float4 *>(row + (size_t)((i >> 2) * g.period + first + (i & 3)) * M) + q);
        }
#pragma unroll
        for (int j = 0; j < kSpSmpBatch; ++j) {
            if (i0 + tid + j * kSpThreads < g.s) {
                const float v[4] = {xs[j].x, xs[j].y, xs[j].z, xs[j].w};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    int b = __float2int_rd(__fmaf_rn(v[c], sh.inv_bw[c], sh.off[c]));
                    b = min(max(b, 0), kSpSBins - 1);
                    atomicAdd(&sh.hist[c][b >> 1], (b & 1) ? 0x10000u : 1u);
                }
            }
        }
    }
    __syncthreads();
    // cumulative counts: 64 threads per metric, WPT words (2 bins each) per thread
    const int c = tid / kSpSmpG, gt = tid % kSpSmpG, gw = gt >> 5;
    constexpr int WPT = kSpSBins / 2 / kSpSmpG;
    uint32_t w[WPT], sum = 0;
#pragma unroll
    for (int i = 0; i < WPT; ++i) { w[i] = sh.hist[c][gt * WPT + i]; sum += (w[i] & 0xFFFFu) + (w[i] >> 16); }
    uint32_t incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, incl, d); if (lane >= d) incl += u; }
    if (lane == 31) sh.warp_tot[c][gw] = incl;
    __syncthreads();
    uint32_t run = (gw ? sh.warp_tot[c][0] : 0u) + incl - sum;
    const uint32_t mid = (uint32_t)g.s / 2u;
#pragma unroll
    for (int i = 0; i < WPT; ++i) {
        const uint32_t c0 = w[i] & 0xFFFFu, c1 = w[i] >> 16;
        const int b = 2 * (gt * WPT + i);
        const uint32_t both = run | ((run + c0) << 16);
        if (mid >= run && mid < run + c0) sh.pos[c] = (float)b + (float)(mid - run) / (float)c0;
        run += c0;
        sh.hist[c][b >> 1] = both;   // (this thread's words; it has read them)
        if (mid >= run && mid < run + c1) sh.pos[c] = (float)(b + 1) + (float)(mid - run) / (float)c1;
        run += c1;
    }
    if (gt == kSpSmpG - 1) sh.hist[c][kSpSBins / 2] = (uint32_t)g.s;
    const uint16_t *cum = reinterpret_cast<const uint16_t *>(sh.hist[c]);
    __syncthreads();
    // the smallest whole number of bins to either side of the median that holds half of the mass
    const float pos = sh.pos[c];
    auto mass = [&](const float v) -> float {   // values below bin coordinate v
        if (v <= 0.0f) return 0.0f;
        if (v >= (float)kSpSBins) return (float)g.s;
        const int i = (int)v;
        const float lo = (float)cum[i];
        return lo + (v - (float)i) * ((float)cum[i + 1] - lo);
    };
    const float halfm = 0.5f * (float)g.s;
    for (int j = gt + 1; j <= kSpSBins / 2; j += kSpSmpG)
        if (mass(pos + (float)j) - mass(pos - (float)j) >= halfm) { atomicMin(&sh.half[c], (uint32_t)j); break; }
    __syncthreads();
    if (gt == 0 && !sh.keep[c]) {
        SpCol &col = cols[c];
        const uint32_t h = sh.half[c];
        const bool ok = sh.ok[c] && h != 0xFFFFFFFFu;
        float med = 0.0f, mad = 0.0f;
        if (ok) {
            const float m1 = mass(pos + (float)h) - mass(pos - (float)h), m0 = mass(pos + (float)(h - 1)) - mass(pos - (float)(h - 1));
            const double inv = 1.0 / (double)sh.inv_bw[c];
            med = (float)(((double)pos - (double)sh.off[c]) * inv);
            mad = (float)(((double)(h - 1) + (m1 > m0 ? (double)((halfm - m0) / (m1 - m0)) : 0.0)) * inv);
        }
        col.c = med;
        col.a = mad;
        col.q = g.q_sample;
        col.extra = 0.01f;     // the bins' share of the error
        col.v = 0.0f;
        col.resample = (uint16_t)sh.again[c];
        col.epoch = ok ? sc.epoch : 0u;
    }
}

// ---- 1. sweep ----------------------------------------------------------------------------------
struct SpSweepShared {
    float sc[kSpMaxM], b[kSpMaxM], hm[kSpMaxM], a[kSpMaxM], ha[kSpMaxM], rlo[kSpMaxM], rhi[kSpMaxM];
    uint32_t any;
    uint32_t nslow[kSpWarps], slow[kSpWarps][kSpSlow];   // ranks with a value beyond rlo (rank << 1 | metric quad)
};

// One value: d = sc * (x - c) (sign of the bad direction folded into sc); acc += below + 1024 * inner; the kept bit;
// chk turns NaN when d is not finite.
template <uint32_t BIT>
__device__ __forceinline__ float sp_cell(const float x, const float sc, const float b, const float hm, const float a, const float ha,
                                         float &acc, uint32_t &mask, float &chk) {
    float d;
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .f32 s, t, e, f, n;\n\t"
        "fma.rn.f32 %0, %4, %5, %6;\n\t"
        "neg.f32 n, %7;\n\t"
        "sub.rn.sat.f32 s, n, %0;\n\t"            // 1 where d < -hm
        "abs.f32 t, %0;\n\t"
        "sub.rn.f32 e, t, %8;\n\t"
        "neg.f32 n, %9;\n\t"
        "sub.rn.sat.f32 f, n, e;\n\t"             // 1 where |d| - a < -ha
        "add.rn.f32 %1, %1, s;\n\t"
        "fma.rn.f32 %1, f, 0f44800000, %1;\n\t"
        "fma.rn.f32 %3, %0, 0f00000000, %3;\n\t"
        "abs.f32 e, e;\n\t"
        "setp.le.f32 p, t, %7;\n\t"
        "setp.le.or.f32 p, e, %9, p;\n\t"
        "@p or.b32 %2, %2, %10;\n\t}"
        : "=&f"(d), "+f"(acc), "+r"(mask), "+f"(chk)
        : "f"(x), "f"(sc), "f"(b), "f"(hm), "f"(a), "f"(ha), "n"(BIT));
    return d;
}
// if (mask & BIT) { shared[addr] = x; addr += 4; }
template <uint32_t BIT>
__device__ __forceinline__ void sp_keep(const float x, const uint32_t mask, uint32_t &addr) {
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tand.b32 t, %1, %3;\n\tsetp.ne.u32 p, t, 0;\n\t@p st.shared.f32 [%0], %2;\n\t@p add.u32 %0, %0, 4;\n\t}"
                 : "+r"(addr)
                 : "r"(mask), "f"(x), "n"(BIT)
                 : "memory");
}
// one step of an inclusive scan over lanes: incl += value of lane (lane - d) where that lane exists
__device__ __forceinline__ void sp_scan_step(uint32_t &incl, const int d) {
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 r;\n\tshfl.sync.up.b32 r|p, %0, %1, 0, 0xffffffff;\n\t@p add.u32 %0, %0, r;\n\t}"
                 : "+r"(incl)
                 : "r"(d));
}

// Kept values: every batch (kSpU ranks x 4 metrics per thread) the lanes of a metric quad scan their four 8-bit kept
// counts (one packed word) and every lane stores its kept values at its own offset of the warp's lists.  A warp owns its
// strip of ranks, its lists and its place in the columns' lists: after the bands are known no warp waits for another.
// Stores past a list's capacity land in the slack behind it; the full list is detected from the counter.
template <int NQ>
__global__ void __launch_bounds__(32 * kSpWarps, 6) xsplit_sweep_kernel(const XrankArgs a, const MetricParams p, const SpGeom g, const SpScratch sc) {
    pdl_wait();
    constexpr int M = 4 * NQ, LPI = 32 / NQ;
    extern __shared__ __align__(16) uint32_t slist[];   // [kSpWarps][M][cap + kSpSlack]
    __shared__ SpSweepShared sh;
    const int chunk = blockIdx.x, t = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int R = a.R;
    const int slot = a.first_slot + t - (t >= a.capacity - a.first_slot ? a.capacity : 0);
    const float *row = a.base + (size_t)slot * a.row_stride;
    uint8_t *maskrow = a.mask_base ? reinterpret_cast<uint8_t *>(a.mask_base) + (size_t)slot * R : nullptr;
    const int r0 = min(R, (chunk * kSpWarps + warp) * g.strip), r1 = min(R, r0 + g.strip);
    SpCol *cols = sc.col + (size_t)t * M;
    const int cap = g.cap;
    const int q = lane & (NQ - 1), rl = lane / NQ;

    float x[kSpU][4];
    auto load = [&](const int base, const bool guard) {
        const float4 *src = reinterpret_cast<const float4 *>(row + (size_t)(base + rl) * M) + q;
#pragma unroll
        for (int j = 0; j < kSpU; ++j) {
            float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (!guard || base + j * LPI + rl < r1) v = __ldg(src + (size_t)j * LPI * NQ);
            x[j][0] = v.x; x[j][1] = v.y; x[j][2] = v.z; x[j][3] = v.w;
        }
    };
    constexpr int span = LPI * kSpU;
    load(r0, true);              // in flight while the bands are worked out
    if (tid < M) {
        const SpBands b = sp_bands(cols[tid], sc.epoch, p, tid);
        const float s = p.dir[tid] < 0 ? -b.sc : b.sc;
        sh.sc[tid] = s;
        sh.b[tid] = -s * b.c;
        sh.hm[tid] = b.hm; sh.a[tid] = b.a; sh.ha[tid] = b.ha; sh.rlo[tid] = b.rlo; sh.rhi[tid] = b.rhi;
        const uint32_t bad = __ballot_sync((1u << M) - 1u, !b.ok);
        if (tid == 0) {
            sh.any = bad != (1u << M) - 1u;
            if (bad && chunk == 0) atomicOr(&sc.fail[t], bad);
        }
    }
    if (lane == 0) sh.nslow[warp] = 0u;
    if (maskrow) {   // this warp's part of the exceedance row starts at zero; bits are OR-ed in
        uint8_t *m0 = maskrow + r0, *m1 = maskrow + r1;
        uint8_t *w0 = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(m0) + 3) & ~(uintptr_t)3);
        uint8_t *w1 = reinterpret_cast<uint8_t *>(reinterpret_cast<uintptr_t>(m1) & ~(uintptr_t)3);
        if (w0 > w1) w0 = w1 = m1;
        for (uint8_t *w = w0 + 4 * lane; w < w1; w += 128) *reinterpret_cast<uint32_t *>(w) = 0u;
        if (lane < 4 && m0 + lane < w0) m0[lane] = 0;
        if (lane >= 4 && lane < 8 && w1 + (lane - 4) < m1) w1[lane - 4] = 0;
    }
    __syncthreads();             // (also: zeroed before any thread ORs a bit in)
    if (!sh.any) return;         // (the finish kernel recomputes the step, non-finite values included)

    float ks[4], kb[4], hm[4], am[4], ha[4], rlo[4], acc[4] = {0.0f, 0.0f, 0.0f, 0.0f}, chk = 0.0f;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int m = 4 * q + c;
        ks[c] = sh.sc[m]; kb[c] = sh.b[m]; hm[c] = sh.hm[m]; am[c] = sh.a[m]; ha[c] = sh.ha[m]; rlo[c] = sh.rlo[m];
    }
    const uint32_t pitch = (uint32_t)(cap + kSpSlack) * 4u;   // bytes between the lists of consecutive metrics
    const uint32_t list_s = (uint32_t)__cvta_generic_to_shared(slist) + (uint32_t)(warp * M + 4 * q) * pitch;
    const uint32_t cap16 = (uint32_t)cap | ((uint32_t)cap << 16);
    uint32_t n01 = 0, n23 = 0;   // kept so far, two 16-bit fields per word

    // A rank (of one metric quad) with a value beyond rlo, tested against the threshold's possible range [rlo, rhi]: the
    // bit is set at once or the decision deferred until the MAD is known.
    auto settle = [&](const int r, const int quad) {
        if (!maskrow) return;
        const float4 v = __ldg(reinterpret_cast<const float4 *>(row + (size_t)r * M) + quad);
        const float xv[4] = {v.x, v.y, v.z, v.w};
        uint32_t eb = 0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int m = 4 * quad + c;
            const float d = __fmaf_rn(xv[c], sh.sc[m], sh.b[m]);
            if (d > sh.rhi[m]) {
                eb |= 1u << m;
            } else if (d > sh.rlo[m]) {
                const uint32_t pos = atomicAdd(sc.namb + t, 1u);
                if (pos < (uint32_t)kSpAmb) sc.amb[(size_t)t * kSpAmb + pos] = ((uint32_t)r << 5) | (uint32_t)m;
            }
        }
        if (eb) {
            const uintptr_t at = reinterpret_cast<uintptr_t>(maskrow + r);
            atomicOr(reinterpret_cast<unsigned int *>(at & ~(uintptr_t)3), eb << (8 * (at & 3)));
        }
    };
    auto batch = [&](const int base, const bool guard) {
        uint32_t mask = 0, slow = 0;   // bit 4 c + j: value of metric c and rank j is kept; rank j has a value beyond rlo
        auto one = [&](auto jc) {
            constexpr int J = decltype(jc)::value;
            if (guard && base + J * LPI + rl >= r1) return;
            const float d0 = sp_cell<1u << J>(x[J][0], ks[0], kb[0], hm[0], am[0], ha[0], acc[0], mask, chk);
            const float d1 = sp_cell<16u << J>(x[J][1], ks[1], kb[1], hm[1], am[1], ha[1], acc[1], mask, chk);
            const float d2 = sp_cell<256u << J>(x[J][2], ks[2], kb[2], hm[2], am[2], ha[2], acc[2], mask, chk);
            const float d3 = sp_cell<4096u << J>(x[J][3], ks[3], kb[3], hm[3], am[3], ha[3], acc[3], mask, chk);
            if (d0 > rlo[0] || d1 > rlo[1] || d2 > rlo[2] || d3 > rlo[3]) slow |= 1u << J;
        };
        one(std::integral_constant<int, 0>{});
        one(std::integral_constant<int, 1>{});
        one(std::integral_constant<int, 2>{});
        one(std::integral_constant<int, 3>{});
        // the rare remainder goes on the warp's list
        for (; slow; slow &= slow - 1u) {
            const int r = base + (__ffs(slow) - 1) * LPI + rl;
            const uint32_t pos = atomicAdd(&sh.nslow[warp], 1u);
            if (pos < (uint32_t)kSpSlow) sh.slow[warp][pos] = ((uint32_t)r << 1) | (uint32_t)q;
            else settle(r, q);
        }
        // kept counts of the four metrics, a byte each
        uint32_t packed = mask - ((mask >> 1) & 0x5555u);
        packed = (packed & 0x3333u) + ((packed >> 2) & 0x3333u);
        packed = (packed | (packed << 8)) & 0x00FF00FFu;
        packed = (packed | (packed << 4)) & 0x0F0F0F0Fu;
        // inclusive scan over the lanes of the same metric quad
        uint32_t incl = packed;
#pragma unroll
        for (int d = NQ; d < 32; d <<= 1) sp_scan_step(incl, d);
        const uint32_t total = __shfl_sync(0xFFFFFFFFu, incl, 32 - NQ + q);
        const uint32_t excl = incl - packed;
        // list positions of this thread's first kept value per metric (two 16-bit fields per word), clamped
        const uint32_t p01 = __vminu2(n01 + __byte_perm(excl, 0, 0x4140), cap16);
        const uint32_t p23 = __vminu2(n23 + __byte_perm(excl, 0, 0x4342), cap16);
        n01 += __byte_perm(total, 0, 0x4140);
        n23 += __byte_perm(total, 0, 0x4342);
        uint32_t addr[4];
        addr[0] = list_s + 4u * (p01 & 0xFFFFu);
        addr[1] = list_s + pitch + 4u * (p01 >> 16);
        addr[2] = list_s + 2u * pitch + 4u * (p23 & 0xFFFFu);
        addr[3] = list_s + 3u * pitch + 4u * (p23 >> 16);
        sp_keep<0x1u>(x[0][0], mask, addr[0]); sp_keep<0x10u>(x[0][1], mask, addr[1]); sp_keep<0x100u>(x[0][2], mask, addr[2]); sp_keep<0x1000u>(x[0][3], mask, addr[3]);
        sp_keep<0x2u>(x[1][0], mask, addr[0]); sp_keep<0x20u>(x[1][1], mask, addr[1]); sp_keep<0x200u>(x[1][2], mask, addr[2]); sp_keep<0x2000u>(x[1][3], mask, addr[3]);
        sp_keep<0x4u>(x[2][0], mask, addr[0]); sp_keep<0x40u>(x[2][1], mask, addr[1]); sp_keep<0x400u>(x[2][2], mask, addr[2]); sp_keep<0x4000u>(x[2][3], mask, addr[3]);
        sp_keep<0x8u>(x[3][0], mask, addr[0]); sp_keep<0x80u>(x[3][1], mask, addr[1]); sp_keep<0x800u>(x[3][2], mask, addr[2]); sp_keep<0x8000u>(x[3][3], mask, addr[3]);
    };
    int base = r0;
    for (; base + span <= r1; base += span) {
        if (base != r0) load(base, false);
        batch(base, false);
    }
    if (base < r1) {
        if (base != r0) load(base, true);
        batch(base, true);
    }
    if (chk != 0.0f && a.check_finite) {   // (NaN) a value that is not finite, or a finite one far from everything: looked at again
        bool bad = false;
        for (int r = r0 + rl; r < r1; r += LPI)
            for (int c = 0; c < 4; ++c) bad |= nonfinite_bits(__float_as_uint(__ldg(row + (size_t)r * M + 4 * q + c)));
        if (bad) atomicOr(a.status, kStatNonFinite);
    }
    __syncwarp();
    // counts, summed over the lanes of a quad class; lane 4 q + c then speaks for its metric
    uint32_t cnt[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint32_t v = (uint32_t)acc[c];
        cnt[c] = (uint32_t)group_sum<NQ>((int)((v & 1023u) | ((v >> 10) << 16)));
    }
    uint32_t mine = 0, pos = 0;
    // (the sums are the same in all lanes with the same q: lane 4 q + c reads metric c from lane q)
    const int from = (lane >> 2) & (NQ - 1);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint32_t s = __shfl_sync(0xFFFFFFFFu, cnt[c], from);
        if ((lane & 3) == c) mine = s;
    }
    const uint32_t s01 = __shfl_sync(0xFFFFFFFFu, n01, from), s23 = __shfl_sync(0xFFFFFFFFu, n23, from);
    const uint32_t nk = (((lane & 2) ? s23 : s01) >> (16 * (lane & 1))) & 0xFFFFu;
    // whole quads of four: every part of a column's list starts on a 16-byte boundary (NaN is in no band)
    const uint32_t npad = (nk + 3u) & ~3u;
    if (lane < M) {
        atomicAdd(&cols[lane].below, mine & 0xFFFFu);
        atomicAdd(&cols[lane].inner, mine >> 16);
        // (a full list of this warp fills the column's beyond its capacity, too)
        pos = atomicAdd(&cols[lane].nk, nk > (uint32_t)cap ? (uint32_t)g.col_cap + 4u : npad);
        if (nk <= (uint32_t)cap)
            for (uint32_t i = nk; i < npad; ++i) slist[(size_t)(warp * M + lane) * (cap + kSpSlack) + i] = 0x7FFFFFFFu;
    }
    const uint32_t nslow = sh.nslow[warp];
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // every lane's stores to the lists, before the copies
    __syncwarp();
    // the lists go out as bulk copies (shared memory to global), a lane per metric
    if (lane < M && nk <= (uint32_t)cap && pos + npad <= (uint32_t)g.col_cap && npad) {
        float *dst = sc.list + ((size_t)t * M + lane) * g.col_cap + pos;
        const uint32_t src = (uint32_t)__cvta_generic_to_shared(slist + (size_t)(warp * M + lane) * (cap + kSpSlack));
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(4u * npad) : "memory");
    }
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    for (uint32_t i = lane; i < min(nslow, (uint32_t)kSpSlow); i += 32) settle((int)(sh.slow[warp][i] >> 1), (int)(sh.slow[warp][i] & 1u));
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");   // (the lists have been written before the CTA gives its shared memory up)
}

// ---- 2. selection ------------------------------------------------------------------------------
// Keys of the two middle ranks among those that key() gives for a list's n values (whole quads; 0xFFFFFFFF: not among them), left in
// sh.v1[0] / sh.v2[0]; the range is in sh.lo / sh.width, the bins are zero.  ranks(k1, k2) gives their places among the
// keys once key() has seen every value, or false.  The steps of ct_select, with the list read again in every pass (it
// is in the first-level cache): what a pass keeps in registers would halve the CTAs that share an SM.
template <int T, class Key, class Ranks>
__device__ __forceinline__ bool sp_pick(Key key, Ranks ranks, const uint32_t n, CtShared<1> &sh) {
    const int tid = threadIdx.x, lane = lane_id(), warp = warp_id();
    const uint32_t hist = (uint32_t)__cvta_generic_to_shared(sh.hist[0]);
    uint32_t k1 = 0, k2 = 0;
    bool searching = true;         // (of warp 0)
#pragma unroll 1
    for (int it = 0; it < kCtMaxIter; ++it) {
        if (tid == 0) sh.any_open[it & 1] = 0u;
        __syncthreads();           // range, counters and bins are ready
        {
            const uint32_t lo = sh.lo[0], width = sh.width[0];
            const int sft = ct_shift(width);
            uint32_t below = 0;
#pragma unroll 2
            for (uint32_t i = tid; i < n / 4u; i += T) {
                const float4 v = key.list[i];
                ct_bin(key(v.x, it == 0), lo, width, sft, hist, below);
                ct_bin(key(v.y, it == 0), lo, width, sft, hist, below);
                ct_bin(key(v.z, it == 0), lo, width, sft, hist, below);
                ct_bin(key(v.w, it == 0), lo, width, sft, hist, below);
            }
            below = __reduce_add_sync(0xFFFFFFFFu, below);
            if (lane == 0) atomicAdd(&sh.below[0], below);
        }
        if (it == 0) key.share();
        __syncthreads();
        if (it == 0 && !ranks(k1, k2)) return false;
        if (warp == 0) ct_scan<1>(sh, 0, k1, k2);
        __syncthreads();
        {
            const uint32_t f0 = sh.f0[0], fw = sh.fe[0] - f0, how = sh.how[0], cutk = sh.cutk[0];
            key.range(f0, sh.fe[0]);
            auto take = [&](const float x) {
                if (!key.near(x)) return;          // (as a rule: no key is worked out)
                const uint32_t k = key(x, false);
                if (k - f0 <= fw) {
                    if (how == 1u) {
                        const uint32_t pos = atomicAdd(&sh.nl[0], 1u);
                        if (pos < (uint32_t)kCtList) sh.list[0][pos] = k;
                    } else if (how >= 2u) {
                        if (how == 3u || k <= cutk) atomicMax(&sh.mx[0], k);
                        if (how == 3u || k > cutk) atomicMin(&sh.mn[0], k);
                    }
                }
            };
#pragma unroll 2
            for (uint32_t i = tid; i < n / 4u; i += T) {
                const float4 v = key.list[i];
                take(v.x);
                take(v.y);
                take(v.z);
                take(v.w);
            }
        }
        __syncthreads();
        if (warp == 0) {
            searching = ct_settle<1>(sh, 0, k2 != k1);
            if (lane == 0 && searching) sh.any_open[it & 1] = 1u;
        }
        __syncthreads();
        if (sh.any_open[it & 1] == 0u) return true;
    }
    if (tid == 0) sh.bad = 1u;
    return true;
}

// Keys of the kept values in the median's band (the very comparisons of the sweep; NaN is in no band), and how many values
// are in either band.
struct SpMedianKey {
    const float4 *list;
    float ks, kb, hm, a, ha;
    uint32_t *s_n;
    uint32_t nm = 0, na = 0;
    float lo = 0.0f, hi = 0.0f;
    __device__ __forceinline__ uint32_t operator()(const float x, const bool count) {
        const float d = fabsf(__fmaf_rn(x, ks, kb));
        const bool in = d <= hm;
        if (count) {
            nm += in;
            na += fabsf(__fsub_rn(d, a)) <= ha;
        }
        return in ? f2key(x) : 0xFFFFFFFFu;
    }
    // values that may have keys from f0 to fe (all of these among them)
    __device__ __forceinline__ void range(const uint32_t f0, const uint32_t fe) { lo = key2f(f0); hi = key2f(fe); }
    __device__ __forceinline__ bool near(const float x) const { return x >= lo && x <= hi; }
    __device__ __forceinline__ void share() {
        const uint32_t tot = __reduce_add_sync(0xFFFFFFFFu, nm | (na << 16));
        if (lane_id() == 0) { atomicAdd(&s_n[0], tot & 0xFFFFu); atomicAdd(&s_n[1], tot >> 16); }
    }
};
// ... and of the exact deviations of those in the MAD's band.
struct SpMadKey {
    const float4 *list;
    float ks, kb, a, ha, med;
    float lo = 0.0f, hi = 0.0f;
    __device__ __forceinline__ uint32_t operator()(const float x, const bool) const {
        const bool in = fabsf(__fsub_rn(fabsf(__fmaf_rn(x, ks, kb)), a)) <= ha;
        return in ? __float_as_uint(__fsub_rn(x, med)) << 1 : 0xFFFFFFFFu;
    }
    __device__ __forceinline__ void range(const uint32_t f0, const uint32_t fe) { lo = __uint_as_float(f0 >> 1); hi = __uint_as_float(fe >> 1); }
    __device__ __forceinline__ bool near(const float x) const {
        const float d = fabsf(__fsub_rn(x, med));
        return d >= lo && d <= hi;
    }
    __device__ __forceinline__ void share() const {}
};

// The median and the MAD of a column from its kept values; why it is not proven, or -1.
template <int T>
__device__ __forceinline__ int sp_select(const float *list, const uint32_t n, const SpBands &b, const float sgn, const uint32_t below, const uint32_t inner,
                                         const int R, CtShared<1> &sh, uint32_t *s_n, float &med, float &mad) {
    const int tid = threadIdx.x;
    const bool even = (R & 1) == 0;
    const uint32_t r1 = (uint32_t)((R - 1) / 2), r2 = (uint32_t)(R / 2);
    const float ks = sgn * b.sc, kb = -ks * b.c, w = b.hm * b.inv;
    for (int i = tid; i < kCtBins; i += T) sh.hist[0][i] = 0u;
    if (tid == 0) {
        sh.below[0] = 0u;
        sh.bad = 0u;
        s_n[0] = 0u;
        s_n[1] = 0u;
        const uint32_t lo = f2key(fdown(b.c - 1.00001f * w)), hi = f2key(fup(b.c + 1.00001f * w));
        sh.lo[0] = lo;
        sh.width[0] = hi - lo;
    }
    bool ok = sp_pick<T>(SpMedianKey{reinterpret_cast<const float4 *>(list), ks, kb, b.hm, b.a, b.ha, s_n},
                      [&](uint32_t &k1, uint32_t &k2) {
                          // (the sweep counted with the sign folded in: below there is above here)
                          const uint32_t nm = s_n[0], blt = sgn > 0.0f ? below : (uint32_t)R - below - nm;
                          k1 = r1 - blt;
                          k2 = r2 - blt;
                          return below + nm <= (uint32_t)R && blt <= r1 && r2 < blt + nm;
                      },
                      n, sh);
    if (!ok) return kWhyMedianMiss;
    med = median_from_keys(sh.v1[0], sh.v2[0], even);
    const float delta = fabsf(__fsub_rn(med, b.c));
    const float am = b.a * b.inv, ha = b.ha * b.inv;
    const float lo = am - ha, hi = am + ha, margin = 1.0e-5f * (am + ha + delta);
    __syncthreads();
    if (tid == 0) {
        const uint32_t l = __float_as_uint(fmaxf(lo - delta - margin, 0.0f)) << 1, h = __float_as_uint(hi + delta + margin) << 1;
        sh.lo[0] = l;
        sh.width[0] = h - l;
    }
    ok = sp_pick<T>(SpMadKey{reinterpret_cast<const float4 *>(list), ks, kb, b.a, b.ha, med},
                 [&](uint32_t &k1, uint32_t &k2) {
                     k1 = r1 - inner;
                     k2 = r2 - inner;
                     return inner <= r1 && r2 < inner + s_n[1];
                 },
                 n, sh);
    if (!ok) return kWhyMadMiss;
    const float v1 = __uint_as_float(sh.v1[0] >> 1), v2 = __uint_as_float(sh.v2[0] >> 1);
    mad = even ? __fmul_rn(0.5f, __fadd_rn(v1, v2)) : v1;
    if (sh.bad) return kWhySelect;
    // every value inside the band's inner end deviates by less than v1, every one beyond its outer end by more than v2;
    // and the exceedance thresholds were worked out for a median and a MAD this close to the estimates
    const bool proven = (inner == 0u || v1 >= lo + delta + margin) && v2 <= hi - delta - margin && delta <= w && fabsf(mad - am) <= b.hd;
    return proven ? -1 : kWhyMadMiss;
}

// T threads: 128 where there are columns enough to fill the GPU (their CTAs hide one another's serial parts), else more.
template <int T>
__global__ void __launch_bounds__(T, 1536 / T) xsplit_select_kernel(const XrankArgs a, const MetricParams p, const SpGeom g, const SpScratch sc,
                                                                        uint32_t *reasons) {
    pdl_wait();
    __shared__ CtShared<1> sh;
    __shared__ SpBands sb;
    __shared__ uint32_t s_n[2], s_col[4];
    const int m = blockIdx.x, t = blockIdx.y, tid = threadIdx.x;
    const int R = a.R, M = a.M;
    const size_t o = (size_t)t * M + m;
    SpCol &col = sc.col[o];
    if (tid == 0) {
        s_col[0] = col.nk;
        s_col[1] = col.below;
        s_col[2] = col.inner;
        s_col[3] = sc.namb[t];
        sb = sp_bands(col, sc.epoch, p, m);
    }
    __syncthreads();
    const SpBands &b = sb;
    if (!b.ok) return;                                 // the sweep has put the column on the step's list
    const uint32_t n = s_col[0];
    const float sgn = p.dir[m] < 0 ? -1.0f : 1.0f;
    float med = 0.0f, mad = 0.0f;
    int why;
    if (n > (uint32_t)g.col_cap) why = kWhyCtaList;
    else if (s_col[3] > (uint32_t)kSpAmb) why = kWhyAmbList;
    else why = sp_select<T>(sc.list + o * g.col_cap, n, b, sgn, s_col[1], s_col[2], R, sh, s_n, med, mad);
    if (tid != 0) return;
    if (why < 0) {
        a.med[o] = med;
        a.mad[o] = mad;
        if (a.med_user) a.med_user[o] = med;
        if (a.mad_user) a.mad_user[o] = mad;
        col.med = med;
        col.rhs = __fmul_rn(p.thrp[m], scale_of(mad, med, p.floor_rel[m], p.floor_abs[m]));
        sp_learn(col, med, mad, false, R);
    } else {
        atomicOr(&sc.fail[t], 0x80000000u | (1u << m));
        if (why == kWhyCtaList) col.rest = kSpRest + 1;
        else if (why != kWhyAmbList) col.resample = kSpRest;
        if (reasons) atomicAdd(reasons + why, 1u);
    }
}

// ---- 3. finish ---------------------------------------------------------------------------------
// Settles the deferred exceedance decisions, and recomputes the columns on the steps' lists with the values in
// registers.  As a rule there is next to nothing to do, and what counts is the number of dependent loads: every CTA
// reads the flags of all steps at once, settles the steps that are its own, and takes its share of the columns.  Few
// columns (one metric with hardly any distinct values, steps that missed) take a cluster of four CTAs each, a quarter of
// the values per thread (118 columns of 8 192 ranks: 22 us, 42 by a CTA each); more than there are clusters a CTA each,
// where one holds a column (16 384 ranks with 512 threads; CTAs of 1 024 wait for whole SMs beside other streams' work).
// V: values per thread of a CTA that takes a column alone, above 32 never.
constexpr int kFinCluster = 4;

template <int V>
__global__ void __cluster_dims__(kFinCluster, 1, 1) __launch_bounds__(512, 2) xsplit_finish_kernel(const XrankArgs a, const MetricParams p, const SpGeom g, const SpScratch sc, const int S) {
    pdl_wait();
    __shared__ CtShared<1> sh;
    __shared__ uint32_t flags[kSplitMaxSteps];
    __shared__ uint16_t before[kSplitMaxSteps + 1];   // columns to recompute before each step
    const int tid = threadIdx.x, R = a.R, M = a.M;
    uint32_t mine = 0;
    for (int t = tid; t < S; t += blockDim.x) {
        flags[t] = sc.fail[t];
        mine |= flags[t];
    }
    const bool any = __syncthreads_or(mine != 0u);
    for (int t = blockIdx.x; t < S; t += gridDim.x) {
        if (a.mask_base) {
            const uint32_t na = min(sc.namb[t], (uint32_t)kSpAmb);
            const int slot = a.first_slot + t - (t >= a.capacity - a.first_slot ? a.capacity : 0);
            const float *row = a.base + (size_t)slot * a.row_stride;
            uint8_t *maskrow = reinterpret_cast<uint8_t *>(a.mask_base) + (size_t)slot * R;
            const SpCol *cols = sc.col + (size_t)t * M;
            for (uint32_t i = tid; i < na; i += blockDim.x) {
                const uint32_t e = sc.amb[(size_t)t * kSpAmb + i];
                const uint32_t r = e >> 5, m = e & 31u;
                if ((flags[t] >> m) & 1u) continue;   // recomputed below, exceedance bits included
                if (exceeds(row[(size_t)r * M + m], cols[m].med, p.dir[m], cols[m].rhs)) {
                    const uintptr_t at = reinterpret_cast<uintptr_t>(maskrow + r);
                    atomicOr(reinterpret_cast<unsigned int *>(at & ~(uintptr_t)3), (1u << m) << (8 * (at & 3)));
                }
            }
        }
    }
    if (!any) return;
    if (tid < 32) {   // one warp: a running sum over the steps
        uint32_t run = 0;
        int redone = 0;
        for (int t0 = 0; t0 < S; t0 += 32) {
            const uint32_t f = t0 + tid < S ? flags[t0 + tid] : 0u;
            uint32_t incl = __popc(f & 0x7FFFFFFFu);
            const uint32_t own = incl;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) { const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, incl, d); if (tid >= d) incl += u; }
            if (t0 + tid < S) before[t0 + tid] = (uint16_t)(run + incl - own);
            run += __shfl_sync(0xFFFFFFFFu, incl, 31);
            redone += __popc(__ballot_sync(0xFFFFFFFFu, (f >> 31) != 0u));
        }
        if (tid == 0) {
            before[S] = (uint16_t)run;
            if (blockIdx.x == 0 && redone && a.fallbacks) atomicAdd(a.fallbacks, (uint32_t)redone);
        }
    }
    __syncthreads();
    const int n = before[S];
    const bool wide = V > 32 || n <= (int)gridDim.x / kFinCluster;      // (the same for all CTAs)
    const int share = wide ? kFinCluster : 1;
    for (int item = blockIdx.x / share; item < n; item += gridDim.x / share) {
        int lo = 0, hi = S;                // the step: before[lo] <= item < before[lo + 1]
        while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if ((int)before[mid] <= item) lo = mid; else hi = mid; }
        uint32_t bits = flags[lo] & 0x7FFFFFFFu;
        for (int f = item - (int)before[lo]; f > 0; --f) bits &= bits - 1u;
        const int m = __ffs(bits) - 1;
        if (wide) ct_row<V / kFinCluster, 1, kFinCluster>(a, p, lo, m, sh);
        else ct_row<(V > 32 ? 1 : V), 1>(a, p, lo, m, sh);
        __syncthreads();
        if (tid == 0 && (!wide || ct_rank() == 0u)) {                    // the result is the next block's estimate
            SpCol &col = sc.col[(size_t)lo * M + m];
            sp_learn(col, sh.med[0], sh.mad[0], true, R);
            if (col.epoch != sc.epoch) col.resample = 0;
            col.epoch = sc.epoch;
            if (col.rest) col.rest -= 1;
        }
    }
    if (wide) ct_sync<kFinCluster>();      // no CTA exits while others may read its shared memory
}

// Kept fraction of a column: 2 hm about the median, 4 ha about the quartiles (normal density, MAD units).
SpGeom split_geometry(int R, int S) {
    SpGeom g{};
    // strips of 512 ranks; shorter ones where that does not fill the GPU
    g.strip = 512;
    while (g.strip > 128 && (long long)S * ((R + g.strip * kSpWarps - 1) / (g.strip * kSpWarps)) < 8 * 148) g.strip /= 2;
    g.chunks = (R + g.strip * kSpWarps - 1) / (g.strip * kSpWarps);
    const int want = R / 4 > 4096 ? R / 4 : 4096;
    g.period = 4 * (R / want > 1 ? R / want : 1);
    g.s = 4 * (R / g.period);
    g.q_sample = (float)sqrt(1.0 / g.s - 1.0 / R > 0.0 ? 1.0 / g.s - 1.0 / R : 0.0);
    const double q_prev = sqrt(2.0 / R), q = q_prev > g.q_sample ? q_prev : g.q_sample;
    const double f = q * (2.0 * kSpMed * 0.2691 + 4.0 * kSpBoth * 0.2143) + 0.03;   // densities at the median and at the quartiles, per MAD
    const double kept = g.strip * f;
    g.cap = (int)ceil(kept + 6.0 * sqrt(kept)) + 16;
    g.cap = (g.cap + 3) / 4 * 4;   // (with the slack a multiple of 16 bytes)
    g.col_cap = (int)ceil(R * f * 1.1) + 128 + 2 * ((R + 127) / 128);
    g.col_cap = (g.col_cap + 31) / 32 * 32;
    return g;
}

size_t split_sweep_smem(const SpGeom &g, int M) { return (size_t)kSpWarps * M * (g.cap + kSpSlack) * sizeof(uint32_t); }

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

bool xrank_split_supported(int R, int M) { return (M == 4 || M == 8) && R >= 4096 && R <= kSpMaxRanks; }

size_t xrank_split_scratch_bytes(int R, int M, int S_max) {
    const SpGeom g = split_geometry(R, S_max);
    size_t b = 0;
    b += align256((size_t)S_max * M * sizeof(SpCol));
    b += align256((size_t)S_max * sizeof(uint32_t)) * 2;
    b += align256((size_t)S_max * kSpAmb * sizeof(uint32_t));
    b += align256((size_t)S_max * M * g.col_cap * sizeof(float));
    return b;
}

cudaError_t launch_xrank_split(const XrankArgs &a, const MetricParams &p, int S, int S_max, SplitState &state, void *scratch, uint32_t *reasons,
                               cudaStream_t st, std::vector<std::pair<cudaEvent_t, cudaEvent_t>> *prof) {
    if (S <= 0) return cudaSuccess;
    const int M = a.M;
    const SpGeom g = split_geometry(a.R, S);
    SpScratch sc{};
    char *b = (char *)scratch;
    sc.col = (SpCol *)b;      b += align256((size_t)S_max * M * sizeof(SpCol));
    sc.fail = (uint32_t *)b;  b += align256((size_t)S_max * sizeof(uint32_t));
    sc.namb = (uint32_t *)b;  b += align256((size_t)S_max * sizeof(uint32_t));
    sc.amb = (uint32_t *)b;   b += align256((size_t)S_max * kSpAmb * sizeof(uint32_t));
    sc.list = (float *)b;
    sc.epoch = a.hint_epoch;
    const size_t smem = split_sweep_smem(g, M);
    static std::mutex attr_mutex;
    static bool attr_set_dev[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    {
        std::lock_guard<std::mutex> lock(attr_mutex);
        bool &attr_set = attr_set_dev[dev & 63];
        if (!attr_set) {
            e = cudaFuncSetAttribute(xsplit_sweep_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(xsplit_sweep_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
            if (e != cudaSuccess) return e;
            attr_set = true;
        }
    }
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    if (prof && (cudaEventCreate(&ev0) != cudaSuccess || cudaEventCreate(&ev1) != cudaSuccess)) return cudaGetLastError();
    // estimates for the step positions and columns that have none (with hints a look at the records, as a rule: 2 us)
    const bool same = state.epoch == a.hint_epoch;
    e = launch_after(xsplit_sample_kernel, dim3(M / 4, S), kSpThreads, st, a, g, sc, !a.hint_fresh && same ? state.rows : 0);
    if (e != cudaSuccess) return e;
    state.rows = same && state.rows > S ? state.rows : S;
    state.epoch = a.hint_epoch;
    if (prof) cudaEventRecord(ev0, st);   // the sweep, the longest kernel
    e = M == 8 ? launch_after_smem(xsplit_sweep_kernel<2>, dim3(g.chunks, S), 32 * kSpWarps, smem, st, a, p, g, sc)
               : launch_after_smem(xsplit_sweep_kernel<1>, dim3(g.chunks, S), 32 * kSpWarps, smem, st, a, p, g, sc);
    if (e != cudaSuccess) return e;
    if (prof) cudaEventRecord(ev1, st);
    // (22 us against 23 for 1 600 columns of some 1 900 values; 9 against 14 for 400 of 2 300)
    const dim3 columns(M, S);
    if ((long long)S * M > 148 * 6) e = launch_after(xsplit_select_kernel<128>, columns, 128, st, a, p, g, sc, reasons);
    else if ((long long)S * M > 148 * 3) e = launch_after(xsplit_select_kernel<256>, columns, 256, st, a, p, g, sc, reasons);
    else e = launch_after(xsplit_select_kernel<512>, columns, 512, st, a, p, g, sc, reasons);
    if (e != cudaSuccess) return e;
    const int T = a.R <= 32 * 128 ? 128 : (a.R <= 32 * 256 ? 256 : 512);
    const int most = 148 * (1024 / T);   // what the SMs hold of them at 64 registers per thread
    const int grid = (min(S * M, most) + kFinCluster - 1) / kFinCluster * kFinCluster;
    e = a.R <= 32 * 512 ? launch_after(xsplit_finish_kernel<32>, grid, T, st, a, p, g, sc, S)
                        : launch_after(xsplit_finish_kernel<64>, grid, T, st, a, p, g, sc, S);
    if (prof) prof->emplace_back(ev0, ev1);
    return e;
}

}  // namespace guard
