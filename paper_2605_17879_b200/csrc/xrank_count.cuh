// Cross-rank selection of rows held in registers: a CTA holds C adjacent metrics of one row (element e of the
// group belongs to metric e mod C, so that a thread's values all belong to one metric and the loads are
// coalesced) and finds each metric's median, then its MAD, the same way:
//   1. a key range that should hold the wanted ranks: around the previous result of the same row position where
//      the caller has one, else between two of 32 spread values sorted by a warp;
//   2. one pass counts the keys below the range and bins those inside (256 bins in shared memory);
//   3. one warp per metric scans its bins for the wanted ranks; a second pass fetches the keys of those one or
//      two bins (a few), and the warp ranks them.
// A few wide columns (a single row of thousands of ranks) take a cluster of NC CTAs each (C = 1): the CTAs bin their
// shares on their own, sum one another's bins and gather one another's few keys through distributed shared memory
// (two cluster barriers a round), and all take the same decisions.
// The counts prove the range; one that misses is moved, and a bin that holds too many keys becomes the next
// range (or the answer, if they are all the same: ties), so any values come out exactly.  A key is 32 bits in
// the order of the values, so that both statistics (and both kinds of range) share one piece of code.
// Bound by latency and by the half-rate integer pipe; what it avoids is what measured worst on the way here:
// branches and returning atomics per value, rounds of pivots (each some 500 cycles of dependent scalar work in one
// warp, whatever the number of values) and column-wise loads (a cache line per lane).  Measured, kernel alone:
// 100 steps of 1 024 ranks x 8 metrics 9.5 us (8-bit radix select of xrank_direct.cuh: 76), 60 steps of 4 096 x 16
// 29 us (576; three CTAs per SM; the instances with 32 values a thread spill 44 and 56 bytes at 64 registers).
#pragma once
#include "kernels.h"

namespace guard {

constexpr int kCtBins = 256;
constexpr int kCtList = 64;        // keys of a bin that are ranked directly (two per lane)
constexpr int kCtMaxIter = 64;     // a range shrinks at least to a 128th whenever its bin is too full
constexpr uint32_t kCtNone = 0xFFFFFFFFu;  // the largest key: a NaN's, and what padding holds (in whatever range it falls, it comes last)
constexpr int kCtAll = 0, kCtStatistics = 1, kCtCut = 2;   // what a CTA (cluster) computes: both, median and MAD, the extra order statistic
// Single rows of 8 metrics, bracketed by the row before / not: one CTA of 1 024 threads per column takes 6.3 / 7.5 us at
// 2 048 ranks, 7.9 / 9.6 at 4 096, 9.5 / 11.6 at 6 000 (and 12.9 / 17.5 at 16 384); a cluster of eight pays two cluster
// barriers and the gathering of bins a round and takes 8.8 / 10.2, 9.1 / 10.8, 9.2 / 11.6 and 10.4 / 15.3 (with up to 512
// threads a CTA).
constexpr int kCtClusterRanks = 4096;
// Threads of the CTAs of a cluster: four values each, while a CTA has 256 of them at most: at 128 registers two such CTAs
// share an SM, so that the clusters of a step's row and of another evaluation's tail find room beside one another and
// beside the window kernels (six deferred steps of 32 768 ranks x 8 take 5 % longer with up to 512 threads; steps that nothing
// runs beside, of 16 384 to 32 768 ranks, the same within 0.5 %).  Clusters of four need 512 to hold the widest rows in sixteen
// values a thread.
__host__ __device__ constexpr int ct_most_threads(const int NC) { return NC >= 8 ? 256 : 512; }
inline int ct_cluster_threads(const int R, const int NC, const int most) {
    int T = 128;
    while (T < most && R > 4 * NC * T) T <<= 1;
    return T;
}
static_assert(16 * 8 * ct_most_threads(8) >= kCountMaxRanks && 16 * 4 * ct_most_threads(4) >= kCountMaxRanks, "every row fits sixteen values a thread");

template <int C>
struct CtShared {
    __align__(16) uint32_t hist[C][kCtBins];
    uint32_t lo[C], width[C];      // the range [lo, lo + width]
    uint32_t below[C];             // keys below it
    uint32_t f0[C], fe[C];         // keys to fetch: [f0, fe]
    uint32_t how[C];               // 0 nothing to fetch, 1 list and rank, 2 largest up to / smallest from `cutk`, 3 smallest and largest
    uint32_t cutk[C];
    uint32_t q1[C];                // rank of k1 among the fetched keys
    uint32_t mx[C], mn[C];
    uint32_t nl[C];                // gathered keys
    uint32_t list[C][kCtList];
    uint32_t all[kCtList];         // (clusters) the lists of all CTAs
    uint32_t v1[C], v2[C];
    uint32_t any_open[2];
    float med[C], mad[C], rhs[C];
    uint32_t bad;
};

// Ascending sort of one key per lane (bitonic network over shuffles).
__device__ __forceinline__ uint32_t ct_warp_sort(uint32_t x, const int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            const uint32_t o = __shfl_xor_sync(0xFFFFFFFFu, x, stride);
            const bool asc = (lane & size) == 0, upper = (lane & stride) != 0;
            x = (asc != upper) ? min(x, o) : max(x, o);
        }
    return x;
}

__device__ __forceinline__ int ct_shift(const uint32_t width) {
    const int bits = 32 - __clz(width);
    return bits > 8 ? bits - 8 : 0;
}

// below += (k < lo); if (k - lo <= width) hist[(k - lo) >> sft] += 1.  (lo + width does not wrap, so the unsigned
// difference of a key below the range is beyond any width.)
__device__ __forceinline__ void ct_bin(const uint32_t k, const uint32_t lo, const uint32_t width, const int sft, const uint32_t hist,
                                       uint32_t &below) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .u32 o, a;\n\t"
        "setp.lt.u32 p, %1, %2;\n\t"
        "sub.u32 o, %1, %2;\n\t"
        "@p add.u32 %0, %0, 1;\n\t"
        "setp.le.u32 q, o, %3;\n\t"
        "shr.u32 o, o, %4;\n\t"
        "mad.lo.u32 a, o, 4, %5;\n\t"
        "@q red.shared.add.u32 [a], 1;\n\t}"
        : "+r"(below)
        : "r"(k), "r"(lo), "r"(width), "r"(sft), "r"(hist)
        : "memory");
}
// if (k - f0 <= fw) hits |= bit
__device__ __forceinline__ void ct_hit(const uint32_t k, const uint32_t f0, const uint32_t fw, const uint32_t bit, uint32_t &hits) {
    asm("{\n\t.reg .pred q;\n\t.reg .u32 o;\n\tsub.u32 o, %1, %2;\n\tsetp.le.u32 q, o, %3;\n\t@q or.b32 %0, %0, %4;\n\t}"
        : "+r"(hits)
        : "r"(k), "r"(f0), "r"(fw), "r"(bit));
}

// Distributed shared memory of a cluster: the address of this CTA's variable p in CTA `rank`, and loads from there.
__device__ __forceinline__ uint32_t ct_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t ct_map(const void *p, const uint32_t rank) {
    uint32_t o;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(o) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return o;
}
__device__ __forceinline__ uint32_t ct_ld(const uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint4 ct_ld4(const uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
// Barrier of all threads that share a column.
template <int NC>
__device__ __forceinline__ void ct_sync() {
    if (NC == 1) __syncthreads();
    else asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Scans the bins of column c (one warp): what to fetch for ranks k1 and k2, or where the range has to move.
template <int C, int NC = 1>
__device__ __forceinline__ void ct_scan(CtShared<C> &sh, const int c, const uint32_t k1, const uint32_t k2) {
    const int lane = lane_id();
    uint4 *h = reinterpret_cast<uint4 *>(&sh.hist[c][lane * 8]);
    uint4 a, b;
    uint32_t below;
    const uint32_t lo = sh.lo[c], width = sh.width[c];
    if (NC == 1) {
        a = h[0];
        b = h[1];
        below = sh.below[c];
        h[0] = make_uint4(0u, 0u, 0u, 0u);
        h[1] = make_uint4(0u, 0u, 0u, 0u);
    } else {   // (the other CTAs read this one's bins as well: cleared after the next cluster barrier)
        a = b = make_uint4(0u, 0u, 0u, 0u);
        const uint32_t part = lane < NC ? ct_ld(ct_map(&sh.below[c], (uint32_t)(lane & (NC - 1)))) : 0u;
        uint4 va[NC], vb[NC];      // (all in flight together; in two halves, which fit 64 registers, a row takes 1.3 us more)
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const uint32_t at = ct_map(h, (uint32_t)k);
            va[k] = ct_ld4(at);
            vb[k] = ct_ld4(at + 16u);
        }
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            a.x += va[k].x; a.y += va[k].y; a.z += va[k].z; a.w += va[k].w;
            b.x += vb[k].x; b.y += vb[k].y; b.z += vb[k].z; b.w += vb[k].w;
        }
        below = __reduce_add_sync(0xFFFFFFFFu, part);
    }
    const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    const uint32_t sum = ((a.x + a.y) + (a.z + a.w)) + ((b.x + b.y) + (b.z + b.w));
    uint32_t incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, incl, d); if (lane >= d) incl += u; }
    const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, sum);
    if (lane == 0) {
        if (NC == 1) sh.below[c] = 0u;
        sh.nl[c] = 0u;
        sh.mx[c] = 0u;
        sh.mn[c] = kCtNone;
    }
    if (k1 >= below && k2 < below + total) {   // the lane that has k1's bin, and the one that has k2's, say so themselves
        const int sft = ct_shift(width);
        const uint32_t in_bin = (1u << sft) - 1u;
        uint32_t r = below + incl - sum, b1 = 0, b2 = 0, q = 0, n = 0;
        const bool has1 = k1 - r < sum && k1 >= r, has2 = k2 - r < sum && k2 >= r;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (k1 >= r && k1 - r < w[j]) { b1 = (uint32_t)(8 * lane + j); q = k1 - r; n = w[j]; }
            if (k2 >= r && k2 - r < w[j]) b2 = (uint32_t)(8 * lane + j);
            r += w[j];
        }
        if (has1) {
            const uint32_t first = lo + (b1 << sft);
            sh.q1[c] = q;
            sh.f0[c] = first;
            sh.cutk[c] = first + in_bin;               // last key of k1's bin
            sh.how[c] = q + (k2 - k1) >= n ? 2u : (n <= (uint32_t)kCtList ? 1u : 3u);
        }
        if (has2) sh.fe[c] = lo + min((b2 << sft) + in_bin, width);
    } else if (lane == 0) {   // the range does not hold both ranks: move or stretch it, sixteenfold
        const uint32_t hi = lo + width, step = width >= 0x07FF0000u ? 0x7FFFFFFFu : 16u * width + 65536u;
        uint32_t nlo = lo, nhi = hi;
        if (below > k1) { nlo = lo > step ? lo - step : 0u; if (below > k2) nhi = lo; }
        if (k2 >= below + total) { nhi = hi < kCtNone - step ? hi + step : kCtNone; if (k1 >= below + total) nlo = hi; }
        sh.lo[c] = nlo;
        sh.width[c] = nhi - nlo;
        sh.f0[c] = kCtNone;
        sh.fe[c] = kCtNone;
        sh.how[c] = 0u;
    }
}

// The answer of column c from the fetched keys (one warp), or the next range; returns whether the search goes on.
template <int C, int NC = 1>
__device__ __forceinline__ bool ct_settle(CtShared<C> &sh, const int c, const bool pair) {
    const int lane = lane_id();
    const uint32_t how = sh.how[c], q1 = sh.q1[c];
    uint32_t n, mx, mn, own = 0, base = 0;
    const uint32_t part = (uint32_t)(lane & (NC - 1));   // (clusters) the CTA whose keys this lane fetches
    if (NC == 1) {
        n = sh.nl[c];
        mx = sh.mx[c];
        mn = sh.mn[c];
    } else {
        own = ct_ld(ct_map(&sh.nl[c], part));
        mx = ct_ld(ct_map(&sh.mx[c], part));
        mn = ct_ld(ct_map(&sh.mn[c], part));
        base = own;
#pragma unroll
        for (int d = 1; d < NC; d <<= 1) { const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, base, d, NC); if ((int)part >= d) base += u; }
        n = __shfl_sync(0xFFFFFFFFu, base, NC - 1);
        base -= own;
        mx = __reduce_max_sync(0xFFFFFFFFu, mx);
        mn = __reduce_min_sync(0xFFFFFFFFu, mn);
    }
    if (how == 0u) return true;                      // the range moved
    if (how != 1u) {
        if (how == 3u && mx != mn) {                 // a full bin of different keys becomes the range
            if (lane == 0) { sh.lo[c] = mn; sh.width[c] = mx - mn; }
            return true;
        }
        if (lane == 0) { sh.v1[c] = mx; sh.v2[c] = mn; }
        return false;
    }
    const uint32_t q2 = pair ? q1 + 1u : q1;
    const uint32_t *list = NC == 1 ? sh.list[c] : sh.all;
    if (NC > 1) {                                    // all CTAs' keys in one list (their bins hold kCtList at most together)
        for (uint32_t e = (uint32_t)(lane / NC); e < own; e += 32u / NC)
            if (base + e < (uint32_t)kCtList) sh.all[base + e] = ct_ld(ct_map(&sh.list[c][e], part));
        __syncwarp();
    }
    for (uint32_t e = (uint32_t)lane; e < n; e += 32u) {
        const uint32_t x = list[e];
        uint32_t lt = 0, le = 0;
#pragma unroll 4
        for (uint32_t j = 0; j < n; ++j) {
            const uint32_t o = list[j];
            lt += o < x;
            le += o <= x;
        }
        if (q1 >= lt && q1 < le) sh.v1[c] = x;
        if (q2 >= lt && q2 < le) sh.v2[c] = x;
    }
    return false;
}

// Keys of 0-based ranks k1 and k2 (k2 == k1 or k1 + 1) of the C columns held by the CTA, left in sh.v1 / sh.v2; the
// columns' ranges are in sh.lo / sh.width, the bins are zero.  All threads of the CTA (of the cluster) call this; returns
// the number of rounds.
template <int V, int C, int NC = 1>
__device__ __forceinline__ int ct_select(const uint32_t (&key)[V], const uint32_t k1, const uint32_t k2, CtShared<C> &sh) {
    const int tid = threadIdx.x, lane = lane_id(), warp = warp_id();
    const int col = tid & (C - 1);
    const uint32_t hist = (uint32_t)__cvta_generic_to_shared(sh.hist[col]);
    bool searching = true;         // (of a warp c < C: column c)
#pragma unroll 1
    for (int it = 0; it < kCtMaxIter; ++it) {
        if (tid == 0) sh.any_open[it & 1] = 0u;
        __syncthreads();           // ranges, counters and bins are ready
        {
            const uint32_t lo = sh.lo[col], width = sh.width[col];
            const int sft = ct_shift(width);
            uint32_t below = 0;
#pragma unroll
            for (int i = 0; i < V; ++i) ct_bin(key[i], lo, width, sft, hist, below);
            if (C == 1) {
                below = __reduce_add_sync(0xFFFFFFFFu, below);
            } else {
#pragma unroll
                for (int d = 16; d >= C; d >>= 1) below += __shfl_xor_sync(0xFFFFFFFFu, below, d);
            }
            if (lane < C) atomicAdd(&sh.below[lane], below);
        }
        ct_sync<NC>();
        if (warp < C && searching) ct_scan<C, NC>(sh, warp, k1, k2);
        __syncthreads();
        {
            const uint32_t f0 = sh.f0[col], fw = sh.fe[col] - f0;
            uint32_t hits = 0;
#pragma unroll
            for (int i = 0; i < V; ++i) ct_hit(key[i], f0, fw, 1u << i, hits);
            if (hits) {            // a few threads
                const uint32_t how = sh.how[col], cutk = sh.cutk[col];
#pragma unroll 1
                for (; hits; hits &= hits - 1u) {
                    const int at = __ffs(hits) - 1;
                    uint32_t k = key[0];
#pragma unroll
                    for (int i = 1; i < V; ++i) k = at == i ? key[i] : k;
                    if (how == 1u) {
                        const uint32_t pos = atomicAdd(&sh.nl[col], 1u);
                        if (pos < (uint32_t)kCtList) sh.list[col][pos] = k;
                    } else if (how >= 2u) {
                        if (how == 3u || k <= cutk) atomicMax(&sh.mx[col], k);
                        if (how == 3u || k > cutk) atomicMin(&sh.mn[col], k);
                    }
                }
            }
        }
        ct_sync<NC>();
        if (NC > 1) {              // every CTA has read the bins
            for (int i = tid; i < C * kCtBins; i += blockDim.x) (&sh.hist[0][0])[i] = 0u;
            if (tid < C) sh.below[tid] = 0u;
        }
        if (warp < C && searching) {
            searching = ct_settle<C, NC>(sh, warp, k2 != k1);
            if (lane == 0) {
                if (searching) sh.any_open[it & 1] = 1u;
                else { sh.lo[warp] = 0xFFFFFFFDu; sh.width[warp] = 0u; sh.f0[warp] = 0xFFFFFFFDu; sh.fe[warp] = 0xFFFFFFFDu; }   // (no key of a number, a computed NaN or padding)
            }
        }
        __syncthreads();
        if (sh.any_open[it & 1] == 0u) return it + 1;
    }
    if (tid == 0) sh.bad = 1u;
    return kCtMaxIter;
}

// Median, MAD (and optional extra order statistic) of metrics [m0, m0 + C) of row s of the launch, and their
// exceedance bits.  C divides M, R * C <= V * NC * blockDim.x, blockDim.x >= 32 * C; C = 1 with clusters.
template <int V, int C, int NC = 1>
__device__ __forceinline__ void ct_row(const XrankArgs &a, const MetricParams &p, const int s, const int m0, CtShared<C> &sh, const int part = kCtAll) {
    const int tid = threadIdx.x, lane = lane_id(), warp = warp_id(), T = blockDim.x;
    const int R = a.R, M = a.M;
    const int col = tid & (C - 1);
    const int slot = a.first_slot + s - (s >= a.capacity - a.first_slot ? a.capacity : 0);   // (s < capacity)
    constexpr bool kCopies = NC == 1 && V <= 8;   // (the larger ones have no registers to spare)
    const float *ring = a.base + (size_t)slot * a.row_stride + m0, *row = kCopies && a.copy_from ? a.copy_from + (size_t)s * a.row_stride + m0 : ring;
    const bool even = (R & 1) == 0;
    const uint32_t k1 = (uint32_t)((R - 1) / 2), k2 = (uint32_t)(R / 2);

    uint32_t key[V];                      // first the values' keys, later those of the deviations
    // this thread's ranks: r0, r0 + dr, ...
    const int crank = NC == 1 ? 0 : (int)ct_rank(), dr = NC * T / C, r0 = crank * T + tid / C;
    const bool speaks = crank == 0;
    bool settled = true;
    float xs = 0.0f, hmed = 0.0f, hmad = -1.0f;
    if (warp < C) {
        xs = __ldg(row + (size_t)(((2 * lane + 1) * (long long)R) >> 6) * M + warp);
        // The result arrays still hold an earlier result of this row position, or of another one.  Only its own with a
        // cluster, whose CTAs have to read the same: another row's leader may be writing there, its own row nobody writes
        // (the launches that write one set of rows follow one another) before the cluster's first barrier has passed.
        // One lane reads for its warp.
        if (NC == 1 ? a.prev_rows > 0 : s < a.prev_rows) {
            const size_t o = (size_t)min(s, a.prev_rows - 1) * M + m0 + warp;
            if (lane == 0) { hmed = a.med[o]; hmad = a.mad[o]; }
        }
    }
#pragma unroll
    for (int i = 0; i < V; ++i) {
        const int r = r0 + i * dr;
        key[i] = 0x7FFFFFFFu;             // a NaN whose keys lie above those of all numbers
        if (r < R) key[i] = __float_as_uint(__ldg(row + (size_t)r * M + col));
    }
    if (warp < C) {                       // (behind the loads of the values: they are all in flight together)
        hmed = __shfl_sync(0xFFFFFFFFu, hmed, 0);
        hmad = __shfl_sync(0xFFFFFFFFu, hmad, 0);
    }
    if (kCopies && a.copy_from) {         // (a copy in front, with its launch, takes 2.5 us more at 64 ranks x 4 x 50)
#pragma unroll
        for (int i = 0; i < V; ++i)
            if (r0 + i * dr < R) const_cast<float *>(ring)[(size_t)(r0 + i * dr) * M + col] = __uint_as_float(key[i]);
    }
    for (int i = tid; i < C * kCtBins / 4; i += T) reinterpret_cast<uint4 *>(&sh.hist[0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tid < C) sh.below[tid] = 0u;
    if (tid == 0) sh.bad = 0u;
    auto range = [&](const uint32_t lo, const uint32_t hi) {   // of the column of this warp
        if (lane == 0) { sh.lo[warp] = lo; sh.width[warp] = hi - lo; }
    };
    // from its spread values: eight or more positions to either side of the wanted rank's (three standard
    // deviations of a sample of 32)
    auto sampled = [&](const uint32_t x, const uint32_t k) {
        const uint32_t sorted = ct_warp_sort(x, lane);
        const int pos = (int)(((long long)k * 32) / R);
        const uint32_t lo = __shfl_sync(0xFFFFFFFFu, sorted, max(pos - 8, 0)), hi = __shfl_sync(0xFFFFFFFFu, sorted, min(pos + 9, 31));
        range(lo, hi);
    };
    // a previous result brackets the new one to four standard errors of the difference of two sample medians /
    // MADs of normal data (2.6 and 1.65 MAD / sqrt(R)): some 5.6 sqrt(R) keys
    const float u = hmad * rsqrtf((float)R);
    const bool hinted = hmad > 0.0f && hmad < 1.0e37f && fabsf(hmed) < 1.0e37f;
    if (warp < C) {
        if (part == kCtCut) sampled(f2key(xs), (uint32_t)a.cut_rank[m0]);   // (the first of C)
        else if (hinted) range(f2key(hmed - 10.0f * u), f2key(hmed + 10.0f * u));
        else sampled(f2key(xs), k1);
    }
    if (a.check_finite) {
        bool bad = false;
#pragma unroll
        for (int i = 0; i < V; ++i) bad |= nonfinite_bits(key[i]) && r0 + i * dr < R;
        if (__any_sync(0xFFFFFFFFu, bad) && lane == 0) atomicOr(a.status, kStatNonFinite);
    }
#pragma unroll
    for (int i = 0; i < V; ++i) key[i] = key_of_bits(key[i]);
    float med = 0.0f;                     // of this thread's column
    // what: 0 the median, 1 the MAD, 2 + c the extra order statistic of metric m0 + c (before the MAD)
#pragma unroll 1
    for (int what = part == kCtCut ? 2 : 0;;) {
        const bool extra = what >= 2;
        const uint32_t q1 = extra ? (uint32_t)a.cut_rank[m0 + what - 2] : k1, q2 = extra ? q1 : k2;
        const int rounds = ct_select<V, C, NC>(key, q1, q2, sh);
        settled = settled && (extra || (hinted && rounds == 1));   // (thread 0's warp knows of a hint)
        if (what == 0) {   // (the keys stand until the next selection settles)
            med = median_from_keys(sh.v1[col], sh.v2[col], even);
            if (tid < C) sh.med[tid] = med;
        } else if (tid < C) {
            const uint32_t v1 = sh.v1[tid], v2 = sh.v2[tid];
            const int m = m0 + tid;
            const size_t o = (size_t)s * M + m;
            if (what == 1) {
                const float lo = __uint_as_float(v1 >> 1), md = sh.med[tid];
                const float mad = even ? __fmul_rn(0.5f, __fadd_rn(lo, __uint_as_float(v2 >> 1))) : lo;
                sh.mad[tid] = mad;
                sh.rhs[tid] = __fmul_rn(p.thrp[m], scale_of(mad, md, p.floor_rel[m], p.floor_abs[m]));
                if (speaks) {
                    a.med[o] = md;
                    a.mad[o] = mad;
                    if (a.med_user) a.med_user[o] = md;
                    if (a.mad_user) a.mad_user[o] = mad;
                    if (NC > 1 && a.hint) {
                        RowHints *h = reinterpret_cast<RowHints *>(a.hint);
                        if (m == 0) atomicAdd(&h->rows, 1u);
                        if (settled) atomicAdd(&h->settled, 1u);
                    }
                }
            } else if (tid == what - 2 && speaks) {
                a.cut[o] = key2f(v1);
                if (a.cut_user) a.cut_user[o] = key2f(v1);
            }
        }
        if (what == 1 || (part == kCtCut && what == C + 1)) {
            if (tid == 0 && speaks && sh.bad && a.status) atomicOr(a.status, kStatInternal);
            break;
        }
        // the metrics' extra ranks first (they need the values), then the deviations
        what = !a.cut || part == kCtStatistics ? 1 : (what == 0 ? 2 : (what - 1 < C ? what + 1 : 1));
        if (what >= 2) {
            if (warp < C) sampled(f2key(xs), (uint32_t)a.cut_rank[m0 + what - 2]);
        } else {
            // the keys of the deviations: their bits with the sign as the lowest bit
            if (warp < C) {
                const float centre = C == 1 ? med : __shfl_sync(0xFFFFFFFFu, med, warp);   // (lane c holds column c's)
                if (hinted) range(__float_as_uint(fmaxf(hmad - 6.6f * u, 0.0f)) << 1, (__float_as_uint(hmad + 6.6f * u) << 1) | 1u);
                else sampled(__float_as_uint(__fsub_rn(xs, centre)) << 1, k1);
            }
#pragma unroll
            for (int i = 0; i < V; ++i) {
                const uint32_t b = __float_as_uint(__fsub_rn(key2f(key[i]), med));
                key[i] = (b << 1) | (b >> 31);   // NaN stays above infinity
            }
        }
    }
    if (!a.mask_base) return;
    __syncthreads();
    const float rhs = sh.rhs[col];
    const bool neg = p.dir[m0 + col] < 0;
    constexpr uint32_t gmask = (1u << C) - 1u;
    // bits this CTA answers for: its metrics', and (first group) those of no metric
    const uint32_t own = (gmask << m0) | (m0 == 0 && M < 32 ? ~((1u << M) - 1u) : 0u);
    uint8_t *out = reinterpret_cast<uint8_t *>(a.mask_base) + (size_t)slot * R * a.mask_bytes;
    // rows whose bytes fall into 32-bit words the same way for every rank quad of a warp
    const bool bytes = a.mask_bytes == 1, words = bytes && C != M && (R & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 3) == 0;
#pragma unroll
    for (int i = 0; i < V; ++i) {
        const float dev = __uint_as_float((key[i] >> 1) | (key[i] << 31));
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, (neg ? -dev : dev) > rhs);
        const int r = r0 + i * dr;
        if (r < R) {
            const uint32_t bits = (bal >> lane) & gmask;
            if (bytes && C == M) {           // the whole row is this CTA's: the first lane of a rank stores its byte
                if (col == 0) out[r] = (uint8_t)bits;
            } else if (words) {              // the row's other CTAs own the other bits: in place, four ranks at a time
                if ((lane & (4 * C - 1)) == 0) {
                    uint32_t four = 0;
#pragma unroll
                    for (int q = 0; q < 4; ++q) four |= ((bal >> ((lane + q * C) & 31)) & gmask) << (8 * q + m0);
                    unsigned int *w = reinterpret_cast<unsigned int *>(out + r);
                    atomicAnd(w, ~((own & 0xFFu) * 0x01010101u));
                    if (four) atomicOr(w, four);
                }
            } else if (bytes) {
                if (col == 0) {
                    const uintptr_t at = reinterpret_cast<uintptr_t>(out + r);
                    const int sft = 8 * (int)(at & 3);
                    unsigned int *w = reinterpret_cast<unsigned int *>(at & ~(uintptr_t)3);
                    atomicAnd(w, ~((own & 0xFFu) << sft));
                    if (bits) atomicOr(w, (bits << m0) << sft);
                }
            } else if (col == 0) {
                unsigned int *w = reinterpret_cast<unsigned int *>(out) + r;
                atomicAnd(w, ~own);
                if (bits) atomicOr(w, bits << m0);
            }
        }
    }
}

}  // namespace guard
