// Node-sweep qualification: per-GPU medians of repeated benchmark results, and the
// pass / fail verdicts against the fleet distribution (GPU level, then node level).
#include <math_constants.h>

#include <cfloat>

#include "binmap.cuh"
#include "colselect.cuh"
#include "kernels.h"
#include "thselect.cuh"
#include "warpselect.cuh"

namespace guard {

namespace {

constexpr int kSweepCols = 128;

// One CTA stages the [reps][M] blocks of GT = 128 / M GPUs, transposed to one column per
// (GPU, metric) series, then every thread selects inside its own column.
__global__ void __launch_bounds__(kSweepCols) sweep_median_kernel(const SweepMedArgs a) {
    extern __shared__ __align__(16) uint32_t tile[];
    const int tid = threadIdx.x, M = a.M, reps = a.reps;
    const int gt = kSweepCols / M;
    const int g0 = blockIdx.x * gt;
    const int ng = min(gt, a.G - g0);
    const int per = reps * M;
    bool bad = false;
    for (int gl = 0; gl < ng; ++gl) {
        const float *src = a.S + (size_t)(g0 + gl) * per;
        for (int i = tid; i < per; i += kSweepCols) {
            const int rep = i / M, m = i - rep * M;
            const uint32_t b = __float_as_uint(src[i]);
            bad |= nonfinite_bits(b);
            tile[(size_t)rep * kSweepCols + gl * M + m] = key_of_bits(b);
        }
    }
    if (a.status && __any_sync(0xFFFFFFFFu, bad) && lane_id() == 0) atomicOr(a.status, kStatNonFinite);
    __syncthreads();
    if (tid >= ng * M) return;
    const float med = col_median(tile + tid, kSweepCols, reps);
    const size_t o = (size_t)g0 * M + tid;
    a.gmed[o] = med;
    if (a.gmed_user) a.gmed_user[o] = med;
}

// Thread-per-series path (32 to 256 repetitions, many series): a series' repetitions scatter around their mean, and the
// mean predicts the median of n repetitions to 0.75 / sqrt(n) of their standard deviation.  Pass A takes mean and standard
// deviation (the GPU's block is read once from HBM and stays in L1 / L2 for pass B); pass B counts the values below
// mean -/+ 2.83 sd / sqrt(n) and keeps those inside (32 of 200, 18 of 64) in the thread's shared-memory column; the two
// middle ranks are then found among the kept keys (pivot search, as for the window medians).  A series whose counts
// do not prove the bracket (or whose column overflows) is left to sweep_median_finish_kernel.
// Bound by the chain of instructions of a series (8 000 of them, 21 warps per SM) and by the loads' cache lines (a
// repetition is another line for every GPU of the warp).  What does not fit a warp per GPU (below) comes here.
constexpr int kSwThreads = 128;
constexpr int kSwSlots = 60;      // kept keys per series (the column format of the thread-per-series selection)
constexpr int kSwRows = 8;        // repetitions in flight per thread
constexpr int kSwMaxPasses = 12;

__global__ void __launch_bounds__(kSwThreads) sweep_median_thread_kernel(const SweepMedArgs a) {
    __shared__ __align__(16) uint32_t kept[kSwThreads * kSwSlots];
    const int tid = threadIdx.x, M = a.M, n = a.reps;
    const long long series = (long long)a.G * M;
    const long long sidx = (long long)blockIdx.x * kSwThreads + tid;
    const bool active = sidx < series;
    const long long sc = active ? sidx : series - 1;
    const int g = (int)(sc / M), m = (int)(sc - (long long)g * M);
    const float *base = a.S + (size_t)g * n * M + m;

    // pass A: mean and variance about the first value (no cancellation for values far from zero); a series
    // whose repetitions all have the same bits is its own median
    const float x0 = __ldg(base);
    const uint32_t bits0 = __float_as_uint(x0);
    float sd1 = 0.0f, sd2 = 0.0f;
    bool bad = false, same = true;
    auto acc = [&](const float xv) {
        const uint32_t b = __float_as_uint(xv);
        bad |= nonfinite_bits(b);
        same = same && (b == bits0);
        const float d = xv - x0;
        sd1 += d;
        sd2 = fmaf(d, d, sd2);
    };
    auto each = [&](auto f) {
        int r = 0;
        for (; r + kSwRows <= n; r += kSwRows) {
            float x[kSwRows];
#pragma unroll
            for (int u = 0; u < kSwRows; ++u) x[u] = __ldg(base + (size_t)(r + u) * M);
#pragma unroll
            for (int u = 0; u < kSwRows; ++u) f(x[u]);
        }
        for (; r < n; ++r) f(__ldg(base + (size_t)r * M));
    };
    each(acc);
    if (a.status && __any_sync(0xFFFFFFFFu, bad && active) && lane_id() == 0) atomicOr(a.status, kStatNonFinite);
    const float inv = 1.0f / (float)n;
    const float mean_d = sd1 * inv;
    const float var = fmaxf(sd2 * inv - mean_d * mean_d, 0.0f);
    const float c = x0 + mean_d, h = 2.83f * sqrtf(var * inv);
    const bool usable = active && !bad && !same && th_usable(c, h);
    const ThRange range = th_range(c, h, usable);

    // pass B (the block is in L1 / L2 by now): count below, keep inside
    const uint32_t kbase = (uint32_t)__cvta_generic_to_shared(kept + tid * kSwSlots), klim = kbase + (uint32_t)(kSwSlots * 4);
    uint32_t kaddr = kbase;
    float cltf = 0.0f;
    if (__any_sync(0xFFFFFFFFu, usable)) {
        each([&](const float x) { th_cell(x, range, klim, cltf, kaddr); });
    }
    const bool even = !(n & 1);
    const int k1 = (n - 1) >> 1, k2 = n >> 1;
    const int nk = (int)((kaddr - kbase) >> 2);
    const int clt = (int)cltf;
    bool ok = usable && clt <= k1 && k2 < clt + nk && nk <= kSwSlots;
    float vb = 0.0f, vu = 0.0f, med = 0.0f;
    th_select_pair<kSwSlots, kSwMaxPasses>(kbase, nk, ok, k2 - clt, range, vb, vu);
    if (ok) med = even ? __fmul_rn(0.5f, __fadd_rn(vb, vu)) : vu;
    if (active && same && !bad) { med = x0; ok = true; }
    if (active && ok) {
        a.gmed[sidx] = med;
        if (a.gmed_user) a.gmed_user[sidx] = med;
    }
    const unsigned todo = __ballot_sync(0xFFFFFFFFu, active && !ok);
    if (lane_id() == 0) a.todo[sidx >> 5] = todo;
}

// One warp per series: the lanes fetch the repetitions, sort their own keys and run the warp selection.
template <int VPL>
__device__ __forceinline__ void sweep_warp_median(const SweepMedArgs &a, const uint32_t sidx, const bool check) {
    const int lane = lane_id(), M = a.M, n = a.reps;
    const int g = (int)(sidx / (uint32_t)M), m = (int)(sidx - (uint32_t)g * (uint32_t)M);
    const float *base = a.S + (size_t)g * n * M + m;
    uint32_t kv[VPL];
    int nreal = 0;
    bool bad = false;
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
        const int rep = lane + 32 * j;
        const bool real = rep < n;
        const uint32_t b = real ? __float_as_uint(__ldg(base + (size_t)rep * M)) : 0u;
        bad |= nonfinite_bits(b);
        kv[j] = real ? key_of_bits(b) : 0xFFFFFFFFu;
        nreal += real;
    }
    if (check && a.status && __any_sync(0xFFFFFFFFu, bad) && lane == 0) atomicOr(a.status, kStatNonFinite);
    lane_sort<VPL>(kv);
    float med = 0.0f;
    const bool ok = warp_median<VPL>(kv, nreal, n, 0u, med);
    if (lane == 0) {
        if (!ok && a.status) atomicOr(a.status, kStatInternal);
        a.gmed[sidx] = med;
        if (a.gmed_user) a.gmed_user[sidx] = med;
    }
}

// The series the thread path left: their bits in a.todo.  A warp takes 32 >> parts series at a time: a whole word's, or
// fewer while that leaves a warp for each (all series of a sweep whose means say nothing about their medians: 33 600 of 64
// repetitions 101 us with whole words, 60 with quarters; 98 304 of 200 245 us by half as many warps, 200 so).
constexpr int kSwFinishCtas = 148 * 8;

template <int VPL>
__global__ void __launch_bounds__(kSwThreads) sweep_median_finish_kernel(const SweepMedArgs a, const int parts) {
    pdl_wait();
    const uint32_t words = (uint32_t)(((long long)a.G * a.M + 31) >> 5), nwarps = gridDim.x * (kSwThreads / 32), share = 32u >> parts;
    for (uint32_t i = blockIdx.x * (kSwThreads / 32) + warp_id(); i < words << parts; i += nwarps) {
        const uint32_t first = (i & ((1u << parts) - 1u)) * share;   // of the word's bits
        for (uint32_t t = __ldcg(a.todo + (i >> parts)) & ((0xFFFFFFFFu >> (32u - share)) << first); t; t &= t - 1u)
            sweep_warp_median<VPL>(a, 32u * (i >> parts) + (uint32_t)(__ffs(t) - 1), false);
    }
}

// Every series.
template <int VPL>
__global__ void __launch_bounds__(kSwThreads) sweep_median_series_kernel(const SweepMedArgs a) {
    pdl_wait();
    const long long sidx = (long long)blockIdx.x * (kSwThreads / 32) + warp_id();
    if (sidx < (long long)a.G * a.M) sweep_warp_median<VPL>(a, (uint32_t)sidx, true);
}

// A warp per GPU, whose block of repetitions is read once, coalesced, into registers: L = 32 / M lanes per metric, lane
// l < L M holds repetitions l / M, l / M + L, ... of metric l % M.  A series' mean and standard deviation bracket its median
// (2.83 sd / sqrt(n) to either side, as in the thread path).  Every lane bins its values (16 bins, the first and the last
// for what lies below and beyond; its counters are a column of shared memory, so that a warp's reductions never meet in a
// bank); the lanes of a series scan their sum for the middle ranks; the values about the wanted bins are gathered, those
// in them counted (as many as the bins say, or the series is not served) and ranked.  Series that are not served, or whose
// wanted bin holds many different values, are sorted by the whole warp on the spot: one in fifty of normal values.  Where all
// of them are (values that spread over decades) that is up to twice as long as a warp for each (1 000 x 200 x 6 28 us and 17,
// 4 096 x 200 x 6 54 and 40, 16 384 x 200 x 6 146 and 215).  Further rounds with ranges a standard deviation wide instead take 19,
// 32 and 75, but in the same kernel they cost all other sweeps 2 to 5 %.
// Bound by instruction issue and latency: 1 400 instructions a warp for 200 repetitions of 6 metrics (a third of them the
// values' passes), 24 warps per SM.  16 384 GPUs x 200 x 6 from HBM 32 us (a thread per series, whose loads take a cache line
// per GPU and pass, 53 + 5 for the series it leaves), 2 048 x 200 x 6 7.4 (a warp per series 16), 4 096 x 64 x 6 7.7 (18).
// With the kept values of the bracket in a column each, binned behind the pass, 43 us; with 32 bins and the lanes of a
// series reading the same column at a time (a bank conflict for each) 41.
constexpr int kSgBins = 16;
constexpr int kSgList = 16;       // wanted values that are ranked directly
constexpr int kSgCtl = 8;         // words per series that its lanes share
constexpr int kSgReps = 256, kSgRows = 64;   // most repetitions, and values per lane
constexpr float kSgMagic = 12582912.0f;   // 1.5 * 2^23: adding it leaves an integer in the low mantissa bits

// if (|x - c| <= h) { shared[addr] = x; addr += 128; }
__device__ __forceinline__ void sg_gather(const float x, const float c, const float h, uint32_t &addr) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t.reg .f32 d;\n\t"
        "sub.rn.f32 d, %1, %2;\n\t"
        "abs.f32 d, d;\n\t"
        "setp.le.f32 q, d, %3;\n\t"
        "@q st.shared.f32 [%0], %1;\n\t"
        "@q add.u32 %0, %0, 128;\n\t}"
        : "+r"(addr)
        : "f"(x), "f"(c), "f"(h)
        : "memory");
}

__host__ __device__ constexpr int sg_rows(const int V) { return V > kSgBins ? V : kSgBins; }
__host__ __device__ constexpr int sg_words(const int V, const int M) { return 32 * sg_rows(V) + (kSgList + kSgCtl) * M; }   // of shared memory per warp

__device__ __forceinline__ void sg_store(const SweepMedArgs &a, const int series, const float med) {
    a.gmed[series] = med;
    if (a.gmed_user) a.gmed_user[series] = med;
}

// The medians of the open series that their ranges [lo, hi] serve; the others are left.  The bins are zero.
template <int V, int M>
__device__ __forceinline__ void sg_round(const SweepMedArgs &a, const float (&x)[V], const int g, const int m, const int q, const bool act, uint32_t *hist,
                                         uint32_t *list, uint32_t *ctl, const float lo, const float hi, const bool open, bool &left) {
    constexpr int L = 32 / M;
    const int lane = lane_id(), n = a.reps;
    const uint32_t k1 = (uint32_t)((n - 1) >> 1), k2 = (uint32_t)(n >> 1);
    const uint32_t column = (uint32_t)__cvta_generic_to_shared(hist + lane);
    const BinMap map = bin_map<kSgBins - 1>(lo, hi);
    const float scale = open ? map.scale : 0.0f, off = open ? map.off : 0.0f;
    auto bin = [&](const float v) -> uint32_t { return __float_as_uint(__fmaf_rn(__saturatef(__fmaf_rn(v, scale, off)), (float)(kSgBins - 1), kSgMagic)); };
    __syncwarp();                 // bins are zero
    {
        const uint32_t at = column - __float_as_uint(kSgMagic) * 128u;
#pragma unroll
        for (int i = 0; i < V; ++i) asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(bin(x[i]) * 128u + at) : "memory");
    }
    if (q == 0) {
        ctl[kSgCtl * m] = 0u;                 // wanted bins: k1's ...
        ctl[kSgCtl * m + 1] = 0u;             // ... and k2's
        ctl[kSgCtl * m + 4] = 0u;             // values found in them
        ctl[kSgCtl * m + 5] = 0u;             // largest key of the first
        ctl[kSgCtl * m + 6] = 0xFFFFFFFFu;    // smallest key of the second
    }
    __syncwarp();
    // ---- scan: the lanes of a series share its bins ----
    constexpr int per = (kSgBins + L - 1) / L;
    const int bin0 = q * per;
    uint32_t sum = 0u, num[per];
#pragma unroll
    for (int j = 0; j < per; ++j) num[j] = 0u;
    int from = q;                 // each lane begins with its own column: no two of a series read the same one at a time
#pragma unroll
    for (int k = 0; k < L; ++k) {
#pragma unroll
        for (int j = 0; j < per; ++j)
            if (bin0 + j < kSgBins && act) num[j] += hist[32 * (bin0 + j) + m + from * M];
        from = from + 1 < L ? from + 1 : 0;
    }
#pragma unroll
    for (int j = 0; j < per; ++j) sum += num[j];
    uint32_t r = 0u;
#pragma unroll
    for (int k = 0; k < L; ++k) {
        const uint32_t o = __shfl_sync(0xFFFFFFFFu, sum, m + k * M);
        if (k < q) r += o;
    }
    if (open && k2 >= r && k1 < r + sum) {
#pragma unroll
        for (int j = 0; j < per; ++j) {
            if (k1 >= r && k1 - r < num[j]) { ctl[kSgCtl * m] = (uint32_t)(bin0 + j); ctl[kSgCtl * m + 2] = r; }
            if (k2 >= r && k2 - r < num[j]) { ctl[kSgCtl * m + 1] = (uint32_t)(bin0 + j); ctl[kSgCtl * m + 3] = r + num[j]; }
            r += num[j];
        }
    }
    __syncwarp();
    const uint32_t b1 = ctl[kSgCtl * m], b2 = ctl[kSgCtl * m + 1], start = ctl[kSgCtl * m + 2], end = ctl[kSgCtl * m + 3];
    const bool served = open && b1 >= 1u && b2 >= 1u && b1 <= kSgBins - 2u && b2 <= kSgBins - 2u;
    // ---- the values about the wanted bins (more than those in them: rounding moves a bin's ends) ----
    const bool listed = served && end - start <= (uint32_t)kSgList;
    uint32_t addr = column;
    if (__any_sync(0xFFFFFFFFu, served)) {
        const float width = map.span * (1.0f / (float)(kSgBins - 3));
        const float gc = lo + (0.5f * (float)(b1 + b2) - 1.0f) * width;
        const float gh = served ? (0.5f * (float)(b2 - b1) + 0.6f) * width + fmaxf(fabsf(lo), fabsf(hi)) * pow2_of(-21) : -1.0f;
#pragma unroll
        for (int i = 0; i < V; ++i) sg_gather(x[i], gc, gh, addr);
    }
    const int hits = (int)((addr - column) >> 7);
    const uint32_t w1 = b1 + __float_as_uint(kSgMagic), w2 = b2 + __float_as_uint(kSgMagic);
    for (int j = 0; j < hits; ++j) {
        const float v = __uint_as_float(hist[32 * j + lane]);
        const uint32_t b = bin(v);
        if (b == w1 || b == w2) {
            const uint32_t key = f2key(v), at = atomicAdd(&ctl[kSgCtl * m + 4], 1u);
            if (listed) {
                if (at < (uint32_t)kSgList) list[kSgList * m + at] = key;
            } else {
                if (b == w1) atomicMax(&ctl[kSgCtl * m + 5], key);
                if (b == w2) atomicMin(&ctl[kSgCtl * m + 6], key);
            }
        }
    }
    __syncwarp();
    const bool counted = served && ctl[kSgCtl * m + 4] == end - start;
    if (counted && listed) {
        const uint32_t cnt = end - start, q1 = k1 - start, q2 = k2 - start;
        for (uint32_t j = (uint32_t)q; j < cnt; j += (uint32_t)L) {
            const uint32_t key = list[kSgList * m + j];
            uint32_t lt = 0u, le = 0u;
            for (uint32_t i = 0; i < cnt; ++i) {
                const uint32_t o = list[kSgList * m + i];
                lt += o < key;
                le += o <= key;
            }
            if (q1 >= lt && q1 < le) ctl[kSgCtl * m + 5] = key;
            if (q2 >= lt && q2 < le) ctl[kSgCtl * m + 6] = key;
        }
    }
    __syncwarp();
    const uint32_t u1 = ctl[kSgCtl * m + 5], u2 = ctl[kSgCtl * m + 6];
    if (counted && (listed || b1 != b2 || u1 == u2)) {   // (the same for all lanes of a series)
        if (q == 0) sg_store(a, g * M + m, median_from_keys(u1, u2, !(n & 1)));
        left = false;
    }
}

// Rows of L repetitions of a GPU's block; the first V - S are whole.
template <int V, int S, int M>
__device__ __forceinline__ bool sg_valid(const int i, const bool act, const int q, const int n) { return i < V - S || (act && i * (32 / M) + q < n); }
template <int V, int S, int M>
__device__ __forceinline__ void sg_load(float (&x)[V], const float *from, const bool act, const int q, const int n) {
#pragma unroll
    for (int i = 0; i < V; ++i) {
        x[i] = FLT_MAX;               // (beyond the repetitions: ranks are counted from below)
        if (sg_valid<V, S, M>(i, act, q, n)) x[i] = __ldg(from + i * (32 / M * M));
    }
}
__device__ __forceinline__ void sg_clear(uint32_t *hist) {
#pragma unroll
    for (int i = 0; i < kSgBins / 4; ++i) reinterpret_cast<uint4 *>(hist)[lane_id() + 32 * i] = make_uint4(0u, 0u, 0u, 0u);
}

// V values per lane, at most S more than there are.
template <int V, int S, int M>
__global__ void __launch_bounds__(kSwThreads, V <= 24 ? 8 : (V <= 40 ? 6 : (V <= 56 ? 5 : 4))) sweep_median_gpu_kernel(const SweepMedArgs a) {
    pdl_wait();
    extern __shared__ __align__(16) uint32_t sg[];   // per warp: bins [kSgBins][32], then gathered values [V][32]; lists [M][kSgList], [M][kSgCtl]
    constexpr int L = 32 / M;
    const int lane = lane_id(), n = a.reps;
    const int g = blockIdx.x * (kSwThreads / 32) + warp_id();
    if (g >= a.G) return;
    uint32_t *hist = sg + warp_id() * sg_words(V, M);
    uint32_t *list = hist + 32 * sg_rows(V), *ctl = list + kSgList * M;
    const int m = lane % M, q = lane / M;
    const bool act = lane < L * M;
    const float *base = a.S + (size_t)g * n * M + min(lane, L * M - 1);   // (idle lanes read a valid column)

    auto valid = [&](const int i) { return sg_valid<V, S, M>(i, act, q, n); };
    float x[V];
    sg_load<V, S, M>(x, base, act, q, n);
    sg_clear(hist);
    uint32_t peers = 0u;          // lanes of this one's series
#pragma unroll
    for (int k = 0; k < L; ++k) peers |= 1u << (m + k * M);

    // mean and variance about the first value (no cancellation for values far from zero)
    const float x0 = __shfl_sync(0xFFFFFFFFu, x[0], m);
    float sd1 = 0.0f, sd2 = 0.0f, sda = 0.0f;
#pragma unroll
    for (int i = 0; i < V; ++i) {
        const float d = valid(i) ? x[i] - x0 : 0.0f;
        sd1 += d;
        sd2 = fmaf(d, d, sd2);
        sda += fabsf(d);
    }
    bool bad = false;
    if (__any_sync(0xFFFFFFFFu, !(sd2 < CUDART_INF_F))) {   // values that are not finite, or far apart
#pragma unroll
        for (int i = 0; i < V; ++i) bad |= nonfinite_bits(__float_as_uint(x[i]));
        if (a.status && __any_sync(0xFFFFFFFFu, bad && act) && lane == 0) atomicOr(a.status, kStatNonFinite);
    }
    bool differ = !(sda == 0.0f);
    if (__any_sync(0xFFFFFFFFu, !differ && __float_as_uint(x0) << 1 == 0u)) {   // zeros of both signs are different values
#pragma unroll
        for (int i = 0; i < V; ++i) differ = differ || (valid(i) && __float_as_uint(x[i]) != __float_as_uint(x0));
    }
    const bool same = (__ballot_sync(0xFFFFFFFFu, differ) & peers) == 0u;   // a constant series is its own median
    float t1 = 0.0f, t2 = 0.0f;
#pragma unroll
    for (int k = 0; k < L; ++k) {
        t1 += __shfl_sync(0xFFFFFFFFu, sd1, m + k * M);
        t2 += __shfl_sync(0xFFFFFFFFu, sd2, m + k * M);
    }
    const float inv = 1.0f / (float)n, mean_d = t1 * inv, var = fmaxf(t2 * inv - mean_d * mean_d, 0.0f);
    const float c = x0 + mean_d, h = 2.83f * sqrtf(var * inv);
    const bool open = act && !same && th_usable(c, h);
    bool left = act;                  // without a result
    if (act && same && !bad) {
        if (q == 0) sg_store(a, g * M + m, x0);
        left = false;
    }
    if (__any_sync(0xFFFFFFFFu, open)) sg_round<V, M>(a, x, g, m, q, act, hist, list, ctl, c - h, c + h, open, left);
    uint32_t todo = __ballot_sync(0xFFFFFFFFu, left && q == 0);
    constexpr int VPL = V * L <= 64 ? 2 : (V * L <= 128 ? 4 : 8);
    for (; todo; todo &= todo - 1u) sweep_warp_median<VPL>(a, (uint32_t)((size_t)g * M) + (uint32_t)(__ffs(todo) - 1), false);
}

// Fallback when the repetitions of one GPU do not fit a tile: bit-by-bit counting
// selection from global memory, one thread per (GPU, metric).
__global__ void sweep_median_global_kernel(const SweepMedArgs a) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= (long long)a.G * a.M) return;
    const int g = (int)(c / a.M), m = (int)(c - (long long)g * a.M);
    const float *src = a.S + (size_t)g * a.reps * a.M + m;
    const int n = a.reps, k = (n - 1) >> 1;
    uint32_t prefix = 0;
    int krem = k;
    bool bad = false;
    for (int bit = 31; bit >= 0; --bit) {
        int zeros = 0;
        for (int j = 0; j < n; ++j) {
            const uint32_t raw = __float_as_uint(src[(size_t)j * a.M]);
            bad |= nonfinite_bits(raw);
            const uint32_t key = key_of_bits(raw);
            const bool match = (bit == 31) || (((key ^ prefix) >> (bit + 1)) == 0);
            zeros += (match && !((key >> bit) & 1u));
        }
        if (krem >= zeros) {
            prefix |= 1u << bit;
            krem -= zeros;
        }
    }
    if (bad && a.status) atomicOr(a.status, kStatNonFinite);
    float med = key2f(prefix);
    if (!(n & 1)) {
        int cle = 0;
        uint32_t above = 0xFFFFFFFFu;
        for (int j = 0; j < n; ++j) {
            const uint32_t key = f2key(src[(size_t)j * a.M]);
            cle += (key <= prefix);
            if (key > prefix) above = min(above, key);
        }
        med = median_from_keys(prefix, cle > k + 1 ? prefix : above, true);
    }
    a.gmed[c] = med;
    if (a.gmed_user) a.gmed_user[c] = med;
}

// One thread per GPU, whole nodes per CTA where they fit: robust-z outlier AND beyond the percentile cut fails a metric;
// a GPU passes with no failed metric; a node passes when all of its GPUs pass.
constexpr int kVerdictThreads = 128;

__global__ void __launch_bounds__(kVerdictThreads) sweep_verdict_kernel(const SweepVerdictArgs a, const MetricParams p) {
    __shared__ float s_F[kMaxMetrics], s_rhs[kMaxMetrics], s_cut[kMaxMetrics];
    __shared__ uint32_t s_bad[kVerdictThreads];
    const int tid = threadIdx.x, gpn = a.gpus_per_node, per = max(kVerdictThreads / gpn, 1);   // nodes of this CTA
    const int node0 = blockIdx.x * per, nn = min(per, a.nodes - node0);
    s_bad[tid] = 0u;
    pdl_wait();
    if (tid < a.M) {
        const float F = a.fleet_med[tid];
        s_F[tid] = F;
        s_rhs[tid] = __fmul_rn(p.thrp[tid], scale_of(a.fleet_mad[tid], F, p.floor_rel[tid], p.floor_abs[tid]));
        s_cut[tid] = a.fleet_cut[tid];
    }
    __syncthreads();
    for (int q = tid; q < nn * gpn; q += kVerdictThreads) {
        const size_t g = (size_t)node0 * gpn + q;
        uint32_t fail = 0;
        for (int m = 0; m < a.M; ++m) {
            const float v = a.gmed[g * a.M + m];
            const bool beyond = p.dir[m] < 0 ? (v < s_cut[m]) : (v > s_cut[m]);
            if (exceeds(v, s_F[m], p.dir[m], s_rhs[m]) && beyond) fail |= 1u << m;
        }
        if (a.fail_mask) a.fail_mask[g] = fail;
        if (a.gpu_pass) a.gpu_pass[g] = (uint8_t)(fail == 0);
        if (fail) s_bad[q / gpn] = 1u;
    }
    __syncthreads();
    if (tid < nn && a.node_pass) a.node_pass[node0 + tid] = (uint8_t)(s_bad[tid] == 0u);
}

}  // namespace

template <int V, int S, int M>
static cudaError_t launch_gpu_medians(const SweepMedArgs &a, cudaStream_t st) {
    constexpr size_t smem = (size_t)(kSwThreads / 32) * sg_words(V, M) * sizeof(uint32_t);
    return launch_after_smem(sweep_median_gpu_kernel<V, S, M>, (unsigned)((a.G + kSwThreads / 32 - 1) / (kSwThreads / 32)), kSwThreads, smem, st, a);
}
// The instance for this many rows: V values per lane, in steps of eight, of sixteen where a metric has three lanes or fewer.
template <int V, int M>
static cudaError_t launch_gpu_medians(const SweepMedArgs &a, const int rows, cudaStream_t st) {
    constexpr int L = 32 / M, S = L > 3 ? 8 : 16, kWanted = (kSgReps + L - 1) / L, kMost = kWanted < kSgRows ? kWanted : kSgRows;
    if constexpr (V < kMost) {
        if (rows > V) return launch_gpu_medians<V + S, M>(a, rows, st);
    }
    return launch_gpu_medians<V, S, M>(a, st);
}
template <int M>
static cudaError_t launch_gpu_medians(const SweepMedArgs &a, const int rows, cudaStream_t st) {
    return launch_gpu_medians<(32 / M > 3 ? 8 : 16), M>(a, rows, st);
}

cudaError_t launch_sweep_medians(const SweepMedArgs &a, cudaStream_t st) {
    const long long series = (long long)a.G * a.M;
    // A warp per GPU where its values fit the registers, with three to sixteen metrics (the lanes of a series share the scan of
    // its bins: 16 384 GPUs x 64 x 1 take 87 us so, by threads 28; x 2 58 and 40), from as many values on as it is the shorter
    // way.  Four to eight metrics: 230 000 (a sweep of 296 x 100 x 6 10.9 us, a warp per series 10.2; 1 000 x 33 x 4 10.6 and
    // 10.1; but 592 x 64 x 8 11.4 and 12.7, 296 x 200 x 4 10.5 and 11.6).  Three, or two to three lanes to a series: 600 000
    // (296 x 100 x 12 14.8 and 11.2, 592 x 100 x 12 13.5 and 13.1, 1 000 x 100 x 12 14.6 and 15.8).  Three metrics have too few
    // repetitions to a lane below 64 (16 384 x 33 x 3 30.9, by threads 28.4; of 64 32 and 37).
    const int L = 32 / a.M, rows = (a.reps + L - 1) / L;
    if (a.reps <= kSgReps && rows <= kSgRows && series < 0x7FFFFFFFLL && series * a.reps >= (a.M >= 4 && a.M <= 8 ? 230000 : 600000)) {
        switch (a.M) {
            case 3:
                if (a.reps >= 64) return launch_gpu_medians<3>(a, rows, st);
                break;
            case 4: return launch_gpu_medians<4>(a, rows, st);
            case 5: return launch_gpu_medians<5>(a, rows, st);
            case 6: return launch_gpu_medians<6>(a, rows, st);
            case 7: return launch_gpu_medians<7>(a, rows, st);
            case 8: return launch_gpu_medians<8>(a, rows, st);
            case 9: return launch_gpu_medians<9>(a, rows, st);
            case 10: return launch_gpu_medians<10>(a, rows, st);
            case 11: return launch_gpu_medians<11>(a, rows, st);
            case 12: return launch_gpu_medians<12>(a, rows, st);
            case 13: return launch_gpu_medians<13>(a, rows, st);
            case 14: return launch_gpu_medians<14>(a, rows, st);
            case 15: return launch_gpu_medians<15>(a, rows, st);
            case 16: return launch_gpu_medians<16>(a, rows, st);
            default: break;
        }
    }
    // (Other numbers of metrics and repetitions.)  A warp per series while they are few: one launch, and no thread's chain over
    // all repetitions (12 288 series of 200 16 us against 29 + 5 by threads, 49 152 of 100 25 against 21 + 3), and for fewer
    // than 32 repetitions, which say too little about their median beforehand.
    if (a.reps <= 256 && series < 0x7FFFFFFFLL && (series <= 32768 || a.reps < 32)) {
        const unsigned grid = (unsigned)((series + kSwThreads / 32 - 1) / (kSwThreads / 32));
        if (a.reps <= 32) return launch_after(sweep_median_series_kernel<1>, grid, kSwThreads, st, a);
        if (a.reps <= 64) return launch_after(sweep_median_series_kernel<2>, grid, kSwThreads, st, a);
        if (a.reps <= 128) return launch_after(sweep_median_series_kernel<4>, grid, kSwThreads, st, a);
        return launch_after(sweep_median_series_kernel<8>, grid, kSwThreads, st, a);
    }
    if (a.reps >= 32 && a.reps <= 256 && series < 0x7FFFFFFFLL) {
        sweep_median_thread_kernel<<<(unsigned)((series + kSwThreads - 1) / kSwThreads), kSwThreads, 0, st>>>(a);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        const long long words = (series + 31) / 32, most = (long long)kSwFinishCtas * (kSwThreads / 32);
        int parts = 0;
        while (parts < 3 && (words << (parts + 1)) <= most) ++parts;
        const int fgrid = (int)((min(words << parts, most) + kSwThreads / 32 - 1) / (kSwThreads / 32));
        if (a.reps <= 64) return launch_after(sweep_median_finish_kernel<2>, fgrid, kSwThreads, st, a, parts);
        if (a.reps <= 128) return launch_after(sweep_median_finish_kernel<4>, fgrid, kSwThreads, st, a, parts);
        return launch_after(sweep_median_finish_kernel<8>, fgrid, kSwThreads, st, a, parts);
    }
    const size_t smem = (size_t)a.reps * kSweepCols * 4;
    if (smem <= 200 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(sweep_median_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        const int gt = kSweepCols / a.M;
        sweep_median_kernel<<<(a.G + gt - 1) / gt, kSweepCols, smem, st>>>(a);
    } else {
        const long long series = (long long)a.G * a.M;
        sweep_median_global_kernel<<<(unsigned)((series + 127) / 128), 128, 0, st>>>(a);
    }
    return cudaGetLastError();
}

cudaError_t launch_sweep_verdict(const SweepVerdictArgs &a, const MetricParams &p, cudaStream_t st) {
    const int per = a.gpus_per_node < kVerdictThreads ? kVerdictThreads / a.gpus_per_node : 1;
    return launch_after(sweep_verdict_kernel, (a.nodes + per - 1) / per, kVerdictThreads, st, a, p);
}

}  // namespace guard
