// Node-sweep qualification: per-GPU medians of repeated benchmark results, and the
// pass / fail verdicts against the fleet distribution (GPU level, then node level).
#include <math_constants.h>

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
// repetition is another line for every GPU of the warp): 39 us at 16 384 GPUs x 200 x 6 with the results in L2, 63 from
// HBM.  Not faster: the next loads in flight ahead of the passes (the same), blocks staged whole in shared memory (seven
// warps per SM: 62 and 64), or in chunks of eight repetitions, asynchronously (84) or through registers (49 and 68).
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

cudaError_t launch_sweep_medians(const SweepMedArgs &a, cudaStream_t st) {
    const long long series = (long long)a.G * a.M;
    // A warp per series while they are few: one launch, and no thread's chain over all repetitions (1 776 series of 33
    // repetitions 2.8 us against 8.9 + 1.9, 12 288 of 200 16 against 29 + 5, 24 576 of 64 18 against 15 + 4, 49 152 of
    // 100 25 against 21 + 3, 98 304 of 200 95 against 45 + 5), and for fewer than 32 repetitions, which say too little
    // about their median beforehand.
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
