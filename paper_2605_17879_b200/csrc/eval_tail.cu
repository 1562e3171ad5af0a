// First launch of an evaluation's tail: the fleet baseline (a cluster, or a CTA, per metric: xrank_count.cuh) and, on
// CTAs of their own beside it, the top-k slowest ranks.  Both read only the windowed medians.
//
// The top-k list: the ranks' keys are held in registers, one cluster (or CTA) for the whole fleet.
//   1. a threshold with at least K keys at or above it: the one the previous evaluation left, where evaluations follow
//      closely, else the K-th largest of the maxima of some 2 K disjoint groups of ranks (K groups have a member at
//      or above it; random data have about 1.4 K keys there), or (lists too long for that) the exact K-th largest key;
//   2. the entries at or above it meet in the first CTA's shared memory, which orders them.
// Where evaluations follow closely, what is wanted is not K but the number of entries that the next evaluation's
// threshold should admit (top_want).
// A threshold that turns out too high (fewer than K) or too low (more than the list holds: ties) is replaced, in the
// second case by the exact K-th largest key, and ranks among the keys equal to it are picked by their number.
// Bound by latency: two cluster barriers and an ordering of some hundred entries, 7 us beside the baseline's 10 (the
// histogram refinement of topk.cu takes 19 us of 16 CTAs at 16 384 ranks, and a stream and two events to run beside).
#include "kernels.h"
#include "xrank_count.cuh"

namespace guard {

namespace {

constexpr int kTopGroups = 512;    // groups at most
constexpr int kTopCap = 1024;      // gathered entries at most (K <= 1024)
constexpr int kTopSlack = 8;       // entries above K that a threshold has to admit at least

struct TopShared {
    unsigned long long list[kTopCap];                // (first CTA)
    __align__(16) uint32_t gmax[kTopGroups];         // this CTA's groups' maxima
    __align__(16) uint32_t all[kTopGroups];          // every group's
    uint32_t n[8];                                   // (first CTA) gathered entries, by attempt
    uint32_t tau;
};

__device__ __forceinline__ uint32_t ct_atomic_add(const uint32_t addr, const uint32_t v) {
    uint32_t o;
    asm volatile("atom.relaxed.cluster.shared::cluster.add.u32 %0, [%1], %2;" : "=r"(o) : "r"(addr), "r"(v) : "memory");
    return o;
}
__device__ __forceinline__ void ct_st64(const uint32_t addr, const unsigned long long v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}

// Descending, list[0, n2), n2 a power of two.
__device__ __forceinline__ void top_sort(unsigned long long *list, const int n2) {
    for (int size = 2; size <= n2; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            __syncthreads();
            for (int t = threadIdx.x; t < n2 / 2; t += blockDim.x) {
                const int i = 2 * t - (t & (stride - 1)), j = i + stride;
                const unsigned long long x = list[i], y = list[j];
                if ((x < y) == ((i & size) == 0)) { list[i] = y; list[j] = x; }
            }
        }
    }
    __syncthreads();
}

// Entries that the threshold left for the next evaluation should admit, or K if it would miss too often: three times K for
// short lists; for long ones most of what the network that orders them has room for, but of the largest half, because
// more than it holds are a miss (single steps of 1 024 ranks x 4: K = 500 29 us with some 509 entries, 34 with 762;
// K = 700 38 us without a threshold that serves, 34 with 862).
__device__ __forceinline__ int top_want(const int K) {
    if (K <= kTopCap / 8) return 3 * K;
    int n2 = kTopCap / 4;
    while (n2 < kTopCap && n2 < K + kTopSlack) n2 <<= 1;
    const int room = n2 - K;
    if (n2 < kTopCap) return n2 - room / 4;
    return room >= 2 * kTopSlack ? K + room / 2 : K;
}

// R <= V * NC * blockDim.x; all threads of the cluster call this.
template <int V, int NC>
__device__ __forceinline__ void top_row(const TopkArgs &a, const MetricParams &p, uint32_t *status, TopShared &ts, CtShared<1> &sh) {
    const int tid = threadIdx.x, lane = lane_id(), T = blockDim.x;
    const int R = a.R, K = a.K, pm = p.primary;
    const int crank = NC == 1 ? 0 : (int)ct_rank(), dr = NC * T, r0 = crank * T + tid;
    const uint32_t list0 = NC == 1 ? (uint32_t)__cvta_generic_to_shared(ts.list) : ct_map(ts.list, 0u);
    const uint32_t n0 = NC == 1 ? (uint32_t)__cvta_generic_to_shared(ts.n) : ct_map(ts.n, 0u);
    // one launch writes the hint's state, in its last step: every CTA reads the same here
    const int want = a.hint ? top_want(K) : K;
    const bool keeps = want > K;   // (this evaluation's threshold serves the next)
    const bool hv = keeps && a.hint->valid;
    uint32_t tau = hv ? a.hint->tau : 0u;
    uint32_t key[V];               // larger is slower; 0 where there is no rank
    uint32_t own = 0u;
#pragma unroll
    for (int i = 0; i < V; ++i) {
        const int r = r0 + i * dr;
        key[i] = 0u;
        if (r < R) {
            const float v = __ldg(a.wmed + (size_t)r * a.M + pm);
            key[i] = f2key(p.dir[pm] < 0 ? -v : v);
        }
        own = max(own, key[i]);
    }
    if (tid < 8) ts.n[tid] = 0u;
    if (tid == 0) ts.tau = 0u;
    // Appends the entries at or above t (ranks up to `last` only) to the list; returns how many there are then.
    auto gather = [&](const uint32_t t, const uint32_t only, const uint32_t last, const int attempt) -> uint32_t {
        uint32_t mine = 0, hits = 0;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const int r = r0 + i * dr;
            if (key[i] >= t && key[i] <= only && r < R && (uint32_t)r <= last) { mine += 1u; hits |= 1u << i; }
        }
        if (__any_sync(0xFFFFFFFFu, mine != 0u)) {
            uint32_t incl = mine;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) { const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, incl, d); if (lane >= d) incl += u; }
            uint32_t base = 0;
            if (lane == 31) base = ct_atomic_add(n0 + 4u * (uint32_t)attempt, incl);
            uint32_t pos = __shfl_sync(0xFFFFFFFFu, base, 31) + incl - mine;
#pragma unroll
            for (int i = 0; i < V; ++i)
                if ((hits >> i) & 1u) {
                    if (pos < (uint32_t)kTopCap)
                        ct_st64(list0 + 8u * pos, ((unsigned long long)key[i] << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)(r0 + i * dr)));
                    pos += 1u;
                }
        }
        ct_sync<NC>();
        return ct_ld(n0 + 4u * (uint32_t)attempt);
    };
    // (a second list would overwrite the first: its readers, the first CTA's last step, come after all of them)
    uint32_t n = 0;
    bool done = false, hit = false;
    if (hv) {
        ct_sync<NC>();
        n = gather(tau, kCtNone, kCtNone, 0);
        hit = done = n >= (uint32_t)K && n <= (uint32_t)kTopCap;
    }
    if (!done) {
        // groups of `lanes` neighbouring lanes (all of their values): at least 128 of them and 4/3 of the wanted number, or of
        // K where there cannot be so many
        const int threads = NC * T;
        const int target = 3 * min(threads, kTopGroups) >= 4 * want ? want : K;
        int lanes = 32;
        while (lanes > 1 && (threads / lanes < 128 || 3 * (threads / lanes) < 4 * target)) lanes >>= 1;
        const int G = threads / lanes, per = G / NC;
        const bool all = R <= 128, grouped = !all && G <= kTopGroups && 3 * G >= 4 * target;
        if (grouped) {
            uint32_t m = own;
            for (int d = 1; d < lanes; d <<= 1) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, d));
            if ((lane & (lanes - 1)) == 0) ts.gmax[tid / lanes] = m;
        }
        ct_sync<NC>();
        tau = 0u;
        if (grouped) {
            for (int g = tid; g < G; g += T) ts.all[g] = NC == 1 ? ts.gmax[g] : ct_ld(ct_map(&ts.gmax[g % per], (uint32_t)(g / per)));
            __syncthreads();
            // the `target`-th largest: the one that `target` - 1 others come before (equal ones in the order of their groups)
            for (int g = tid; g < G; g += T) {
                const uint32_t x = ts.all[g], x1 = x == 0u ? 0u : x - 1u;
                const uint4 *q = reinterpret_cast<const uint4 *>(ts.all);
                int before = 0;
#pragma unroll 4
                for (int j = 0; j < G / 4; ++j) {
                    const uint4 o = q[j];
                    const uint32_t c = j < g / 4 ? x1 : x;
                    before += (int)(o.x > c) + (int)(o.y > c) + (int)(o.z > c) + (int)(o.w > c);
                }
                for (int j = g & ~3; j < g; ++j) before += ts.all[j] == x;
                if (before == target - 1) ts.tau = x;
            }
            __syncthreads();
            tau = ts.tau;
        }
        if (all || grouped) {
            n = gather(tau, kCtNone, kCtNone, 1);
            done = n <= (uint32_t)kTopCap;
        }
    }
    if (!done) {
        // the exact largest of that place (ranks that do not exist lie below all keys); where ties make too many of it, the K-th
        for (int i = tid; i < kCtBins; i += T) sh.hist[0][i] = 0u;
        if (tid == 0) { sh.below[0] = 0u; sh.bad = 0u; }
        uint32_t kth;
        for (int target = min(want, R);; target = K) {
            if (tid == 0) { sh.lo[0] = 0u; sh.width[0] = kCtNone; }
            const uint32_t at = (uint32_t)(V * NC * T - target);
            ct_select<V, 1, NC>(key, at, at, sh);
            kth = tau = sh.v1[0];
            n = gather(kth, kCtNone, kCtNone, target == K ? 3 : 2);
            if (n <= (uint32_t)kTopCap || target == K) break;
        }
        if (n > (uint32_t)kTopCap) {                 // more equal ones than the list holds: those of the lowest ranks
            const uint32_t above = kth == kCtNone ? 0u : gather(kth + 1u, kCtNone, kCtNone, 4);
            uint32_t rk[V];
#pragma unroll
            for (int i = 0; i < V; ++i) rk[i] = key[i] == kth && r0 + i * dr < R ? (uint32_t)(r0 + i * dr) : kCtNone;
            if (tid == 0) { sh.lo[0] = 0u; sh.width[0] = (uint32_t)R; }
            const uint32_t nth = (uint32_t)K - above - 1u;
            ct_select<V, 1, NC>(rk, nth, nth, sh);
            n = gather(kth, kth, sh.v1[0], 4);
        }
        if (sh.bad && crank == 0 && tid == 0) atomicOr(status, kStatInternal);
    }
    if (crank != 0) return;
    auto put = [&](const int at, const unsigned long long e) {
        const int32_t r = (int32_t)(0xFFFFFFFFu - (uint32_t)e);
        if (at < K) a.idx_keep[at] = r;
        if (a.hint && at == min((int)n, want) - 1) {
            a.hint->valid = keeps ? 1u : 0u;
            a.hint->tau = (int)n >= want ? (uint32_t)(e >> 32) : tau;   // (never higher than what admitted too few)
            if (hit) a.hint->hits += 1u; else a.hint->misses += 1u;
        }
    };
    if (n <= 128u) {               // each entry counts those before it
        for (int i = tid; i < (int)n; i += T) {
            const unsigned long long e = ts.list[i];
            int at = 0;
#pragma unroll 4
            for (int j = 0; j < (int)n; ++j) at += ts.list[j] > e;
            put(at, e);
        }
    } else {
        int n2 = 256;
        while (n2 < (int)n) n2 <<= 1;
        for (int i = (int)n + tid; i < n2; i += T) ts.list[i] = 0ull;
        top_sort(ts.list, n2);
        for (int i = tid; i < (int)n; i += T) put(i, ts.list[i]);
    }
}

template <int V, int NC>
__global__ void __cluster_dims__(NC, 1, 1) __launch_bounds__(NC == 1 ? 1024 : 512, 1) eval_tail_kernel(const XrankArgs x, const TopkArgs t, const MetricParams p) {
    __shared__ CtShared<1> sh;
    __shared__ TopShared ts;
    pdl_wait();
    pdl_trigger();                 // (the score pass counts exceedances meanwhile)
    if ((int)blockIdx.x < x.M * NC) ct_row<V, 1, NC>(x, p, 0, blockIdx.x / NC, sh);
    else top_row<V, NC>(t, p, x.status, ts, sh);
    if (NC > 1) ct_sync<NC>();     // no CTA exits while others may read its shared memory
}

template <int NC>
cudaError_t launch(const XrankArgs &x, const TopkArgs &t, const MetricParams &p, const int most, cudaStream_t st) {
    const int T = ct_cluster_threads(x.R, NC, most), v = (x.R + NC * T - 1) / (NC * T), grid = (x.M + (t.K > 0 ? 1 : 0)) * NC;
    if (v <= 4) return launch_after(eval_tail_kernel<4, NC>, grid, T, st, x, t, p);
    if (v <= 8) return launch_after(eval_tail_kernel<8, NC>, grid, T, st, x, t, p);
    return launch_after(eval_tail_kernel<16, NC>, grid, T, st, x, t, p);
}

}  // namespace

// The fleet baseline x (one row, no exceedance bits) and, with t.K > 0, the top-k list t (no scores) of one evaluation;
// R <= kCountMaxRanks.  steps: evaluations follow one another by a few steps.  Their tails share the GPU with the clusters of
// the next steps' rows: CTAs of up to 256 threads, two to an SM, where four values a thread would ask for 512 (deferred single
// steps of 16 384 ranks x 8 24.3 us, with 512 26.1; of 24 000 28.3 and 32.4).  After a block up to 512 where 256 would hold sixteen
// values a thread, a longer chain (blocks of 50 steps of 24 000 x 8, W = 100, 163.4 us, with 256 166.2; of 32 768 205.6 and
// 208.9), but not with eight, where the next blocks' kernels need the room (a hundred blocks of 200 steps of 16 384 x 8, W =
// 200, 10.48 ms, with 512 10.68).
cudaError_t launch_eval_tail(const XrankArgs &x, const TopkArgs &t, const MetricParams &p, const bool steps, cudaStream_t st) {
    if (x.R <= kCtClusterRanks) {
        int T = 32;
        while (T < 1024 && x.R > 4 * T) T <<= 1;
        return launch_after(eval_tail_kernel<4, 1>, x.M + (t.K > 0 ? 1 : 0), T, st, x, t, p);
    }
    const bool few = steps || x.R <= 8 * 8 * ct_most_threads(8);
    return (x.M + 1) * 8 <= 148 ? launch<8>(x, t, p, few ? ct_most_threads(8) : 512, st) : launch<4>(x, t, p, 512, st);
}

}  // namespace guard
